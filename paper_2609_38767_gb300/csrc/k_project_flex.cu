// k_project_flex.cu -- factored projection (Eq. 2) on the tcgen05 tensor cores with
// tiles and clusters cut to the batch, for any k_in, k_out up to 64: fp32 factors of
// any batch, and bf16 factors where whole examples per SM would leave SMs idle.
//
// fp32 factors: every value is cut into three bf16 pieces, x = h + m + l (8 significant bits each, by
// truncation: h + m + l = x exactly), and the signs S are +-1, so the products h S, m S, l S are exact and
// only sums round: sum h S in one fp32 accumulator, sum (m + l) S in another. bf16 factors are the MMA's A
// operand as TMA wrote them, one accumulator.
//
// Accuracy: the tensor pipe adds 16 features at a time into its accumulators with truncation. Among values
// of similar size it loses almost nothing (the terms are coarse against the sum's ulp), but every loss
// points to zero, so that wide layers with a few large features drift (cubed normals, 49152 features: 5.3e-5
// off in one sum; rounded fp32 chain 4.0e-6, bf16 1.9e-6). So an accumulator takes four chunks (256 features;
// eight where the streaming kernel's one sum is the alternative), and the epilogue adds it to the token's row
// of At or Bt with round-to-nearest (3.8e-7; bf16 3.5e-7, in runs of eight 5.2e-7). The accumulators form
// groups in two TMEM buffers: one group is added beside the next one's MMAs, and bf16 has four accumulators a
// group, so that barriers and commits are rare. At the end of a tile the epilogue contracts the rows, Phi +=
// Bt^T At, in fp32, as the other kernels do. One sum a side against this: fp32 2048 -> 2048, k = 64, 64 x 512
// tokens 134 and 128 us; bf16 4096 -> 4096, k = 64 x 48, 64 x 300 tokens 95 and 95 us; at worst (narrow
// layers of many tokens, bound by the epilogue: 128 -> 1528, k = 64 x 32, 201 x 300) 77 and 84 us.
//
// The pieces go to TMEM, not to shared memory: the MMA takes its A operand from
// TMEM (a lane per token, two bf16 features per column), the split warps read
// each TMA-written fp32 row once (a thread per token row: the 128-byte swizzle
// makes its 16-byte loads conflict-free) and write three pieces with
// tcgen05.st. Shared memory carries 8 bytes per value instead of 20 (write,
// read, three pieces written and read), which at HBM speed (5.4 values a clock
// and SM) would exceed its 128 bytes a clock.
//
// Token tiles of R <= 128 rows and clusters of 1 to 8 CTAs that share an example's
// tiles, chosen by a model of the chunk time (plan()): few examples fill the chip
// with smaller tiles and larger clusters, and a token count just past a tile is
// split evenly. T <= R packs floor(R/T) whole examples in a tile. The members'
// partial blocks are reduce-scattered over distributed shared memory: every CTA
// sums and writes 1/cs of Phi.
//
// Signs: a byte of a sign word becomes eight bf16 signs by one table read. bf16 factors at k = 64 have
// two pairs of generator warps that take every other stage (96 x 130 tokens, 1000 -> 4096: 70 us
// with one pair, 60 us with two); elsewhere a second pair costs 1 to 3 %.
//
// Measured, fp32: 64 examples of 512 tokens, 2048 -> 2048, k = 32 (537 MB): 7.6 ms
// on the CUDA cores, 102 us here. bf16: see plan_bf16_flex().
//
// Warp roles (fp32 512, bf16 256 or 320 threads, one persistent CTA per SM): warp 0 TMA
// producer; warp 1 TMEM allocator and MMA issuer; warps 2-3 (8-9) sign generators;
// warps 4-7 epilogue; fp32: warps 8-15 split. Every wait is bounded (about 1 s); on
// expiry the kernel records kErrTimeout, drains its copies, frees its TMEM and
// returns.
#include <cuda.h>

#include <mutex>

#include "tda_internal.cuh"

namespace tda {
namespace {

constexpr int kTileM = 128;   // MMA M
constexpr int kChunkK = 64;   // features per stage: one bf16 box or two 32-feature fp32 boxes
constexpr uint32_t kBoxBytes = kTileM * 128;  // room of one box (a 128-byte row per token)
constexpr size_t kSmemMax = 232448;
constexpr int kMaxStages = 8;
constexpr int kSR = 64;       // token rows added in one chain
constexpr int kPieceCols = kChunkK / 2;       // TMEM columns of one piece of a chunk
constexpr int kACols = 3 * kPieceCols;
constexpr int kABufs = 2;
constexpr size_t kLutBytes = 256 * 16;

template <int K, bool F32>
struct Cfg {
    static constexpr int kSignPairs = !F32 && K >= 64 ? 2 : 1;  // warps 2-3, 8-9
    static constexpr int kThreads = F32 ? 512 : 256 + 64 * (kSignPairs - 1);
    static constexpr uint32_t kTileBytes = (F32 ? 2 : 1) * kBoxBytes;
    static constexpr uint32_t kSignBytes = K * 128;
    static constexpr uint32_t kStageBytes = kTileBytes + kSignBytes;
    static constexpr int kAccs = F32 ? 2 : 4;              // accumulators of a group: h and m + l, or of one run of chunks each
    static constexpr int kBufCols = kAccs * K;
    static constexpr int kAOff = 2 * kBufCols;             // first column of the A pieces (fp32)
    static constexpr int kStageLd = K + 4;
    static constexpr size_t kStaging = 2ull * kTileM * kStageLd * 4;
    static constexpr size_t kTail = kLutBytes + 8 * (4 * kMaxStages + 2 * kABufs + 4 + 3) + 16;
    static constexpr int kFit = (int)((kSmemMax - 1024 - kStaging - kTail) / kStageBytes);
    static constexpr int kStages = kFit > kMaxStages ? kMaxStages : kFit;
    static constexpr size_t kSmem = 1024 + (size_t)kStages * kStageBytes + kStaging + kTail;
    static constexpr int RB = K / 16, CB = K / 8;          // 16 x 8 threads contract a K x K block
    static constexpr int kPer = RB * CB;
    static_assert(kAOff + (F32 ? kABufs * kACols : 0) <= 512, "TMEM columns");
    static_assert(kStages >= 3 && kSmem <= kSmemMax && kStageBytes % 1024 == 0, "shared memory per CTA");
    static_assert((size_t)K * K * 4 <= kStaging, "the other members' slices fit the staging rows");
};

struct Params {
    int64_t N, T, ld_phi, n_slots;
    uint64_t key_in, key_out;
    float scale;
    float* phi;
    unsigned int* err;
    int R;           // token rows per tile
    int n_ttiles;    // token tiles per slot
    int pack;        // examples per tile, or 1
    int k_in, k_out, nk_in, nk_out;
    int cs;          // CTAs per cluster sharing one example's tiles
    int run;         // log2 of the chunks that an accumulator takes before it is drained
};

#include "tc_ptx.cuh"

__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// D[tmem] (+)= A[tmem] * B[smem]^T, bf16 inputs, fp32 accumulation.
__device__ __forceinline__ void mma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(
            d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 32 lanes x N consecutive fp32 columns of TMEM into registers, one wait.
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[N]) {
    static_assert(N == 16 || N == 32 || N == 64, "columns");
    uint32_t r[N];
#pragma unroll
    for (int c = 0; c < N; c += 16)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[c]), "=r"(r[c + 1]), "=r"(r[c + 2]), "=r"(r[c + 3]), "=r"(r[c + 4]), "=r"(r[c + 5]), "=r"(r[c + 6]),
              "=r"(r[c + 7]), "=r"(r[c + 8]), "=r"(r[c + 9]), "=r"(r[c + 10]), "=r"(r[c + 11]), "=r"(r[c + 12]),
              "=r"(r[c + 13]), "=r"(r[c + 14]), "=r"(r[c + 15])
            : "r"(taddr + c));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < N; ++c) {
        asm volatile("" : "+r"(r[c]));  // not read before the wait
        v[c] = __uint_as_float(r[c]);
    }
}

// The upper halves of two fp32 bit patterns: the truncated bf16 pair (lo in the low half).
__device__ __forceinline__ uint32_t pack_hi(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }

// x = h + m + l, each the upper half of its fp32 pattern. An infinite x has m = l = 0.
__device__ __forceinline__ void split3(float x, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = __float_as_uint(x);
    const float hf = __uint_as_float(h & 0xFFFF0000u);
    float r = x - hf;
    if (fabsf(x) == __int_as_float(0x7F800000)) r = 0.f;
    m = __float_as_uint(r);
    l = __float_as_uint(r - __uint_as_float(m & 0xFFFF0000u));
}

// The sequence of token tiles one CTA works on, identical for every warp role:
// slots cid, cid + ncl, ... and, within a slot, the tiles crank, crank + cs, ...
struct Units {
    int64_t x;
    int tt;
    __device__ __forceinline__ void next(const Params& p, uint32_t ncl, uint32_t crank) {
        tt += p.cs;
        if (tt >= p.n_ttiles) {
            tt = (int)crank;
            x += ncl;
        }
    }
};

template <int K, bool F32>
__global__ void __launch_bounds__(Cfg<K, F32>::kThreads, 1)
project_flex_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const Params p) {
    using C = Cfg<K, F32>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float* stX = (float*)(smem + (size_t)C::kStages * C::kStageBytes);  // [kTileM][K+4] At rows
    float* stY = stX + kTileM * C::kStageLd;                            // [kTileM][K+4] Bt rows
    uint8_t* lut = smem + (size_t)C::kStages * C::kStageBytes + C::kStaging;
    uint64_t* bars = (uint64_t*)(lut + kLutBytes);
    uint64_t* full = bars;                     // [stages] boxes landed (count 1 + tx)
    uint64_t* rempty = bars + kMaxStages;      // [stages] fp32: boxes read by the split warps (8)
    uint64_t* sready = bars + 2 * kMaxStages;  // [stages] signs written (2)
    uint64_t* sempty = bars + 3 * kMaxStages;  // [stages] MMAs done with the signs, bf16: and the boxes (1)
    uint64_t* afull = bars + 4 * kMaxStages;   // [2] pieces in TMEM (8)
    uint64_t* aempty = afull + kABufs;         // [2] MMAs done with the pieces (1)
    uint64_t* tfull = aempty + kABufs;         // [2] a group is accumulated (1)
    uint64_t* tempty = tfull + 2;              // [2] the accumulators are drained (4)
    uint64_t* mma_done = tempty + 2;
    uint64_t* red_go = mma_done + 1;           // the other members' staging rows are free (cs - 1)
    uint64_t* red_full = red_go + 1;           // the other members' slices have landed here (cs - 1)
    uint32_t* tmem_slot = (uint32_t*)(red_full + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&rempty[s]), 8);
            mbar_init(smem_u32(&sready[s]), 2);
            mbar_init(smem_u32(&sempty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&afull[b]), 8);
            mbar_init(smem_u32(&aempty[b]), 1);
            mbar_init(smem_u32(&tfull[b]), 1);
            mbar_init(smem_u32(&tempty[b]), 4);
        }
        mbar_init(smem_u32(mma_done), 1);
        mbar_init(smem_u32(red_go), p.cs > 1 ? p.cs - 1 : 1);
        mbar_init(smem_u32(red_full), p.cs > 1 ? p.cs - 1 : 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (threadIdx.x < 256) {  // entry e: bit j of e as the bf16 sign of element j
        const uint32_t e = threadIdx.x;
        uint32_t q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            q[i] = (0x3F80u | (((e >> (2 * i)) & 1u) << 15)) | ((0x3F80u | (((e >> (2 * i + 1)) & 1u) << 15)) << 16);
        *reinterpret_cast<uint4*>(lut + e * 16) = make_uint4(q[0], q[1], q[2], q[3]);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // every CTA's barriers exist before any remote arrive
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t crank = cluster_rank(), cid = blockIdx.x / p.cs, ncl = gridDim.x / p.cs;
    const int nk_tot = p.nk_in + p.nk_out;
    const int group = F32 ? 1 << p.run : C::kAccs << p.run;  // chunks of a group
    Units it{(int64_t)cid, (int)crank};

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer
        uint32_t s = 0, ph = 0, last_par[C::kStages];
        bool issued[C::kStages], ok = true;
        for (int i = 0; i < C::kStages; ++i) issued[i] = false;
        const uint32_t box = (uint32_t)p.R * 128u;
        uint64_t* const free_bar = F32 ? rempty : sempty;
        for (; ok && it.x < p.n_slots; it.next(p, ncl, crank)) {
            const int row = p.pack > 1 ? (int)(it.x * p.pack * p.T) : it.tt * p.R;
            const int ex = p.pack > 1 ? 0 : (int)it.x;
            for (int kc = 0; kc < nk_tot; ++kc) {
                if (!wait_bounded(smem_u32(&free_bar[s]), ph ^ 1u, abort, p.err)) {
                    ok = false;
                    break;
                }
                const bool side_b = kc >= p.nk_in;
                const int d0 = (side_b ? kc - p.nk_in : kc) * kChunkK;
                const uint32_t dst = smem_u32(smem + (size_t)s * C::kStageBytes), bar = smem_u32(&full[s]);
                mbar_arrive_tx(bar, F32 ? 2 * box : box);
                tma_load_3d(dst, side_b ? &tmB : &tmA, d0, row, ex, bar);
                if constexpr (F32) tma_load_3d(dst + kBoxBytes, side_b ? &tmB : &tmA, d0 + 32, row, ex, bar);
                issued[s] = true;
                last_par[s] = ph;
                if (++s == (uint32_t)C::kStages) s = 0, ph ^= 1u;
            }
        }
        for (int i = 0; i < C::kStages; ++i)
            if (issued[i]) {
                const uint64_t t0 = global_ns();
                while (!mbar_try_wait(smem_u32(&full[i]), last_par[i]))
                    if (global_ns() - t0 > kTimeoutNs) {
                        atomicOr(p.err, kErrTimeout);
                        break;
                    }
            }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the warp waits, one lane issues
        uint32_t s = 0, ph = 0, cnt = 0, grp = 0;
        bool ok = true;
        constexpr uint32_t idesc = idesc_bf16(kTileM, K);
        for (; ok && it.x < p.n_slots; it.next(p, ncl, crank))
            for (int k0 = 0; ok && k0 < nk_tot; ++grp) {  // groups end with a side
                const uint32_t b = grp & 1u;
                const int side_end = k0 < p.nk_in ? p.nk_in : nk_tot;
                const int n = side_end - k0 < group ? side_end - k0 : group;
                if (!warp_wait(smem_u32(&tempty[b]), ((grp >> 1) & 1u) ^ 1u, abort, p.err)) {
                    ok = false;
                    break;
                }
                for (int c = 0; c < n; ++c, ++cnt) {
                    const uint32_t a = cnt & 1u;
                    if (!warp_wait(smem_u32(&sready[s]), ph, abort, p.err) ||
                        !(F32 ? warp_wait(smem_u32(&afull[a]), (cnt >> 1) & 1u, abort, p.err)
                              : warp_wait(smem_u32(&full[s]), ph, abort, p.err))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = smem_u32(smem + (size_t)s * C::kStageBytes);
                    const uint64_t bd = sw128_desc(st + C::kTileBytes);
                    const uint32_t dh = tmem + b * C::kBufCols + (F32 ? 0 : (c >> p.run) * K), dl = dh + K;
                    const bool clear = (c & ((1 << p.run) - 1)) == 0;
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < kChunkK / 16; ++k) {  // K = 16: 32 bytes of bf16, 8 columns of pieces
                            const uint32_t acc = clear && k == 0 ? 0u : 1u;
                            if constexpr (F32) {
                                const uint32_t at = tmem + C::kAOff + a * kACols;
                                mma_bf16_ta(dh, at + 8 * k, bd + 2 * k, idesc, acc);
                                mma_bf16_ta(dl, at + kPieceCols + 8 * k, bd + 2 * k, idesc, acc);
                                mma_bf16_ta(dl, at + 2 * kPieceCols + 8 * k, bd + 2 * k, idesc, 1u);
                            } else {
                                mma_bf16(dh, sw128_desc(st) + 2 * k, bd + 2 * k, idesc, acc);
                            }
                        }
                        if constexpr (F32) mma_commit(smem_u32(&aempty[a]));
                        mma_commit(smem_u32(&sempty[s]));
                    }
                    __syncwarp();
                    if (++s == (uint32_t)C::kStages) s = 0, ph ^= 1u;
                }
                if (!ok) break;
                if (elect_one()) mma_commit(smem_u32(&tfull[b]));
                __syncwarp();
                k0 += n;
            }
        if (elect_one()) {
            mma_commit(smem_u32(mma_done));
            const uint64_t t0 = global_ns();
            while (!mbar_try_wait(smem_u32(mma_done), 0))
                if (global_ns() - t0 > kTimeoutNs) {
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
        }
        __syncwarp();
    } else if (warp == 2 || warp == 3 || (C::kSignPairs == 2 && warp >= 8)) {
        // ---------------- sign generators: a pair of warps takes a stage, its 64 threads share a tile's K
        // rows, kParts threads per row; two pairs take turns
        constexpr int kParts = 64 / K, kChunks = 8 / kParts;
        const int g = (warp & 1) * 32 + lane, col = g / kParts, part = g % kParts;
        const uint32_t lut_s = smem_u32(lut);
        uint32_t s = 0, ph = 0, turn = warp >= 8 ? 1u : 0u;
        bool ok = true;
        for (; ok && it.x < p.n_slots; it.next(p, ncl, crank))
            for (int kc = 0; kc < nk_tot; ++kc, turn ^= 1u) {
                if (C::kSignPairs == 2 && turn) {  // the other pair's
                    if (++s == (uint32_t)C::kStages) s = 0, ph ^= 1u;
                    continue;
                }
                const bool side_b = kc >= p.nk_in;
                const uint64_t w = sign_word(side_b ? p.key_out : p.key_in, (uint32_t)col,
                                             (uint64_t)(side_b ? kc - p.nk_in : kc));
                uint4 q[kChunks];
#pragma unroll
                for (int c = 0; c < kChunks; ++c)
                    q[c] = lds128(lut_s + ((((uint32_t)(w >> (8 * (part * kChunks + c)))) & 0xFFu) << 4));
                bool got = warp_wait(smem_u32(&sempty[s]), ph ^ 1u, abort, p.err);
                if (!got) {
                    ok = false;
                    break;
                }
                uint8_t* row = smem + (size_t)s * C::kStageBytes + C::kTileBytes + (col >> 3) * 1024 + (col & 7) * 128;
#pragma unroll
                for (int c = 0; c < kChunks; ++c)
                    *reinterpret_cast<uint4*>(row + (((part * kChunks + c) ^ (col & 7)) << 4)) = q[c];
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sready[s]));
                if (++s == (uint32_t)C::kStages) s = 0, ph ^= 1u;
            }
    } else if (F32 && warp >= 8) {
        // ---------------- split warps: a thread per token row, 32 features (one box) each
        const int q4 = warp & 3, half = (warp - 8) >> 2, row = q4 * 32 + lane;
        const bool active = q4 * 32 < p.R;
        uint32_t s = 0, ph = 0, cnt = 0;
        bool ok = true;
        for (; ok && it.x < p.n_slots; it.next(p, ncl, crank))
            for (int kc = 0; kc < nk_tot; ++kc, ++cnt) {
                const uint32_t a = cnt & 1u;
                bool got = warp_wait(smem_u32(&full[s]), ph, abort, p.err);
                if (!got) {
                    ok = false;
                    break;
                }
                uint32_t h[16], m[16], l[16];
                if (active) {
                    const uint32_t src = smem_u32(smem + (size_t)s * C::kStageBytes) + (uint32_t)half * kBoxBytes +
                                         (uint32_t)row * 128u;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint4 v = lds128(src + (uint32_t)((c ^ (row & 7)) << 4));
                        uint32_t hh[4], mm[4], ll[4];
                        split3(__uint_as_float(v.x), hh[0], mm[0], ll[0]);
                        split3(__uint_as_float(v.y), hh[1], mm[1], ll[1]);
                        split3(__uint_as_float(v.z), hh[2], mm[2], ll[2]);
                        split3(__uint_as_float(v.w), hh[3], mm[3], ll[3]);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            h[2 * c + i] = pack_hi(hh[2 * i], hh[2 * i + 1]);
                            m[2 * c + i] = pack_hi(mm[2 * i], mm[2 * i + 1]);
                            l[2 * c + i] = pack_hi(ll[2 * i], ll[2 * i + 1]);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&rempty[s]));
                if (!warp_wait(smem_u32(&aempty[a]), ((cnt >> 1) & 1u) ^ 1u, abort, p.err)) {
                    ok = false;
                    break;
                }
                if (active) {
                    tc_fence_after();
                    const uint32_t dst = tmem + ((uint32_t)(q4 * 32) << 16) + C::kAOff + a * kACols + half * 16;
                    tmem_st16(dst, h);
                    tmem_st16(dst + kPieceCols, m);
                    tmem_st16(dst + 2 * kPieceCols, l);
                    tmem_wait_st();
                    tc_fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&afull[a]));
                if (++s == (uint32_t)C::kStages) s = 0, ph ^= 1u;
            }
    } else if (warp >= 4) {
        // ---------------- epilogue: groups of chunks -> sums in shared memory -> Phi += Bt^T At
        const int q4 = warp & 3, et = threadIdx.x - 128, rg = et >> 3, cg = et & 7;
        uint32_t grp = 0, red_use = 0;
        bool ok = true;
        float acc[C::RB][C::CB];
        auto clear = [&]() {
#pragma unroll
            for (int i = 0; i < C::RB; ++i)
#pragma unroll
                for (int j = 0; j < C::CB; ++j) acc[i][j] = 0.f;
        };
        auto contract = [&](int t0, int t1) {  // acc += rows t0 .. t1 - 1 (at most kSR) of At, Bt
            // into sums of their own where there are registers: a chain of at most kSR rows, not of the
            // CTA's share of the example, rounds less (560 tokens: 3.1e-7 off in one chain)
            constexpr bool kOwn = !F32 || K < 64;
            float sum[C::RB][C::CB];
            auto& to = *(kOwn ? &sum : &acc);
            if constexpr (kOwn)
#pragma unroll
                for (int i = 0; i < C::RB; ++i)
#pragma unroll
                    for (int j = 0; j < C::CB; ++j) sum[i][j] = 0.f;
#pragma unroll 2
            for (int t = t0; t < t1; ++t) {
                float y[C::RB], x[C::CB];
#pragma unroll
                for (int i = 0; i < C::RB; ++i) y[i] = stY[t * C::kStageLd + rg * C::RB + i];
#pragma unroll
                for (int j = 0; j < C::CB; ++j) x[j] = stX[t * C::kStageLd + cg * C::CB + j];
#pragma unroll
                for (int i = 0; i < C::RB; ++i)
#pragma unroll
                    for (int j = 0; j < C::CB; ++j) to[i][j] = fmaf(y[i], x[j], to[i][j]);
            }
            if constexpr (kOwn)
#pragma unroll
                for (int i = 0; i < C::RB; ++i)
#pragma unroll
                    for (int j = 0; j < C::CB; ++j) acc[i][j] += sum[i][j];
        };
        auto write = [&](int64_t n) {
            float* out = p.phi + n * p.ld_phi;
#pragma unroll
            for (int i = 0; i < C::RB; ++i)
#pragma unroll
                for (int j = 0; j < C::CB; ++j) {
                    const int r = rg * C::RB + i, c = cg * C::CB + j;
                    if (r < p.k_out && c < p.k_in) out[r * p.k_in + c] = acc[i][j] * p.scale;
                }
        };
        // Phi of example n, summed over the cluster: thread et's elements belong to member
        // et * cs / 128; every other member sends them there, in slots of 128 / cs threads each.
        auto flush = [&](int64_t n) -> bool {
            if (p.cs > 1) {
                const int per = 128 / p.cs, own = et / per;
                bool got = true;
                epi_sync();  // this CTA's staged rows are read
                if (et < p.cs && et != (int)crank) mbar_arrive_remote(smem_u32(red_go), (uint32_t)et);
                if (lane == 0) got = wait_bounded_cluster(smem_u32(red_go), red_use & 1u, abort, p.err);
                got = __shfl_sync(0xffffffffu, got, 0);
                if (epi_any(!got)) return false;
                if (own != (int)crank) {
                    const uint32_t slot = crank < (uint32_t)own ? crank : crank - 1;  // senders in rank order
                    const uint32_t dst = map_rank(smem_u32(stX) + (slot * per + (et - own * per)) * C::kPer * 4u, own);
#pragma unroll
                    for (int i = 0; i < C::RB; ++i)
#pragma unroll
                        for (int j = 0; j < C::CB; ++j) st_cluster_f32(dst + (i * C::CB + j) * 4u, acc[i][j]);
                }
                fence_acq_rel_cluster();
                epi_sync();
                if (et < p.cs && et != (int)crank) mbar_arrive_remote(smem_u32(red_full), (uint32_t)et);
                if (lane == 0) got = wait_bounded_cluster(smem_u32(red_full), red_use & 1u, abort, p.err);
                got = __shfl_sync(0xffffffffu, got, 0);
                if (epi_any(!got)) return false;
                ++red_use;
                if (own == (int)crank) {
                    for (int r = 0; r < p.cs - 1; ++r) {
                        const float* part = stX + (size_t)(r * per + (et - own * per)) * C::kPer;
#pragma unroll
                        for (int i = 0; i < C::RB; ++i)
#pragma unroll
                            for (int j = 0; j < C::CB; ++j) acc[i][j] += part[i * C::CB + j];
                    }
                    write(n);
                }
                epi_sync();  // the slices are read: staging rows free for the next tile
            } else {
                write(n);
            }
            return true;
        };
        clear();
        while (ok && it.x < p.n_slots) {
            const int64_t cur = it.x;
            const int rows = p.pack > 1 ? p.pack * (int)p.T : p.R;
            // every accumulator is added with round-to-nearest to this thread's row of At or Bt, in shared
            // memory or (bf16, which has the registers) in registers
            for (int side = 0; ok && side < 2; ++side) {
                const int nk = side ? p.nk_out : p.nk_in;
                const bool active = q4 * 32 < rows;
                float* dst = (side ? stY : stX) + (q4 * 32 + lane) * C::kStageLd;
                float sum[K];  // bf16
#pragma unroll
                for (int i = 0; i < K; ++i) sum[i] = 0.f;
                for (int k0 = 0; k0 < nk; k0 += group, ++grp) {
                    const uint32_t b = grp & 1u;
                    ok = warp_wait(smem_u32(&tfull[b]), (grp >> 1) & 1u, abort, p.err);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t tb = tmem + ((uint32_t)(q4 * 32) << 16) + b * C::kBufCols;
                    if (F32 && active) {
#pragma unroll
                        for (int c0 = 0; c0 < K; c0 += 16) {
                            float v[16], lo[16];
                            tmem_ld16(tb + c0, v);
                            tmem_ld16(tb + K + c0, lo);
#pragma unroll
                            for (int i = 0; i < 16; i += 4) {
                                float4* d4 = reinterpret_cast<float4*>(dst + c0 + i);
                                const float4 o = k0 > 0 ? *d4 : make_float4(0.f, 0.f, 0.f, 0.f);
                                *d4 = make_float4(o.x + (v[i] + lo[i]), o.y + (v[i + 1] + lo[i + 1]),
                                                  o.z + (v[i + 2] + lo[i + 2]), o.w + (v[i + 3] + lo[i + 3]));
                            }
                        }
                    } else if (active) {
                        for (int a = 0; a < C::kAccs && k0 + (a << p.run) < nk; ++a) {
                            float v[K];
                            tmem_ld<K>(tb + a * K, v);
#pragma unroll
                            for (int i = 0; i < K; ++i) sum[i] += v[i];
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&tempty[b]));
                }
                if (!F32 && active)
#pragma unroll
                    for (int i = 0; i < K; i += 4)
                        *reinterpret_cast<float4*>(dst + i) = make_float4(sum[i], sum[i + 1], sum[i + 2], sum[i + 3]);
            }
            if (epi_any(!ok)) break;  // the rows are whole
            if (p.pack == 1) {
                for (int t = 0; t < rows; t += kSR) contract(t, t + kSR < rows ? t + kSR : rows);
            } else {
                for (int j = 0; j < p.pack; ++j) {  // example j of the tile: T <= kSR rows
                    const int64_t e = cur * p.pack + j;
                    if (e >= p.N) break;
                    contract(j * (int)p.T, (j + 1) * (int)p.T);
                    write(e);
                    clear();
                }
            }
            epi_sync();  // the rows are read
            it.next(p, ncl, crank);
            if (p.pack == 1 && it.x != cur) {
                ok = flush(cur);
                clear();
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    cluster_sync();  // no CTA leaves while a peer may still write to it
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)f;
    });
    return fn;
}

// 3-D map over X[N][T][d]: box of one 128-byte row (32 fp32, 64 bf16) x rows x 1 (example),
// 128-byte swizzle, zero fill.
bool make_map(CUtensorMap* tm, const void* X, int64_t N, int64_t T, int64_t d, int rows, bool f32) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const int el = f32 ? 4 : 2;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)T, (cuuint64_t)N};
    cuuint64_t strides[2] = {(cuuint64_t)(d * el), (cuuint64_t)(T * d * el)};
    cuuint32_t box[3] = {(cuuint32_t)(128 / el), (cuuint32_t)rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(X),
               dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int device_sms() {
    static std::atomic<int> sms{0};
    int n = sms.load(std::memory_order_relaxed);
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
        sms.store(n, std::memory_order_relaxed);
    }
    return n;
}

template <int K, bool F32>
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int cs, cudaStream_t s) {
    cfg = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(cs * (device_sms() / cs)));
    cfg.blockDim = dim3(Cfg<K, F32>::kThreads);
    cfg.dynamicSmemBytes = Cfg<K, F32>::kSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// Clusters of cs CTAs that fit the device at once (queried once per device and size).
template <int K, bool F32>
int max_clusters(int cs) {
    static std::atomic<int> cache[64][4];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = -1;
    const int slot = cs >= 8 ? 3 : (cs >= 4 ? 2 : cs - 1);
    if (dev >= 0) {
        const int v = cache[dev][slot].load(std::memory_order_relaxed);
        if (v) return v;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cluster_config<K, F32>(cfg, attr, cs, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, project_flex_kernel<K, F32>, &cfg) != cudaSuccess || n < 1) n = device_sms() / cs;
    if (dev >= 0) cache[dev][slot].store(n, std::memory_order_relaxed);
    return n;
}

// Clocks of a 64-feature chunk, measured over 1 to 700 examples of 20 to 1024 tokens. Here: 4.2 a bf16
// row of the tile (what one SM draws from L2 and HBM), 9 an fp32 row, at least the signs and the
// barriers of a stage, or the splitting of fp32 rows.
// k_project_tc.cu: per 128-row tile, without and with the workspace's equal runs (bal).
template <int K, bool F32>
double chunk_clocks(int R) {
    const double data = R * (F32 ? 9.0 : 4.2), least = F32 ? 800.0 : (K <= 16 ? 430.0 : (K <= 32 ? 460.0 : 590.0));
    return data > least ? data : least;
}
double stream_chunk_clocks(int K, bool bal) { return K >= 64 ? 950.0 : (bal ? 600.0 : 560.0); }
double row_clocks(int K) { return K >= 64 ? 110.0 : (K >= 32 ? 50.0 : 35.0); }  // contraction of a token row
double hbm_clocks(const tda_layer_desc& L, int64_t N, int el, int sms) {        // 22 bytes a clock and SM
    return (double)N * L.T * (L.d_in + L.d_out) * el / (22.0 * sms);
}

// bf16 with k_in = k_out in {16, 32, 64}: whether this kernel's plan beats the streaming kernel of
// k_project_tc.cu. That one takes 128-row tiles, whole examples per CTA, clusters of 2 or 4 below one
// example per SM, or with the workspace (bal) equal runs of tiles. With two tiles a stage (four
// tiles per SM and more) and whole examples or equal runs for every SM it runs at HBM speed and is
// kept. 4096 -> 4096, k = 64: 64 examples of 1024 tokens with the workspace 241 us there and 209 us
// here, 16 of them 84 us there and 114 us here, without the workspace 130 us there.
bool plan_bf16_flex(const tda_layer_desc& L, int64_t N, int sms, double cost, int K, bool bal) {
    const int pack = L.T <= 64 ? (int)(kTileM / L.T) : 1;
    const int64_t slots = (N + pack - 1) / pack, nt = pack > 1 ? 1 : (L.T + kTileM - 1) / kTileM;
    const bool two = slots * nt >= 4 * (int64_t)sms;
    bal = bal && pack == 1;
    if (two && (pack > 1 || bal || N >= sms)) return false;
    int cs = 1;
    if (pack == 1 && N < sms) cs = 2 * N >= sms ? 2 : 4;
    while (cs > nt) cs >>= 1;
    const double chunks = (double)((L.d_in + kChunkK - 1) / kChunkK + (L.d_out + kChunkK - 1) / kChunkK);
    const int64_t room = sms / cs, rounds = (slots + room - 1) / room;
    const double tile = chunks * stream_chunk_clocks(K, bal) + kTileM * row_clocks(K), hbm = hbm_clocks(L, N, 2, sms);
    double stream = bal ? (double)((slots * nt + sms - 1) / sms) * tile + 3000.0
                        : rounds * ((double)((nt + cs - 1) / cs) * tile + (cs > 1 ? 3000.0 : 500.0));
    if (stream < hbm) stream = hbm;
    return cost < 0.97 * stream;
}

struct Plan {
    int R, cs, pack, n_ttiles;
    int64_t slots, clusters;
    double cost;  // clocks
};

// Tile rows and cluster size with the least time of the busiest CTA (its tiles, their contraction, the
// reductions over the cluster), but at least what HBM takes in all; ties go to fewer, larger tiles and
// smaller clusters. T past a multiple of the tile is cut into equal tiles (T = 130: two of 65 rows).
template <int K, bool F32>
Plan plan(const tda_layer_desc& L, int64_t N, int sms) {
    Plan best{};
    const double chunks = (double)((L.d_in + kChunkK - 1) / kChunkK + (L.d_out + kChunkK - 1) / kChunkK);
    const double floor_clk = hbm_clocks(L, N, F32 ? 4 : 2, sms);
    auto consider = [&](int R, int pack, int nt) {
        const double t = chunk_clocks<K, F32>(R);
        const int64_t slots = (N + pack - 1) / pack;
        for (int cs = 1; cs <= 8 && cs <= nt; cs *= 2) {
            const int64_t room = sms / cs, fit = max_clusters<K, F32>(cs) < room ? max_clusters<K, F32>(cs) : room;
            if (fit < 1) continue;
            const int64_t clusters = slots < fit ? slots : fit, rounds = (slots + clusters - 1) / clusters;
            const double tiles = (double)rounds * ((nt + cs - 1) / cs);
            double cost = tiles * (chunks * t + R * row_clocks(K)) + rounds * (cs > 1 ? 3000.0 : 500.0);
            if (cost < floor_clk) cost = floor_clk;
            if (best.R == 0 || cost < best.cost * 0.98) best = Plan{R, cs, pack, nt, slots, clusters, cost};
        }
    };
    if (L.T <= kTileM)
        for (int pack = (int)(kTileM / L.T); pack >= 1; pack >>= 1) {  // whole examples per tile
            const int rows = (int)(pack * L.T);
            consider((rows + 7) / 8 * 8, pack, 1);
        }
    const int64_t nt0 = (L.T + kTileM - 1) / kTileM;
    for (int64_t nt = nt0; nt <= 4 * nt0 && nt < (1 << 24); nt = nt < 2 * nt0 ? nt + (nt0 + 3) / 4 : 2 * nt) {
        const int R = (int)(((L.T + nt - 1) / nt + 7) / 8 * 8);
        consider(R, 1, (int)((L.T + R - 1) / R));
    }
    return best;
}

template <int K, bool F32>
cudaError_t launch_k(const tda_layer_desc& L, const void* A, const void* B, int64_t N, float* phi, int64_t ld_phi,
                     unsigned int* err, cudaStream_t s, bool force, bool bal) {
    constexpr int el = F32 ? 4 : 2;
    const int budget = sm_budget();
    const int sms = budget > 0 && budget < device_sms() ? budget : device_sms();
    cudaError_t e = smem_attr_once<project_flex_kernel<K, F32>>((int)Cfg<K, F32>::kSmem);  // before occupancy queries
    if (e != cudaSuccess) return e;
    const Plan pl = plan<K, F32>(L, N, sms);
    if (!force && !F32 && !plan_bf16_flex(L, N, sms, pl.cost, K, bal)) return cudaErrorNotSupported;
    // packed rows are one [1][N*T][d] view: 32-bit row coordinates, strides below 2^40 bytes
    if (pl.pack > 1) {
        const int64_t d_max = L.d_in > L.d_out ? L.d_in : L.d_out;
        int64_t most = ((int64_t)1 << 30) / L.T;
        const int64_t by_stride = (((int64_t)1 << 40) - 1) / (L.T * d_max * el);
        if (by_stride < most) most = by_stride;
        most = most / 128 * 128;
        if (most < 128) return cudaErrorNotSupported;
        if (N > most) {
            for (int64_t e0 = 0; e0 < N; e0 += most) {
                e = launch_k<K, F32>(L, (const char*)A + e0 * L.T * L.d_in * el, (const char*)B + e0 * L.T * L.d_out * el,
                                     N - e0 < most ? N - e0 : most, phi + e0 * ld_phi, ld_phi, err, s, true, bal);
                if (e != cudaSuccess) return e;
            }
            return cudaSuccess;
        }
    }
    CUtensorMap mA, mB;
    const bool flat = pl.pack > 1;
    if (!make_map(&mA, A, flat ? 1 : N, flat ? N * L.T : L.T, L.d_in, pl.R, F32) ||
        !make_map(&mB, B, flat ? 1 : N, flat ? N * L.T : L.T, L.d_out, pl.R, F32))
        return cudaErrorNotSupported;
    Params p;
    p.N = N;
    p.T = L.T;
    p.ld_phi = ld_phi;
    p.n_slots = pl.slots;
    p.key_in = side_key(L.seed, L.layer, 0);
    p.key_out = side_key(L.seed, L.layer, 1);
    p.scale = projection_scale(L);
    p.phi = phi;
    p.err = err;
    p.R = pl.R;
    p.n_ttiles = pl.n_ttiles;
    p.pack = pl.pack;
    p.k_in = L.k_in;
    p.k_out = L.k_out;
    p.nk_in = (int)((L.d_in + kChunkK - 1) / kChunkK);
    p.nk_out = (int)((L.d_out + kChunkK - 1) / kChunkK);
    p.cs = pl.cs;
    // fp32 and other k: sums of 256 features. k_in = k_out of 16, 32 or 64, which the streaming kernel sums
    // at once: 512, for half of the drains' time.
    p.run = !F32 && L.k_in == L.k_out && L.k_in == K ? 3 : 2;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cluster_config<K, F32>(cfg, attr, pl.cs, s);
    cfg.gridDim = dim3((unsigned)(pl.clusters * pl.cs));
    note_launches(1);
    e = cudaLaunchKernelEx(&cfg, project_flex_kernel<K, F32>, mA, mB, p);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <bool F32>
cudaError_t launch_any(const tda_layer_desc& L, const void* A, const void* B, int64_t N, float* phi, int64_t ld_phi,
                       unsigned int* err, cudaStream_t s, bool force, bool bal) {
    const int k = L.k_in > L.k_out ? L.k_in : L.k_out;
    if (k <= 16) return launch_k<16, F32>(L, A, B, N, phi, ld_phi, err, s, force, bal);
    if (k <= 32) return launch_k<32, F32>(L, A, B, N, phi, ld_phi, err, s, force, bal);
    return launch_k<64, F32>(L, A, B, N, phi, ld_phi, err, s, force, bal);
}

}  // namespace

bool project_flex_supported(const tda_layer_desc& L, tda_dtype dt, const void* A, const void* B) {
    static int sm103 = -1;
    if (sm103 < 0) {
        int dev = 0, major = 0, minor = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
        sm103 = (major == 10 && minor == 3) ? 1 : 0;
    }
    if (!sm103 || !encode_fn() || L.kind != TDA_PROJ_RADEMACHER) return false;
    if (L.k_in < 1 || L.k_out < 1 || L.k_in > 64 || L.k_out > 64) return false;
    const int q = dt == TDA_F32 ? 4 : 8;
    if (L.d_in % q || L.d_out % q || L.T < 1) return false;
    if (((uintptr_t)A & 15) || ((uintptr_t)B & 15)) return false;
    // TMA: 32-bit coordinates, an example's stride below 2^40 bytes
    const int64_t d_max = L.d_in > L.d_out ? L.d_in : L.d_out;
    if (L.T > (1LL << 30) || d_max > (1LL << 30) || L.T * d_max >= (1LL << 38)) return false;
    return true;
}

cudaError_t launch_project_flex(const tda_layer_desc& L, tda_dtype dt, const void* A, const void* B, int64_t N,
                                float* phi, int64_t ld_phi, unsigned int* err, cudaStream_t s, bool force, bool bal) {
    if (N == 0) return cudaSuccess;
    return dt == TDA_F32 ? launch_any<true>(L, A, B, N, phi, ld_phi, err, s, force, bal)
                         : launch_any<false>(L, A, B, N, phi, ld_phi, err, s, force, bal);
}

}  // namespace tda
