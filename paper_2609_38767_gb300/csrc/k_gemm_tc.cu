// k_gemm_tc.cu -- the score GEMM on the 5th-generation tensor cores:
//   S[n][m] = beta * S[n][m] + sum_k Phi[m][k] * Qhat[n][k]
// (gradient inner products between training features Phi and preconditioned
// query features Qhat, Sec. 3.2 / Eq. 4's left side) for fp32 operands.
//
// fp32 accuracy from TF32 tensor cores ("3xTF32"): every operand x is split as
// x = hi + lo with hi = x truncated to TF32 (exact) and lo = x - hi (exact in
// fp32); the product is hi*hi' + hi*lo' + lo*hi', dropping lo*lo' (relative
// size ~2^-22). Each K=8 step therefore issues three tcgen05.mma.kind::tf32.
//
// gemm3t_kernel (below) is the general kernel: persistent, A operand in TMEM. score3x_kernel serves
// products with too few tiles for the chip: a CTA tile of 128 rows of Phi (MMA M, one TMEM lane
// each) x BN query columns (MMA N), a thread-block cluster of cs CTAs splitting K. There lane 0 of
// warp 9 copies the fp32 chunks of both operands with TMA (32 features = one 128-byte row per
// operand row, 128B swizzle: already the K-major operand layout) into the hi tiles of a stage;
// warps 0-3 write lo to the lo tile at the same offset (the fp32 tile itself is the hi operand);
// lane 0 of warp 8 issues the MMAs; warps 4-7 read the accumulators from TMEM. The members'
// partial tiles are summed into the leader CTA over distributed shared memory (deterministic, no
// workspace) before the leader writes S. All waits are bounded (see tc_ptx.cuh).
#include <cuda.h>

#include <mutex>

#include "tda_internal.cuh"

namespace tda {
namespace {

#include "tc_ptx.cuh"

constexpr int kThreads = 320;  // score3x_kernel
constexpr int kBM = 128;       // Phi rows per tile
constexpr int kKC = 32;        // fp32 elements per K chunk (one 128-byte operand row)
constexpr uint32_t kRowBytes = kKC * 4;

template <int BN>
struct GCfg {
    static constexpr int kStages = BN <= 64 ? 4 : (BN <= 128 ? 3 : 2);
    static constexpr uint32_t kABytes = kBM * kRowBytes;   // 16 KiB
    static constexpr uint32_t kBBytes = BN * kRowBytes;
    static constexpr uint32_t kStageBytes = 2 * kABytes + 2 * kBBytes;  // hi and lo of both operands
    // The tensor pipe's fp32 accumulation truncates (about a quarter ulp per addition,
    // always toward zero), so every K chunk (12 additions) goes to the next of kAcc accumulators (all 512 TMEM
    // columns) and the epilogue warps add it into round-to-nearest fp32 registers while the MMAs fill the next
    // ones. 11 x 211 scores of 256 features: 6.7e-7 off, 9.2e-7 with two chunks each (8.6 and 8.3 us).
    static constexpr int kAcc = 512 / BN < 8 ? 512 / BN : 8;
    static constexpr uint32_t kTmemCols = 512;
    static constexpr size_t kSmem =
        1024 + (size_t)kStages * kStageBytes + 8 * (3 * kStages + 2 * kAcc + 3) + 16;  // + barriers, TMEM slot, abort flag
};

struct GParams {
    const float* A;  // Phi, n_t rows
    const float* B;  // Qhat, n_q rows
    float* S;
    int64_t n_t, n_q, K, lda, ldb, ld_S;
    float beta, alpha;     // S = beta * S + alpha * (product); the score uses alpha = 1
    int lower;             // square product (n_t == n_q, BN == kBM): only tiles with m0 <= n0
    int cs, tiles_n;
    int64_t kslice, slab;  // split-K over gridDim.y: K slice per CTA row, S stride per slice (0: no split)
    int splits;            // gridDim.y
    int batched;           // grid z = batch entry: A and B maps are 3-D (z the third coordinate)
    int64_t s_z;           // S element offset between batch entries
    int64_t tiles_z;       // persistent kernel: tiles per batch entry
    int64_t tiles_1;       // of which with the first B (all, without a second product)
    int tiles_n2;          // second product, the same A: its tiles along B, B2 rows, output
    int64_t n_q2, ld_S2, s_z2;
    float* S2;
    int red;               // add to S through TMA (beta = 1; S, its rows and entries 16-byte aligned)
    int nz;                // persistent kernel: batch entries
    int gm;                // persistent kernel: chunks accumulated before they are drained, less one (0 or 1)
    unsigned int* err;
};

// Instruction descriptor, kind::tf32: tf32 A and B (format 2), fp32 D, both K-major.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void split_tf32(float x, float& hi, float& lo) {
    hi = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
    lo = x - hi;
}

// Split a TMA-written fp32 tile: lo = x - hi (hi = x truncated to TF32) goes to
// the lo tile at the same byte offset (the swizzle is the same for both). The
// fp32 tile itself serves as the hi operand: a kind::tf32 MMA reads only the
// upper 19 bits of each element, which is hi exactly, so it is not rewritten.
// 128 threads, one 16-byte group each per pass (conflict-free).
template <uint32_t BYTES>
__device__ __forceinline__ void split_tile(const uint8_t* hi, uint8_t* lo, int pt) {
#pragma unroll 4
    for (uint32_t off = (uint32_t)pt * 16u; off < BYTES; off += 128u * 16u) {
        const float4 v = *reinterpret_cast<const float4*>(hi + off);
        float4 h, l;
        split_tf32(v.x, h.x, l.x);
        split_tf32(v.y, h.y, l.y);
        split_tf32(v.z, h.z, l.z);
        split_tf32(v.w, h.w, l.w);
        *reinterpret_cast<float4*>(lo + off) = l;
    }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
score3x_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GParams p) {
    using C = GCfg<BN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = (uint64_t*)(smem + (size_t)C::kStages * C::kStageBytes);
    uint64_t* full = bars;                   // count 4 (producer warps)
    uint64_t* empty = bars + C::kStages;     // count 1 (MMA commit)
    uint64_t* raw_full = empty + C::kStages; // [kStages] TMA bytes landed (count 1 + tx)
    uint64_t* acc_full = raw_full + C::kStages;  // [kAcc] a chunk is in the accumulator (MMA commit)
    uint64_t* acc_empty = acc_full + C::kAcc;    // [kAcc] the accumulator is drained (count 4)
    uint64_t* red_go = acc_empty + C::kAcc;  // count 1 (leader's remote arrive)
    uint64_t* red_full = red_go + 1;         // count cs-1
    uint64_t* mma_done = red_full + 1;       // count 1
    uint32_t* tmem_slot = (uint32_t*)(mma_done + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) {
            mbar_init(smem_u32(&full[s]), 4);
            mbar_init(smem_u32(&empty[s]), 1);
            mbar_init(smem_u32(&raw_full[s]), 1);
        }
        for (int a = 0; a < C::kAcc; ++a) {
            mbar_init(smem_u32(&acc_full[a]), 1);
            mbar_init(smem_u32(&acc_empty[a]), 4);
        }
        mbar_init(smem_u32(red_go), 1);
        mbar_init(smem_u32(red_full), p.cs > 1 ? p.cs - 1 : 1);
        mbar_init(smem_u32(mma_done), 1);
        *abort = 0;
        fence_mbar_init();
    }
    constexpr int kMmaWarp = 8, kTmaWarp = 9;
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32(tmem_slot), C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const uint32_t crank = cluster_rank();
    const int64_t tile = blockIdx.x / p.cs;
    int64_t m0 = (tile / p.tiles_n) * kBM, n0 = (tile % p.tiles_n) * BN;
    if (p.lower) {
        // tile t of the lower triangle: row tile i (n), column tile j (m) <= i, t = i(i+1)/2 + j
        int64_t i = (int64_t)((sqrtf(8.f * (float)tile + 1.f) - 1.f) * 0.5f);  // fp64 is a slow pipe here
        while (i * (i + 1) / 2 > tile) --i;
        while ((i + 1) * (i + 2) / 2 <= tile) ++i;
        n0 = i * BN;
        m0 = (tile - i * (i + 1) / 2) * kBM;
    }
    // split-K slice z covers features [z*kslice, z*kslice + Kz) and writes its own slab of S
    const int64_t kbase = (int64_t)blockIdx.y * p.kslice;
    const int64_t Kz = p.kslice ? ((p.K - kbase) < p.kslice ? (p.K - kbase) : p.kslice) : p.K;
    float* Sz = p.S + (int64_t)blockIdx.y * p.slab + (int64_t)blockIdx.z * p.s_z;
    const int zc = (int)blockIdx.z;
    const int64_t nkc = (Kz + kKC - 1) / kKC;
    const int64_t per = (nkc + p.cs - 1) / p.cs;
    const int64_t kc0 = crank * per, kc1 = (kc0 + per) < nkc ? (kc0 + per) : nkc;

    if (warp < 4) {
        // ---------------- split warps: raw fp32 (TMA) -> hi in place + lo
        const int pt = threadIdx.x;
        uint32_t it = 0;
        for (int64_t kc = kc0; kc < kc1; ++kc, ++it) {
            const int s = it % C::kStages;
            const uint32_t ph = (it / C::kStages) & 1u;
            bool got = warp_wait(smem_u32(&raw_full[s]), ph, abort, p.err);
            if (!got) break;
            uint8_t* st = smem + (size_t)s * C::kStageBytes;
            split_tile<C::kABytes>(st, st + C::kABytes, pt);
            split_tile<C::kBBytes>(st + 2 * C::kABytes, st + 2 * C::kABytes + C::kBBytes, pt);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&full[s]));
        }
    }
    if (warp == kTmaWarp && lane == 0) {
        // ---------------- TMA producer: fp32 chunks of Phi rows m0.. and Qhat rows n0..
        // (features past the slice end belong to the next slice only when the slice
        // is not the last; slices are multiples of 32 features, so no chunk crosses one)
        uint32_t it = 0, last_par[C::kStages];
        bool issued[C::kStages];
        for (int s = 0; s < C::kStages; ++s) issued[s] = false;
        for (int64_t kc = kc0; kc < kc1; ++kc, ++it) {
            const int s = it % C::kStages;
            const uint32_t ph = (it / C::kStages) & 1u;
            if (!wait_bounded(smem_u32(&empty[s]), ph ^ 1u, abort, p.err)) break;
            const uint32_t st = smem_u32(smem + (size_t)s * C::kStageBytes), bar = smem_u32(&raw_full[s]);
            const int k = (int)(kbase + kc * kKC);
            mbar_arrive_tx(bar, C::kABytes + C::kBBytes);
            if (p.batched) {
                tma_load_3d(st, &tmA, k, (int)m0, zc, bar);
                tma_load_3d(st + 2 * C::kABytes, &tmB, k, (int)n0, zc, bar);
            } else {
                tma_load_2d(st, &tmA, k, (int)m0, bar);
                tma_load_2d(st + 2 * C::kABytes, &tmB, k, (int)n0, bar);
            }
            issued[s] = true;
            last_par[s] = ph;
        }
        // copies still in flight when the consumers stopped early land before the CTA exits
        for (int s = 0; s < C::kStages; ++s)
            if (issued[s]) {
                const uint64_t t0 = global_ns();
                while (!mbar_try_wait(smem_u32(&raw_full[s]), last_par[s]))
                    if (global_ns() - t0 > kTimeoutNs) {
                        atomicOr(p.err, kErrTimeout);
                        break;
                    }
            }
    }
    if (warp == kMmaWarp) {
        // ---------------- MMA issuer: the warp waits, one lane issues
        const uint32_t idesc = idesc_tf32(kBM, BN);
        uint32_t it = 0;
        for (int64_t kc = kc0; kc < kc1; ++kc, ++it) {
            const int s = it % C::kStages;
            const uint32_t ph = (it / C::kStages) & 1u;
            const uint32_t a = it % C::kAcc;  // this chunk's accumulator
            if (!warp_wait(smem_u32(&acc_empty[a]), ((it / C::kAcc) & 1u) ^ 1u, abort, p.err)) break;
            if (!warp_wait(smem_u32(&full[s]), ph, abort, p.err)) break;
            tc_fence_after();
            const uint32_t st = smem_u32(smem + (size_t)s * C::kStageBytes);
            const uint64_t ahi = sw128_desc(st), alo = sw128_desc(st + C::kABytes);
            const uint64_t bhi = sw128_desc(st + 2 * C::kABytes), blo = sw128_desc(st + 2 * C::kABytes + C::kBBytes);
            const uint32_t d = tmem + a * BN;
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < kKC / 8; ++k) {  // K = 8 tf32 = 32 bytes per instruction
                    mma_tf32(d, ahi + 2 * k, bhi + 2 * k, idesc, k == 0 ? 0u : 1u);
                    mma_tf32(d, ahi + 2 * k, blo + 2 * k, idesc, 1u);
                    mma_tf32(d, alo + 2 * k, bhi + 2 * k, idesc, 1u);
                }
                mma_commit(smem_u32(&empty[s]));
                mma_commit(smem_u32(&acc_full[a]));
            }
            __syncwarp();
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
    }
    __syncwarp();
    if (warp >= 4 && warp < 8) {
        // ---------------- epilogue: TMEM chunks -> registers -> (cluster reduction) -> S
        const int q = warp & 3;
        const int row = q * 32 + lane;  // Phi row within the tile
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16);
        const uint32_t groups = kc1 > kc0 ? (uint32_t)(kc1 - kc0) : 0u;
        float acc[BN];
#pragma unroll
        for (int c = 0; c < BN; ++c) acc[c] = 0.f;
        bool got = true;
        for (uint32_t g = 0; g < groups; ++g) {
            const uint32_t a = g % C::kAcc;
            got = warp_wait(smem_u32(&acc_full[a]), (g / C::kAcc) & 1u, abort, p.err);
            if (!got) break;
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < BN; c0 += 16) {
                float v[16];
                tmem_ld16(tbase + a * BN + c0, v);
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[c0 + i] += v[i];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[a]));
        }
        if (!epi_any(!got)) {
            bool ok = true;
            if (p.cs > 1) {
                // partial tiles of members 1..cs-1 land in the leader's stage buffers
                float* red = (float*)smem;
                const uint32_t slot = smem_u32(red) + (uint32_t)(row * BN) * 4u;
                if (crank == 0) {
                    if (threadIdx.x == 128)
                        for (int r = 1; r < p.cs; ++r) mbar_arrive_remote(smem_u32(red_go), (uint32_t)r);
                    bool g2 = true;
                    if (lane == 0) g2 = wait_bounded_cluster(smem_u32(red_full), 0, abort, p.err);
                    g2 = __shfl_sync(0xffffffffu, g2, 0);
                    ok = !epi_any(!g2);
                    if (ok)
                        for (int r = 1; r < p.cs; ++r) {
                            const float* part = red + (size_t)(r - 1) * kBM * BN + (size_t)row * BN;
#pragma unroll
                            for (int c = 0; c < BN; c += 4) {
                                const float4 v = *reinterpret_cast<const float4*>(part + c);
                                acc[c] += v.x;
                                acc[c + 1] += v.y;
                                acc[c + 2] += v.z;
                                acc[c + 3] += v.w;
                            }
                        }
                } else {
                    bool g2 = true;
                    if (lane == 0) g2 = wait_bounded_cluster(smem_u32(red_go), 0, abort, p.err);
                    g2 = __shfl_sync(0xffffffffu, g2, 0);
                    ok = !epi_any(!g2);
                    if (ok) {
                        const uint32_t dst = map_rank(slot, 0) + (crank - 1) * (uint32_t)(kBM * BN) * 4u;
#pragma unroll
                        for (int c = 0; c < BN; ++c) st_cluster_f32(dst + (uint32_t)c * 4u, acc[c]);
                        fence_acq_rel_cluster();
                        epi_sync();
                        if (threadIdx.x == 128) mbar_arrive_remote(smem_u32(red_full), 0u);
                    }
                    ok = false;  // members write nothing to S
                }
            }
            if (ok) {
                const int64_t m = m0 + row;
                if (m < p.n_t) {
                    if (p.beta == 0.f) {
#pragma unroll
                        for (int c = 0; c < BN; ++c) {
                            const int64_t n = n0 + c;
                            if (n < p.n_q) Sz[n * p.ld_S + m] = p.alpha * acc[c];
                        }
                    } else {
                        // the previous values of 16 columns are loaded before any is stored, so
                        // the loads are in flight together instead of one round trip per column
#pragma unroll
                        for (int c0 = 0; c0 < BN; c0 += 16) {
                            float old[16];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int64_t n = n0 + c0 + i;
                                old[i] = n < p.n_q ? __ldcg(Sz + n * p.ld_S + m) : 0.f;
                            }
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const int64_t n = n0 + c0 + i;
                                if (n < p.n_q) Sz[n * p.ld_S + m] = p.beta * old[i] + p.alpha * acc[c0 + i];
                            }
                        }
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, C::kTmemCols);
    }
    cluster_sync();
}

// ---------------------------------------------------------------------------
// The same product without a split of K, and the Fisher fit, with the A operand in TMEM: persistent
// CTAs, one per SM, walk the tiles of all batch entries and feature slices. With PAIR the two CTAs
// of a cluster share a tile of 256 rows of A x BN rows of B (cta_group::2): each has its own 128
// rows of A and of the accumulators, and half of B.
//
// What bounds a tile: three TF32 products of 32 features take 768 clocks (BN = 128). At 128 bytes a
// clock, shared memory with both operands there takes 1536 (768 of operand reads, 256 of TMA
// writes, 512 of splitting), with A in TMEM and one CTA 1152, and a pair needs 700. The rest is
// latency, a chain of waits per chunk in every role. One lane polling and then a shuffle took about
// 250 clocks a wait, and MMAs issued behind `lane == 0` about 80 clocks each (1000 a chunk, the
// bound of the whole kernel), so whole warps poll and an elected lane issues. A chunk now takes
// 980 clocks (scores) to 1040 (fit), one CTA a tile 1290 and 1080.
//
// FIT: M_l += Phi_l^T Phi_l, lower triangle, layer l's features at column l*D of each row of Phi.
// The operands are features x examples, K-major, but Phi holds examples x features, so a chunk
// is 32 examples in boxes of 32 features (128-byte swizzle). A: a lane per feature, 32 lanes on one
// 128-byte row. B: a lane per example, 16 bytes of features a load, 4-byte stores of 32 lanes into
// one row of the operand. All of these are free of bank conflicts. A's rows are columns of
// M, so that a warp's 32 lanes are 32 neighbouring entries of a row of M.
//
// A's hi is the fp32 value as it is (a kind::tf32 MMA reads its upper 19 bits).
//
// Accuracy: the tensor pipe's fp32 accumulation rounds toward zero, so a long same-sign sum (a
// diagonal entry of M) drifts low by up to an ulp per accumulate. Groups of two chunks (24 accumulates; scores
// of up to 384 features: one) alternate between two accumulators, and eight epilogue warps (two per TMEM lane
// quadrant, half of the columns each) add every finished group into round-to-nearest registers
// beside the next group's MMAs, then write the tile beside the next tile's.
//
// RED: S += alpha * product with TMA reductions from shared memory (one rounding, as in registers).
// For products of few features, whose epilogue's loads of the old values took longer than the
// MMAs: the rank-256 updates of 7 x 4096 rows take 49 us on average, 101 us before. L2 flushes subnormal sums, so the fit
// and the scores keep the loads.
//
// Measured: scores of 256 x 8192, 7168 features: 205 us with both operands in shared memory and one
// pass over the accumulators (1.3e-5 off), 188 us with A in TMEM (9e-7 off), 114 us in pairs.
// Fit of seven layers of D = 4096, 8192 examples: 6.74 ms, 6.24 ms, 3.61 ms.
//
// Warps: 0-3 A into TMEM, 4-7 B's hi and lo into the operand slots, 8-15 epilogue, 16 MMA issuer (of
// the pair: in CTA 0), 17 TMA. Every wait is bounded.
constexpr int kThreadsT = 18 * 32;

template <int BN, bool PAIR, bool RED = false>
struct TCfg {
    static constexpr int kCtas = PAIR ? 2 : 1;
    static constexpr int kBRows = BN / kCtas;             // rows of B in this CTA
    static constexpr uint32_t kABytes = kBM * kRowBytes;  // 16 KiB
    static constexpr uint32_t kBBytes = kBRows * kRowBytes;
    static constexpr uint32_t kRawBytes = kABytes + kBBytes;
    static constexpr int kRaw = PAIR && !RED ? 6 : 4;     // raw chunks
    static constexpr int kSlots = PAIR ? 4 : 3;           // A in TMEM, B's hi and lo in shared memory
    static constexpr uint32_t kSlotBytes = 2 * kBBytes;
    static constexpr int kCols = BN / 2;                  // columns per epilogue thread
    static constexpr int kAOff = 2 * BN;                  // first TMEM column of A: [slot][hi 32 | lo 32]
    static constexpr size_t kOutOff = (size_t)kRaw * kRawBytes + (size_t)kSlots * kSlotBytes;
    static constexpr uint32_t kOutBytes = kCols * 128;    // RED: kCols rows of 32 output columns, per epilogue warp
    static constexpr size_t kBarOff = kOutOff + (RED ? 8 * kOutBytes : 0);
    static constexpr size_t kSmem = 1024 + kBarOff + 8 * (2 * kRaw + 2 * kSlots + 5) + 16;
    static_assert(kAOff + kSlots * 64 <= 512 && kSmem <= 232448, "TMEM columns, shared memory");
};

// D[tmem] (+)= A[tmem] * B[smem]^T, tf32 inputs.
template <bool PAIR>
__device__ __forceinline__ void mma_tf32_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    if constexpr (PAIR)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::tf32 [%0], [%1], %2, %3, p;\n}" ::"r"(
                d_tmem),
            "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}" ::"r"(
                d_tmem),
            "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
}

// Tile t: first rows m0 (of A, this CTA's) and n0 (of B), batch entry z, feature slice y.
struct TileAt {
    int64_t m0, n0;
    int z, y;
    bool second;
};
template <int BN, bool PAIR>
__device__ __forceinline__ TileAt tile_at(const GParams& p, int64_t t, uint32_t rank) {
    TileAt a;
    const int64_t per_z = p.tiles_z * p.splits;
    a.z = (int)(t / per_z);
    t -= (int64_t)a.z * per_z;
    a.y = (int)(t / p.tiles_z);
    const int64_t tile = t - (int64_t)a.y * p.tiles_z;
    a.second = PAIR && tile >= p.tiles_1;
    if (a.second) {
        a.m0 = (tile - p.tiles_1) / p.tiles_n2 * (2 * kBM);
        a.n0 = (tile - p.tiles_1) % p.tiles_n2 * BN;
    } else if (p.lower && PAIR) {
        // row tiles 2q and 2q + 1 of B have q + 1 tiles of A each
        int64_t q = (int64_t)(sqrtf((float)tile + 0.25f) - 0.5f);
        while (q * (q + 1) > tile) --q;
        while ((q + 1) * (q + 2) <= tile) ++q;
        const int64_t r = tile - q * (q + 1), odd = r >= q + 1 ? 1 : 0;
        a.n0 = (2 * q + odd) * BN;
        a.m0 = (r - odd * (q + 1)) * 2 * kBM;
    } else if (p.lower) {
        int64_t i = (int64_t)((sqrtf(8.f * (float)tile + 1.f) - 1.f) * 0.5f);
        while (i * (i + 1) / 2 > tile) --i;
        while ((i + 1) * (i + 2) / 2 <= tile) ++i;
        a.n0 = i * BN;
        a.m0 = (tile - i * (i + 1) / 2) * kBM;
    } else {
        a.m0 = (tile / p.tiles_n) * (PAIR ? 2 * kBM : kBM);
        a.n0 = (tile % p.tiles_n) * BN;
    }
    a.m0 += rank * kBM;
    return a;
}
// 32-feature chunks of slice y
__device__ __forceinline__ int64_t chunks_of(const GParams& p, int y) {
    const int64_t kbase = (int64_t)y * p.kslice;
    const int64_t Kz = p.kslice ? ((p.K - kbase) < p.kslice ? (p.K - kbase) : p.kslice) : p.K;
    return (Kz + kKC - 1) / kKC;
}

template <int BN, bool PAIR, bool FIT, bool RED>
__global__ void __launch_bounds__(kThreadsT, 1)
gemm3t_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmS,
              const __grid_constant__ CUtensorMap tmS2, const GParams p) {
    using C = TCfg<BN, PAIR, RED>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* slots = smem + (size_t)C::kRaw * C::kRawBytes;
    uint64_t* raw_full = (uint64_t*)(smem + C::kBarOff);  // [kRaw] TMA bytes landed (count 1 + tx)
    uint64_t* raw_empty = raw_full + C::kRaw;             // [kRaw] chunk read (8 warps)
    uint64_t* ready = raw_empty + C::kRaw;                // [kSlots] operands written (8 warps a CTA; CTA 0's)
    uint64_t* empty = ready + C::kSlots;                  // [kSlots] MMAs done reading (count 1)
    uint64_t* acc_full = empty + C::kSlots;               // [2] a group is accumulated (count 1)
    uint64_t* acc_empty = acc_full + 2;                   // [2] the accumulator is drained (8 warps a CTA; CTA 0's)
    uint64_t* mma_done = acc_empty + 2;
    uint32_t* tmem_slot = (uint32_t*)(mma_done + 1);
    volatile int* abort = (volatile int*)(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    if (threadIdx.x == 0) {
        for (int r = 0; r < C::kRaw; ++r) {
            mbar_init(smem_u32(&raw_full[r]), 1);
            mbar_init(smem_u32(&raw_empty[r]), 8);
        }
        for (int s = 0; s < C::kSlots; ++s) {
            mbar_init(smem_u32(&ready[s]), 8 * C::kCtas);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), 8 * C::kCtas);
        }
        mbar_init(smem_u32(mma_done), 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == 16) {
        if constexpr (PAIR) {
            tmem_alloc2(smem_u32(tmem_slot), 512);
        } else {
            tmem_alloc(smem_u32(tmem_slot), 512);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const int64_t total = p.tiles_z * p.splits * p.nz;
    const int64_t t0 = PAIR ? blockIdx.x >> 1 : blockIdx.x, tstep = PAIR ? gridDim.x >> 1 : gridDim.x;

    if (warp < 8) {
        // ---------------- split warps: 0-3 A's rows into TMEM, 4-7 B's hi and lo into shared memory
        uint32_t it = 0;
        bool ok = true;
        for (int64_t t = t0; ok && t < total; t += tstep) {
            const int64_t nkc = chunks_of(p, tile_at<BN, PAIR>(p, t, rank).y);
            for (int64_t kc = 0; kc < nkc; ++kc, ++it) {
                const uint32_t r = it % C::kRaw, rph = (it / C::kRaw) & 1u;
                const uint32_t s = it % C::kSlots, ph = (it / C::kSlots) & 1u;
                if (!warp_wait(smem_u32(&raw_full[r]), rph, abort, p.err)) {
                    ok = false;
                    break;
                }
                const uint8_t* raw = smem + (size_t)r * C::kRawBytes;
                auto release = [&]() {  // the raw chunk is in registers; wait for the slot
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&raw_empty[r]));
                    return warp_wait(smem_u32(&empty[s]), ph ^ 1u, abort, p.err);
                };
                if (warp < 4) {
                    uint32_t x[32];
                    if constexpr (FIT) {
                        const uint8_t* box = raw + (uint32_t)warp * 4096u + (lane & 3) * 4;
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            x[e] = *reinterpret_cast<const uint32_t*>(box + e * kRowBytes + (((lane >> 2) ^ (e & 7)) << 4));
                    } else {
                        const int row = warp * 32 + lane;
                        const uint8_t* src = raw + (uint32_t)row * kRowBytes;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            const uint4 v = *reinterpret_cast<const uint4*>(src + ((c ^ (row & 7)) << 4));
                            x[4 * c] = v.x, x[4 * c + 1] = v.y, x[4 * c + 2] = v.z, x[4 * c + 3] = v.w;
                        }
                    }
                    if (!release()) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t dst = tmem + ((uint32_t)(warp * 32) << 16) + C::kAOff + s * 64u;
                    tmem_st16(dst, x);
                    tmem_st16(dst + 16, x + 16);
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        float h, l;
                        split_tf32(__uint_as_float(x[e]), h, l);
                        x[e] = __float_as_uint(l);
                    }
                    tmem_st16(dst + 32, x);
                    tmem_st16(dst + 48, x + 16);
                    tmem_wait_st();
                    tc_fence_before();
                } else {
                    constexpr int kPer = C::kBRows / 16;  // 16-byte groups a thread
                    const int pt = threadIdx.x - 128, w = warp - 4;
                    const uint8_t* src = raw + C::kABytes;
                    float4 v[kPer];
                    if constexpr (FIT) {
                        // warp w: features kBRows / 4 * w ..., lane: example
                        const uint8_t* row = src + (uint32_t)(w * kPer / 8) * 4096u + (uint32_t)lane * kRowBytes;
#pragma unroll
                        for (int j = 0; j < kPer; ++j)
                            v[j] = *reinterpret_cast<const float4*>(row + (((j + w * kPer % 8) ^ (lane & 7)) << 4));
                    } else {
#pragma unroll
                        for (int j = 0; j < kPer; ++j)
                            v[j] = *reinterpret_cast<const float4*>(src + (uint32_t)(pt + 128 * j) * 16u);
                    }
                    if (!release()) {
                        ok = false;
                        break;
                    }
                    uint8_t* hi = slots + (size_t)s * C::kSlotBytes;
                    uint8_t* lo = hi + C::kBBytes;
#pragma unroll
                    for (int j = 0; j < kPer; ++j) {
                        const float in[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
                        float h, l[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) split_tf32(in[i], h, l[i]);
                        if constexpr (FIT) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int fr = 4 * (kPer * w + j) + i;  // feature row of the operand
                                const uint32_t off =
                                    (uint32_t)fr * kRowBytes + (uint32_t)((((lane >> 2) ^ (fr & 7)) << 4) + (lane & 3) * 4);
                                *reinterpret_cast<float*>(hi + off) = in[i];
                                *reinterpret_cast<float*>(lo + off) = l[i];
                            }
                        } else {
                            const uint32_t off = (uint32_t)(pt + 128 * j) * 16u;
                            *reinterpret_cast<float4*>(hi + off) = v[j];
                            *reinterpret_cast<float4*>(lo + off) = make_float4(l[0], l[1], l[2], l[3]);
                        }
                    }
                    fence_proxy_async();
                }
                __syncwarp();
                if (lane == 0) arrive_leader<PAIR>(smem_u32(&ready[s]));
            }
        }
        if (PAIR && ok && threadIdx.x == 0)
            // every arrival of the pair's MMAs on this CTA's barriers lands before it exits
            for (uint32_t k = it > (uint32_t)C::kSlots ? it - C::kSlots : 0u; k < it; ++k)
                if (!wait_bounded(smem_u32(&empty[k % C::kSlots]), (k / C::kSlots) & 1u, abort, p.err)) break;
    } else if (warp < 16) {
        // ---------------- epilogue: groups -> registers -> S
        const int q4 = warp & 3, half = (warp - 8) >> 2, row = q4 * 32 + lane;
        const uint32_t tbase = tmem + ((uint32_t)(q4 * 32) << 16) + half * C::kCols;
        uint32_t cnt = 0;
        bool got = true;
        for (int64_t t = t0; got && t < total; t += tstep) {
            const TileAt at = tile_at<BN, PAIR>(p, t, rank);
            const uint32_t groups = (uint32_t)((chunks_of(p, at.y) + p.gm) >> p.gm);
            const int64_t m = at.m0 + row, nb = at.n0 + half * C::kCols;
            // (the upper half of a pair's tile on the diagonal lies above it)
            const bool write = !(PAIR && p.lower && !at.second && at.m0 > at.n0);
            float* Sz = (at.second ? p.S2 + (int64_t)at.z * p.s_z2 : p.S + (int64_t)at.y * p.slab + (int64_t)at.z * p.s_z) + m;
            const int64_t ld_S = at.second ? p.ld_S2 : p.ld_S, n_q = at.second ? p.n_q2 : p.n_q;
            const int lim = (int)(n_q - nb < C::kCols ? n_q - nb : C::kCols);
            // the previous values start on their way to L2: short products (256 features) end before
            // HBM has answered. A warp's 32 values of a column are one or two lines.
            if (!RED && p.beta != 0.f && write)
#pragma unroll
                for (int c = lane; c < C::kCols; c += 32)
                    if (c < lim && at.m0 + q4 * 32 < p.n_t)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(Sz - lane + (nb + c) * ld_S));
            float acc[C::kCols];
#pragma unroll
            for (int c = 0; c < C::kCols; ++c) acc[c] = 0.f;
            for (uint32_t g = 0; g < groups; ++g, ++cnt) {
                const uint32_t b = cnt & 1u;
                got = warp_wait(smem_u32(&acc_full[b]), (cnt >> 1) & 1u, abort, p.err);
                if (!got) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < C::kCols; c0 += 16) {
                    float v[16];
                    tmem_ld16(tbase + b * BN + c0, v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) acc[c0 + i] += v[i];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_leader<PAIR>(smem_u32(&acc_empty[b]));
            }
            if constexpr (RED) {
                if (!got || !write || at.m0 + q4 * 32 >= p.n_t || lim <= 0) continue;
                uint8_t* out = smem + C::kOutOff + (size_t)(warp - 8) * C::kOutBytes;
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the last tile has left
                __syncwarp();
#pragma unroll
                for (int c = 0; c < C::kCols; ++c) *reinterpret_cast<float*>(out + c * 128 + lane * 4) = p.alpha * acc[c];
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    asm volatile(
                        "cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                            (uint64_t)(at.second ? &tmS2 : &tmS)),
                        "r"((int)at.m0 + q4 * 32), "r"((int)nb), "r"(at.z), "r"(smem_u32(out))
                        : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                continue;
            }
            if (!got || m >= p.n_t || !write) continue;
            if (p.beta == 0.f) {
#pragma unroll
                for (int c = 0; c < C::kCols; ++c)
                    if (c < lim) Sz[(nb + c) * ld_S] = p.alpha * acc[c];
            } else {
                // 8 previous values are on their way together
#pragma unroll
                for (int c0 = 0; c0 < C::kCols; c0 += 8) {
                    float old[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) old[i] = c0 + i < lim ? __ldcg(Sz + (nb + c0 + i) * ld_S) : 0.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (c0 + i < lim) Sz[(nb + c0 + i) * ld_S] = p.beta * old[i] + p.alpha * acc[c0 + i];
                }
            }
        }
        if (RED && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else if (warp == 17 && lane == 0) {
        // ---------------- TMA producer
        uint32_t it = 0, last_par[C::kRaw];
        bool issued[C::kRaw], ok = true;
        for (int r = 0; r < C::kRaw; ++r) issued[r] = false;
        for (int64_t t = t0; ok && t < total; t += tstep) {
            const TileAt at = tile_at<BN, PAIR>(p, t, rank);
            const int64_t nkc = chunks_of(p, at.y);
            const int64_t kbase = (int64_t)at.y * p.kslice;
            const int m0 = (int)at.m0, n0 = (int)at.n0 + (int)rank * C::kBRows;
            for (int64_t kc = 0; kc < nkc; ++kc, ++it) {
                const uint32_t r = it % C::kRaw, ph = (it / C::kRaw) & 1u;
                if (!wait_bounded(smem_u32(&raw_empty[r]), ph ^ 1u, abort, p.err)) {
                    ok = false;
                    break;
                }
                const uint32_t st = smem_u32(smem + (size_t)r * C::kRawBytes), bar = smem_u32(&raw_full[r]);
                const int k = (int)(kbase + kc * kKC);
                mbar_arrive_tx(bar, C::kRawBytes);
                if constexpr (FIT) {
                    const int x = (int)(at.z * p.n_t);
#pragma unroll
                    for (int b = 0; b < kBM / 32; ++b) tma_load_2d(st + 4096u * b, &tmA, x + m0 + 32 * b, k, bar);
#pragma unroll
                    for (int b = 0; b < C::kBRows / 32; ++b)
                        tma_load_2d(st + C::kABytes + 4096u * b, &tmA, x + n0 + 32 * b, k, bar);
                } else if (p.batched) {
                    tma_load_3d(st, &tmA, k, m0, at.z, bar);
                    tma_load_3d(st + C::kABytes, at.second ? &tmB2 : &tmB, k, n0, at.z, bar);
                } else {
                    tma_load_2d(st, &tmA, k, m0, bar);
                    tma_load_2d(st + C::kABytes, at.second ? &tmB2 : &tmB, k, n0, bar);
                }
                issued[r] = true;
                last_par[r] = ph;
            }
        }
        // copies still in flight when the consumers stopped early land before the CTA exits
        for (int r = 0; r < C::kRaw; ++r)
            if (issued[r]) {
                const uint64_t ns = global_ns();
                while (!mbar_try_wait(smem_u32(&raw_full[r]), last_par[r]))
                    if (global_ns() - ns > kTimeoutNs) {
                        atomicOr(p.err, kErrTimeout);
                        break;
                    }
            }
    } else if (warp == 16 && rank == 0) {
        // ---------------- MMA issuer: the warp waits, one lane issues
        constexpr uint32_t idesc = idesc_tf32(kBM * C::kCtas, BN);
        uint32_t it = 0, cnt = 0;
        bool ok = true;
        for (int64_t t = t0; ok && t < total; t += tstep) {
            const int nkc = (int)chunks_of(p, tile_at<BN, PAIR>(p, t, rank).y);
            for (int kc = 0; kc < nkc; ++kc, ++it) {
                const uint32_t s = it % C::kSlots, ph = (it / C::kSlots) & 1u, b = cnt & 1u;
                const bool start = (kc & p.gm) == 0, last = (kc & p.gm) == p.gm || kc == nkc - 1;
                if ((start && !warp_wait(smem_u32(&acc_empty[b]), ((cnt >> 1) & 1u) ^ 1u, abort, p.err)) ||
                    !warp_wait(smem_u32(&ready[s]), ph, abort, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t st = smem_u32(slots + (size_t)s * C::kSlotBytes);
                const uint32_t ahi = tmem + C::kAOff + s * 64u, alo = ahi + 32u, d = tmem + b * BN;
                const uint64_t bhi = sw128_desc(st), blo = sw128_desc(st + C::kBBytes);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kKC / 8; ++k) {  // K = 8 tf32: 8 TMEM columns, 32 bytes of shared memory
                        mma_tf32_ta<PAIR>(d, ahi + 8 * k, bhi + 2 * k, idesc, start && k == 0 ? 0u : 1u);
                        mma_tf32_ta<PAIR>(d, ahi + 8 * k, blo + 2 * k, idesc, 1u);
                        mma_tf32_ta<PAIR>(d, alo + 8 * k, bhi + 2 * k, idesc, 1u);
                    }
                    commit_all<PAIR>(smem_u32(&empty[s]));
                    if (last) commit_all<PAIR>(smem_u32(&acc_full[b]));
                }
                __syncwarp();
                cnt += last;
            }
        }
        if (elect_one()) {
            if constexpr (PAIR)
                commit_pair_local(smem_u32(mma_done));
            else
                mma_commit(smem_u32(mma_done));
            const uint64_t ns = global_ns();
            while (!mbar_try_wait(smem_u32(mma_done), 0))
                if (global_ns() - ns > kTimeoutNs) {
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
        }
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    if (warp == 16) {
        tc_fence_after();
        if constexpr (PAIR)
            tmem_dealloc2(tmem, 512);
        else
            tmem_dealloc(tmem, 512);
    }
}

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

// 2-D map over fp32 X[rows][ld] (features 0..K-1 used): box 32 features x box_rows rows,
// 128-byte swizzle, zero fill past K and past the last row.
bool make_map_f32(CUtensorMap* tm, const float* X, int64_t rows, int64_t K, int64_t ld, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 4)};
    cuuint32_t box[2] = {(cuuint32_t)kKC, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(X), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D map over nz batch entries of fp32 X[rows][ld] (features 0..K-1 used), entry z at byte
// offset z * z_bytes from X; box 32 features x box_rows rows x 1 entry, 128-byte swizzle.
bool make_map_f32_3d(CUtensorMap* tm, const float* X, int64_t rows, int64_t K, int64_t ld, int64_t nz,
                     size_t z_bytes, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)nz};
    cuuint64_t strides[2] = {(cuuint64_t)(ld * 4), (cuuint64_t)z_bytes};
    cuuint32_t box[3] = {(cuuint32_t)kKC, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(X), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 256 x 128 tiles that hold the 128 x 128 tiles of a lower triangle of nt x nt
int64_t pair_lower_tiles(int64_t nt) {
    const int64_t q = nt / 2;
    return nt & 1 ? (q + 1) * (q + 1) : q * (q + 1);
}

template <int BN, bool FIT, bool RED>
cudaError_t launch_pairs(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmB2, const CUtensorMap& tmS,
                         const CUtensorMap& tmS2, const GParams& p, int sms, cudaStream_t s) {
    using T = TCfg<BN, true, RED>;
    cudaError_t e = smem_attr_once<gemm3t_kernel<BN, true, FIT, RED>>((int)T::kSmem);
    if (e != cudaSuccess) return e;
    const int64_t total = p.tiles_z * p.splits * p.nz, half = sms > 1 ? sms / 2 : 1;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(2 * (total < half ? total : half)));
    cfg.blockDim = dim3(kThreadsT);
    cfg.dynamicSmemBytes = T::kSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launches(1);
    e = cudaLaunchKernelEx(&cfg, gemm3t_kernel<BN, true, FIT, RED>, tmA, tmB, tmB2, tmS, tmS2, p);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// 3-D map over nz outputs fp32 S[rows][ld] (columns 0..cols-1), entry z s_z floats from the last; box
// 32 columns x box_rows rows, no swizzle.
bool make_map_out(CUtensorMap* tm, float* S, int64_t rows, int64_t cols, int64_t ld, int64_t nz, int64_t s_z,
                  int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)nz};
    cuuint64_t strides[2] = {(cuuint64_t)(ld * 4), (cuuint64_t)((nz > 1 ? s_z : ld) * 4)};
    cuuint32_t box[3] = {32, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, S, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN>
cudaError_t launch_bn(GParams p, cudaStream_t s, int64_t nz = 1, size_t a_z_bytes = 0, size_t b_z_bytes = 0,
                      const GemmSecond* second = nullptr) {
    using C = GCfg<BN>;
    CUtensorMap tmA, tmB;
    if (nz > 1) {
        if (!make_map_f32_3d(&tmA, p.A, p.n_t, p.K, p.lda, nz, a_z_bytes, kBM) ||
            !make_map_f32_3d(&tmB, p.B, p.n_q, p.K, p.ldb, nz, b_z_bytes, BN))
            return cudaErrorInvalidValue;
        p.batched = 1;
    } else if (!make_map_f32(&tmA, p.A, p.n_t, p.K, p.lda, kBM) || !make_map_f32(&tmB, p.B, p.n_q, p.K, p.ldb, BN)) {
        return cudaErrorInvalidValue;
    }
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    const int64_t tiles_m = (p.n_t + kBM - 1) / kBM, tiles_n = (p.n_q + BN - 1) / BN;
    const int64_t tiles = p.lower ? tiles_n * (tiles_n + 1) / 2 : tiles_m * tiles_n;
    const int64_t nkc = ((p.kslice ? p.kslice : p.K) + kKC - 1) / kKC;
    int cs = 1;
    // split K over a cluster only while the tiles of all batch entries leave SMs idle
    while (!second && cs < 4 && tiles * p.splits * nz * cs * 2 <= sms && nkc >= 8 * cs * 2) cs *= 2;
    // the leader's stage buffers must hold the members' partial tiles
    while (cs > 1 && (size_t)(cs - 1) * kBM * BN * 4 > (size_t)C::kStages * C::kStageBytes) cs >>= 1;
    p.cs = cs;
    p.tiles_n = (int)tiles_n;
    if (cs == 1) {
        p.nz = (int)nz;
        // Scores of up to 384 features: one chunk a group, 6.8e-7 off (two: 9.1e-7; 256 x 8192 scores of 256 features
        // 12.3 and 11.9 us, of 384 14.4 and 13.8 us). Longer ones: two, 9.1e-7 whatever their length (7168 features 102 us, with one 7.2e-7
        // and 113 us); so do the preconditioner's products (alpha = -1).
        p.gm = p.alpha == 1.f && nkc <= 12 ? 0 : 1;
        // A pair's chunk takes about three quarters of a single CTA's (see above), so its whole rounds of
        // tiles decide: few or odd 128-row tiles can leave half of the pairs' rows empty.
        int64_t pairs = p.lower ? pair_lower_tiles(tiles_n) : (tiles_m + 1) / 2 * tiles_n;
        CUtensorMap tmB2 = tmB;
        if (second) {  // always in pairs
            p.tiles_1 = pairs;
            p.tiles_n2 = (int)((second->n_b + BN - 1) / BN);
            pairs += (tiles_m + 1) / 2 * p.tiles_n2;
            p.n_q2 = second->n_b;
            p.S2 = second->C;
            p.ld_S2 = second->ldc;
            p.s_z2 = second->c_z;
            if (nz > 1 ? !make_map_f32_3d(&tmB2, second->B, second->n_b, p.K, second->ldb, nz, second->b_z_bytes, BN / 2)
                       : !make_map_f32(&tmB2, second->B, second->n_b, p.K, second->ldb, BN / 2))
                return cudaErrorInvalidValue;
        } else {
            p.tiles_1 = pairs;
        }
        const int64_t per = (int64_t)p.splits * nz, half = sms > 1 ? sms / 2 : 1;
        if (second || 3 * ((pairs * per + half - 1) / half) <= 4 * ((tiles * per + sms - 1) / sms)) {
            p.tiles_z = pairs;
            // B's box: the half of a tile's rows that one CTA of the pair loads
            if (nz > 1 ? !make_map_f32_3d(&tmB, p.B, p.n_q, p.K, p.ldb, nz, b_z_bytes, BN / 2)
                       : !make_map_f32(&tmB, p.B, p.n_q, p.K, p.ldb, BN / 2))
                return cudaErrorInvalidValue;
            if (p.red) {
                // output boxes: 32 columns x the rows of half a tile
                CUtensorMap tmS, tmS2;
                if (!make_map_out(&tmS, p.S, p.n_q, p.n_t, p.ld_S, nz, p.s_z, BN / 2)) return cudaErrorInvalidValue;
                tmS2 = tmS;
                if (second && !make_map_out(&tmS2, p.S2, p.n_q2, p.n_t, p.ld_S2, nz, p.s_z2, BN / 2))
                    return cudaErrorInvalidValue;
                return launch_pairs<BN, false, true>(tmA, tmB, tmB2, tmS, tmS2, p, sms, s);
            }
            return launch_pairs<BN, false, false>(tmA, tmB, tmB2, tmA, tmA, p, sms, s);
        }
        using T = TCfg<BN, false>;
        p.tiles_z = tiles;
        const int64_t total = tiles * per;
        cudaError_t e = smem_attr_once<gemm3t_kernel<BN, false, false, false>>((int)T::kSmem);
        if (e != cudaSuccess) return e;
        note_launches(1);
        gemm3t_kernel<BN, false, false, false><<<(unsigned)(total < sms ? total : sms), kThreadsT, T::kSmem, s>>>(tmA, tmB, tmB, tmA, tmA, p);
        return cudaGetLastError();
    }
    if (second) return cudaErrorInvalidValue;
    // few tiles: a cluster of cs CTAs splits K
    cudaError_t e = smem_attr_once<score3x_kernel<BN>>((int)C::kSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(tiles * cs), (unsigned)p.splits, (unsigned)nz);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launches(1);
    e = cudaLaunchKernelEx(&cfg, score3x_kernel<BN>, tmA, tmB, p);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

bool score_tc_supported(tda_dtype qdt, const void* Qhat, int64_t n_q, int64_t ld_q, const float* Phi, int64_t n_t,
                        int64_t ld_phi, int64_t D) {
    static int sm103 = -1;
    if (sm103 < 0) {
        int dev = 0, major = 0, minor = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
        sm103 = (major == 10 && minor == 3) ? 1 : 0;
    }
    if (!sm103 || qdt != TDA_F32 || !encode_fn()) return false;
    // TMA: 32-bit coordinates, row strides of whole 16-byte groups below 2^40 bytes
    if (n_q < 1 || n_t < 1 || D < 64 || D >= (1LL << 31) || n_q > (1LL << 24) || n_t > (1LL << 31) / kBM * kBM)
        return false;
    if (ld_q * 4 >= (1LL << 40) || ld_phi * 4 >= (1LL << 40)) return false;
    if ((ld_q & 3) || (ld_phi & 3)) return false;
    if (((uintptr_t)Qhat & 15) || ((uintptr_t)Phi & 15)) return false;
    return true;
}

cudaError_t launch_score_tc(const float* Qhat, int64_t n_q, int64_t ld_q, const float* Phi, int64_t n_t, int64_t ld_phi,
                            int64_t D, float* S, int64_t ld_S, float beta, unsigned int* err, cudaStream_t s) {
    GParams p{};
    p.A = Phi;
    p.B = Qhat;
    p.S = S;
    p.n_t = n_t;
    p.n_q = n_q;
    p.K = D;
    p.lda = ld_phi;
    p.ldb = ld_q;
    p.ld_S = ld_S;
    p.beta = beta;
    p.alpha = 1.f;
    p.kslice = 0;
    p.slab = 0;
    p.splits = 1;
    p.err = err;
    if (n_q <= 64) return launch_bn<64>(p, s);
    return launch_bn<128>(p, s);
}

int score_tc_tiles(int64_t n_q, int64_t n_t) {
    const int64_t bn = n_q <= 64 ? 64 : 128;
    const int64_t t = ((n_t + kBM - 1) / kBM) * ((n_q + bn - 1) / bn);
    return t > (1 << 30) ? (1 << 30) : (int)t;
}

// Partial scores of `splits` feature slices: part[z][q][i] = sum over slice z of
// Phi[i][f] Qhat[q][f] (slices of a multiple of 32 features; part holds
// splits * n_q * n_t floats). The caller sums the slabs.
cudaError_t launch_score_tc_slices(const float* Qhat, int64_t n_q, int64_t ld_q, const float* Phi, int64_t n_t,
                                   int64_t ld_phi, int64_t D, int splits, float* part, unsigned int* err,
                                   cudaStream_t s) {
    GParams p{};
    p.A = Phi;
    p.B = Qhat;
    p.n_t = n_t;
    p.n_q = n_q;
    p.K = D;
    p.lda = ld_phi;
    p.ldb = ld_q;
    int64_t kslice = (D + splits - 1) / splits;
    kslice = (kslice + kKC - 1) / kKC * kKC;
    p.kslice = kslice;
    p.splits = (int)((D + kslice - 1) / kslice);
    p.slab = n_q * n_t;
    p.S = part;
    p.ld_S = n_t;
    p.beta = 0.f;
    p.alpha = 1.f;
    p.err = err;
    if (p.splits > 65535) return cudaErrorInvalidValue;
    if (n_q <= 64) return launch_bn<64>(p, s);
    return launch_bn<128>(p, s);
}

// C[n][m] = beta * C[n][m] + alpha * sum_k A[m][k] B[n][k] (C row stride ldc): the
// score GEMM with a sign, used by the blocked Cholesky and triangular solves. With
// lower = true, A and B must be the same n x n operand rows (a symmetric rank-K
// update) and only the 128 x 128 tiles on or below the diagonal (m0 <= n0) are
// formed; entries above the diagonal inside a diagonal tile are written too. `second` (batch
// entries as in the first): C2 = beta * C2 + alpha * A B2^T with the same A, in the same launch.
cudaError_t launch_gemm_nt_tc_batched(const float* A, int64_t n_a, int64_t lda, size_t a_z_bytes, const float* B,
                                      int64_t n_b, int64_t ldb, size_t b_z_bytes, int64_t K, float* C, int64_t ldc,
                                      int64_t c_z, int64_t nz, float alpha, float beta, bool lower,
                                      unsigned int* err, cudaStream_t s, const GemmSecond* second) {
    if (nz < 1 || nz > 65535) return cudaErrorInvalidValue;
    if (nz > 1 && ((a_z_bytes & 15) || (b_z_bytes & 15) || !a_z_bytes || !b_z_bytes)) return cudaErrorInvalidValue;
    GParams p{};
    p.A = A;
    p.B = B;
    p.S = C;
    p.n_t = n_a;
    p.n_q = n_b;
    p.K = K;
    p.lda = lda;
    p.ldb = ldb;
    p.ld_S = ldc;
    p.beta = beta;
    p.alpha = alpha;
    p.lower = lower ? 1 : 0;
    p.kslice = 0;
    p.slab = 0;
    p.splits = 1;
    p.s_z = c_z;
    p.err = err;
    if (lower && n_a != n_b) return cudaErrorInvalidValue;
    auto aligned = [](const float* S, int64_t ld, int64_t z) { return !(((uintptr_t)S | (size_t)(ld * 4) | (size_t)(z * 4)) & 15); };
    p.red = beta == 1.f && aligned(C, ldc, c_z) && (!second || aligned(second->C, second->ldc, second->c_z));
    if (n_b <= 64 && !lower) return launch_bn<64>(p, s, nz, a_z_bytes, b_z_bytes, second);
    return launch_bn<128>(p, s, nz, a_z_bytes, b_z_bytes, second);
}

bool gemm_tc_available() {
    static int ok = -1;
    if (ok < 0) {
        int dev = 0, major = 0, minor = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
        ok = (major == 10 && minor == 3 && encode_fn()) ? 1 : 0;
    }
    return ok == 1;
}

bool fit_tc_supported(int n_layers, int64_t D, const float* phi, int64_t n, int64_t ld) {
    int dev = 0, major = 0, minor = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
    if (!(major == 10 && minor == 3) || !encode_fn()) return false;
    // TMA: 32-bit coordinates, 16-byte aligned base and row stride below 2^40 bytes, feature
    // coordinates a multiple of 4 (every tile starts at l*D + 128*j)
    if (D < 128 || (D & 3) || (ld & 3) || ((uintptr_t)phi & 15)) return false;
    if ((int64_t)n_layers * D >= (1LL << 31) || n >= (1LL << 31) - kKC || ld * 4 >= (1LL << 40)) return false;
    return true;
}

cudaError_t launch_fit_tc(int n_layers, int64_t D, void* state, size_t state_bytes, const float* phi, int64_t n,
                          int64_t ld, unsigned int* err, cudaStream_t s) {
    // features of all layers, examples as rows; zero fill past the last layer's features and the last example
    CUtensorMap tm;
    if (!make_map_f32(&tm, phi, n, (int64_t)n_layers * D, ld, kKC)) return cudaErrorInvalidValue;
    GParams p{};
    p.S = (float*)((char*)state + 64);
    p.s_z = (int64_t)(state_bytes / 4);
    p.n_t = p.n_q = p.ld_S = D;
    p.K = n;
    p.alpha = p.beta = 1.f;
    p.lower = 1;
    p.splits = 1;
    p.nz = n_layers;
    p.gm = 1;
    p.tiles_z = p.tiles_1 = pair_lower_tiles((D + kBM - 1) / kBM);
    p.err = err;
    static std::atomic<int> sms_cache{0};
    int sms = sms_cache.load(std::memory_order_relaxed);
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
        sms_cache.store(sms, std::memory_order_relaxed);
    }
    return launch_pairs<128, true, false>(tm, tm, tm, tm, tm, p, sms, s);
}

}  // namespace tda
