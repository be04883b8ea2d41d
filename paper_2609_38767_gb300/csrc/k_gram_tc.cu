// k_gram_tc.cu -- route (c), the factored Gram identity (Eq. 4), on the
// tcgen05 tensor cores of sm_103a for bf16 factors, for any token count:
//
//   <DW_q, DW_i>_F = sum_{t,s} (A_q A_i^T)[t][s] * (B_q B_i^T)[t][s],
//
// and the norms ||DW_i||^2 by the same identity with both sides example i.
//
// Both token Grams are dense contractions over the feature dimension, K-major
// in memory (a token's activations are contiguous), so they map directly onto
// tcgen05.mma: a 128-row tile of query tokens (M) against a 256-row tile of
// train tokens (N), first X = A_q A_i^T (K = d_in), then Y = B_q B_i^T
// (K = d_out).
//
// Token tiles: for T <= 128 a query tile packs floor(128 / T) whole query
// examples and a train tile floor(256 / T) train examples (their tokens are
// consecutive rows), so one tile pair yields a whole block of S; rows past the
// last whole example belong to the next tile's examples and are left out of
// the sums. For T > 128 a (query, train) pair is a loop over its
// ceil(T/128) x ceil(T/256) tile pairs (tokens past T read as zero rows).
//
// Accuracy: the tensor pipe adds into its fp32 accumulators with truncation,
// a loss of about a quarter ulp per addition that always points to zero (d =
// 2048, 128 additions: 3.6e-6 low). So K goes in blocks of one to four 64-feature
// chunks, each into one of two 256-column TMEM buffers, and the epilogue adds
// the blocks in registers with round-to-nearest: X's blocks are summed (128
// registers a thread), and since the identity is bilinear every Y block is
// multiplied into the sums as it arrives, sum_s X[t][s] Y_b[t][s], and need not
// be kept. The buffers alternate, so the epilogue of one block overlaps the
// MMAs of the next.
//
// What bounds it: in one CTA, each M = 128, N = 256, K = 16 MMA reads 12 KB of
// operands from shared memory and the TMA writes as much, ~190 B/clock per SM against
// ~128 B/clock of shared-memory bandwidth, so the tile tops out near two
// thirds of the MMA rate. Pairs of CTAs (PAIR, cta_group::2) read 8 KB. The epilogue
// (256 threads, 128 columns each) reads 128 KB of TMEM per block, more than
// half the time of a two-chunk block's MMAs; sixteen warps for it were 12 % slower.
//
// Measured (similarity alone): 2048 -> 2048, T = 50, 16 x 512 pairs 34.9 ms on the
// CUDA cores (T not a power of two), now 0.22 ms = 0.76 PFLOP/s useful (100 of 128
// and 250 of 256 tile rows), then 0.142 ms in pairs and blocks of 256; 8192 -> 8192 at T = 8 / 32 / 128 / 512: 1.14 / 1.25 /
// 1.27 / 0.99 PFLOP/s with one accumulation per tile and no overlap between tiles,
// now 1.80 / 1.73 / 1.77 / 1.49.
//
// Norms (SELF): one 128-row tile of packed examples against itself needs one
// 16 KB copy per chunk (A and B operand are the same tile) and is bound by
// HBM (512 examples of 50 tokens, 2048 -> 2048: 3.9 ms on the CUDA cores, now
// 58 us); T > 128 loops over the tile pairs i <= j, off-diagonal ones doubled.
//
// Warp roles (320 threads, one persistent CTA per SM): warp 0 TMA producer,
// warp 1 TMEM allocator and MMA issuer (of a pair: in CTA 0), warps 2-9 epilogue (two warps
// per TMEM lane quadrant, each half of the columns). Waits are bounded (about
// 1 s) and set kErrTimeout on expiry, as in the projection kernel.
#include <cuda.h>
#include <cuda_bf16.h>

#include <mutex>

#include "tda_internal.cuh"

namespace tda {
namespace {

constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kTM = 128;                                 // query token rows per tile (MMA M)
constexpr int kChunkK = 64;                              // K elements per stage
constexpr uint32_t kABytes = kTM * kChunkK * 2;          // 16 KiB
constexpr uint32_t kTmemCols = 512;                      // two accumulator buffers of at most 256 columns
constexpr int kMaxStages = 8;
constexpr size_t kSmemMax = 232448;                      // 227 KiB of dynamic shared memory per CTA
constexpr size_t kTailBytes = 16 * 8 + 8 * (3 * kMaxStages + 5) + 16;  // warp sums, barriers, TMEM slot, abort flag

template <bool SELF, bool PAIR = false>
struct Cfg {
    static constexpr int kTN = SELF ? 128 : 256;         // train token rows per tile (MMA N)
    static constexpr int kCols = kTN / 2;                // columns per epilogue thread
    static constexpr int kBRows = PAIR ? kTN / 2 : kTN;  // of which in this CTA
    static constexpr uint32_t kStageBytes = kABytes + kBRows * kChunkK * 2;
};

struct GParams {
    int64_t n_q, n_t, T, ld_S;
    int nk_in, nk_out;      // K chunks per side
    int kbx, kby;           // chunks per accumulation block of X and of Y
    int stages;
    int pq, pt;             // examples per query tile and per train tile (T <= 128), else 0
    int ldr;                // floats per row of the per-example partial sums (packed)
    int64_t n_units;        // tile pairs (packed) or example pairs (T > 128); SELF: tiles or examples
    int64_t n_qtiles;       // packed query tiles, or pairs of them
    int tiles_q, tiles_t;   // token tiles per query / train example (T > 128)
    float alpha, beta;
    float* S;
    unsigned int* err;
};

#include "tc_ptx.cuh"

// mma_bf16 of one CTA or a pair
template <bool PAIR>
__device__ __forceinline__ void mma_bf16_g(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate) {
    if constexpr (PAIR)
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
                d_tmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    else
        mma_bf16(d_tmem, adesc, bdesc, idesc, accumulate);
}

__device__ __forceinline__ void emit(const GParams& p, int64_t q, int64_t i, float v) {
    float* dst = p.S + q * p.ld_S + i;
    *dst = p.beta == 0.f ? p.alpha * v : p.beta * (*dst) + p.alpha * v;
}

// OR of v over the epilogue threads (named barrier 1).
__device__ __forceinline__ bool epi_or(bool v) {
    uint32_t r;
    __syncwarp();
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(32 * kEpiWarps)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One Y block of a packed tile for T = TS < 16: this thread's columns are kCols / TS whole train
// examples, so every boundary is known when compiled (a run-time test per column cost 2.6 times
// the MMAs' time at T = 8).
template <int TS, int COLS>
__device__ __forceinline__ void y_block_short(const float (&x)[COLS], uint32_t tb, float* myred, bool first) {
    constexpr int kUse = COLS / TS * TS;
    float s = 0.f;
#pragma unroll
    for (int c0 = 0; c0 < kUse; c0 += 16) {
        float v[16];
        tmem_ld16(tb + c0, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (c0 + i >= kUse) break;
            s = (c0 + i) % TS == 0 ? x[c0 + i] * v[i] : fmaf(x[c0 + i], v[i], s);
            if ((c0 + i + 1) % TS == 0) {
                float* dst = myred + (c0 + i) / TS;
                *dst = first ? s : *dst + s;
            }
        }
    }
}

template <bool SELF, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
gram_tc_kernel(const __grid_constant__ CUtensorMap tmAq, const __grid_constant__ CUtensorMap tmAt,
               const __grid_constant__ CUtensorMap tmBq, const __grid_constant__ CUtensorMap tmBt,
               const GParams p) {
    using C = Cfg<SELF, PAIR>;
    constexpr int kTN = C::kTN, kCols = C::kCols;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float* wsum = (float*)(smem + (size_t)p.stages * C::kStageBytes);  // [8 warps] sums of a (query, train) pair
    uint64_t* bars = (uint64_t*)(wsum + 32);
    uint64_t* full = bars;                  // [stages] landed (count 1 + tx)
    uint64_t* empty = bars + kMaxStages;    // [stages] MMAs done with the stage
    uint64_t* tfull = bars + 2 * kMaxStages;  // [2] block accumulated
    uint64_t* tempty = tfull + 2;           // [2] block drained (one arrive per epilogue warp)
    uint64_t* mma_done = tempty + 2;
    uint64_t* pfull = mma_done + 1;         // [stages] PAIR: landed in CTA 1
    uint32_t* tmem_slot = (uint32_t*)(pfull + kMaxStages);
    volatile int* abort = (volatile int*)(tmem_slot + 1);
    float* red = (float*)(tmem_slot + 4);   // packed: [2 column halves][128 rows][ldr examples] partial sums

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
            mbar_init(smem_u32(&pfull[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&tfull[b]), 1);
            mbar_init(smem_u32(&tempty[b]), PAIR ? 2 * kEpiWarps : kEpiWarps);
        }
        mbar_init(smem_u32(mma_done), 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            tmem_alloc2(smem_u32(tmem_slot), kTmemCols);
        } else {
            tmem_alloc(smem_u32(tmem_slot), kTmemCols);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const int64_t u0 = PAIR ? blockIdx.x >> 1 : blockIdx.x, ustep = PAIR ? gridDim.x >> 1 : gridDim.x;
    // packed: this CTA's query tile of unit u
    auto qtile = [&](int64_t u) { return SELF ? u : (PAIR ? 2 * (u % p.n_qtiles) + rank : u % p.n_qtiles); };
    const bool packed = p.pq > 0;
    const int nk_tot = p.nk_in + p.nk_out;
    const int nbx = (p.nk_in + p.kbx - 1) / p.kbx, nb = nbx + (p.nk_out + p.kby - 1) / p.kby;
    // tile pairs per unit: SELF takes only i <= j
    const int tpp = packed ? 1 : (SELF ? p.tiles_q * (p.tiles_q + 1) / 2 : p.tiles_q * p.tiles_t);

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer
        uint32_t s = 0, ph = 0, last_par[kMaxStages];
        bool issued[kMaxStages], ok = true;
        for (int i = 0; i < kMaxStages; ++i) issued[i] = false;
        for (int64_t u = u0; ok && u < p.n_units; u += ustep) {
            int ti = 0, tj = 0;
            for (int tp = 0; ok && tp < tpp; ++tp) {
                int rq, eq, rt, et;
                if (packed) {  // rows of the [n*T][d] views
                    rq = (int)(qtile(u) * p.pq * p.T);
                    rt = SELF ? rq : (int)((u / p.n_qtiles) * p.pt * p.T) + (int)rank * C::kBRows;
                    eq = et = 0;
                } else {       // token tiles of one query and one train example
                    eq = (int)(SELF ? u : u % p.n_q);
                    et = SELF ? eq : (int)(u / p.n_q);
                    rq = ti * kTM;
                    rt = tj * kTN;
                }
                const bool one = SELF && ti == tj;  // both operands are the same tile
                for (int kc = 0; kc < nk_tot; ++kc) {
                    if (!wait_bounded(smem_u32(&empty[s]), ph ^ 1u, abort, p.err)) {
                        ok = false;
                        break;
                    }
                    const bool side_b = kc >= p.nk_in;
                    const int d0 = (side_b ? kc - p.nk_in : kc) * kChunkK;
                    uint8_t* st = smem + (size_t)s * C::kStageBytes;
                    mbar_arrive_tx(smem_u32(&full[s]), one ? kABytes : C::kStageBytes);
                    tma_load_3d(smem_u32(st), side_b ? &tmBq : &tmAq, d0, rq, eq, smem_u32(&full[s]));
                    if (!one)
                        tma_load_3d(smem_u32(st + kABytes), side_b ? &tmBt : &tmAt, d0, rt, et, smem_u32(&full[s]));
                    issued[s] = true;
                    last_par[s] = ph;
                    if (++s == (uint32_t)p.stages) s = 0, ph ^= 1u;
                }
                if (++tj == p.tiles_t) tj = SELF ? ++ti : (++ti, 0);
            }
        }
        for (int i = 0; i < p.stages; ++i)
            if (issued[i]) {
                const uint64_t t0 = global_ns();
                while (!mbar_try_wait(smem_u32(&full[i]), last_par[i]))
                    if (global_ns() - t0 > kTimeoutNs) {
                        atomicOr(p.err, kErrTimeout);
                        break;
                    }
                // every arrival of the pair's MMAs on this CTA's barriers lands before it exits
                if (PAIR && ok && !wait_bounded(smem_u32(&empty[i]), last_par[i], abort, p.err)) ok = false;
            }
    } else if (warp == 1 && rank == 1) {
        // ---------------- CTA 1 of a pair: tells CTA 0, which issues the MMAs, that a stage has landed
        uint32_t s = 0, ph = 0;
        bool ok = true;
        for (int64_t u = u0; ok && u < p.n_units; u += ustep)
            for (int kc = 0; kc < nk_tot; ++kc) {
                if (!warp_wait(smem_u32(&full[s]), ph, abort, p.err)) {
                    ok = false;
                    break;
                }
                if (lane == 0) arrive_leader<PAIR>(smem_u32(&pfull[s]));
                if (++s == (uint32_t)p.stages) s = 0, ph ^= 1u;
            }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the warp waits, one lane issues
        uint32_t s = 0, ph = 0, cnt = 0;
        bool ok = true;
        constexpr uint32_t idesc = idesc_bf16(PAIR ? 2 * kTM : kTM, kTN);
        for (int64_t u = u0; ok && u < p.n_units; u += ustep) {
            int ti = 0, tj = 0;
            for (int tp = 0; ok && tp < tpp; ++tp) {
                const uint32_t boff = SELF && ti == tj ? 0u : kABytes;
                for (int blk = 0; ok && blk < nb; ++blk, ++cnt) {
                    const uint32_t b = cnt & 1u;
                    if (!warp_wait(smem_u32(&tempty[b]), ((cnt >> 1) & 1u) ^ 1u, abort, p.err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const bool side_b = blk >= nbx;
                    const int kb = side_b ? p.kby : p.kbx;
                    const int left = side_b ? p.nk_out - (blk - nbx) * kb : p.nk_in - blk * kb;
                    const int n = left < kb ? left : kb;
                    for (int c = 0; c < n; ++c) {
                        if (!warp_wait(smem_u32(&full[s]), ph, abort, p.err) ||
                            (PAIR && !warp_wait(smem_u32(&pfull[s]), ph, abort, p.err))) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t st = smem_u32(smem + (size_t)s * C::kStageBytes);
                        const uint64_t ad = sw128_desc(st), bd = sw128_desc(st + boff);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < kChunkK / 16; ++k)
                                mma_bf16_g<PAIR>(tmem + b * 256u, ad + 2 * k, bd + 2 * k, idesc, (c > 0 || k > 0) ? 1u : 0u);
                            commit_all<PAIR>(smem_u32(&empty[s]));
                        }
                        __syncwarp();
                        if (++s == (uint32_t)p.stages) s = 0, ph ^= 1u;
                    }
                    if (!ok) break;
                    if (elect_one()) commit_all<PAIR>(smem_u32(&tfull[b]));
                    __syncwarp();
                }
                if (++tj == p.tiles_t) tj = SELF ? ++ti : (++ti, 0);
            }
        }
        if (elect_one()) {
            if constexpr (PAIR)
                commit_pair_local(smem_u32(mma_done));
            else
                mma_commit(smem_u32(mma_done));
            const uint64_t t0 = global_ns();
            while (!mbar_try_wait(smem_u32(mma_done), 0))
                if (global_ns() - t0 > kTimeoutNs) {
                    atomicOr(p.err, kErrTimeout);
                    break;
                }
        }
        __syncwarp();
    } else if (warp >= 2) {
        // ---------------- epilogue: warp ew covers TMEM lane quadrant warp % 4, column half h
        const int ew = warp - 2, q4 = warp & 3, h = ew >> 2, row = q4 * 32 + lane;
        const int et = threadIdx.x - 64, T = (int)p.T;
        // this thread's columns [c_lo, c_lo + kCols): half the tile, or for packed T < 16 whole examples
        const bool brief = packed && !SELF && T < 16;
        const int c_lo = h * (brief ? kCols / T * T : kCols);
        const int g_lo = packed && !SELF ? c_lo / T : 0;     // first train example among them
        const uint32_t tbase = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c_lo;
        float* myred = red + (size_t)(h * kTM + row) * p.ldr;
        // SELF packed: the columns of this row's own example
        const int own = packed && SELF ? row / T * T : 0;
        uint32_t cnt = 0;
        bool ok = true, stop = false;
        for (int64_t u = u0; !stop && u < p.n_units; u += ustep) {
            float tot = 0.f;  // T > 128 and SELF: this thread's share of the sum
            int ti = 0, tj = 0;
            for (int tp = 0; tp < tpp; ++tp) {
                float x[kCols], tile = 0.f;
#pragma unroll
                for (int c = 0; c < kCols; ++c) x[c] = 0.f;
                for (int blk = 0; ok && blk < nb; ++blk, ++cnt) {
                    const uint32_t b = cnt & 1u;
                    ok = warp_wait(smem_u32(&tfull[b]), (cnt >> 1) & 1u, abort, p.err);
                    if (!ok) break;  // the other roles see the abort flag; the barrier below ends the unit
                    tc_fence_after();
                    const uint32_t tb = tbase + b * 256u;
                    if (blk < nbx) {
#pragma unroll
                        for (int c0 = 0; c0 < kCols; c0 += 16) {
                            float v[16];
                            tmem_ld16(tb + c0, v);
#pragma unroll
                            for (int i = 0; i < 16; ++i) x[c0 + i] += v[i];
                        }
                    } else if (SELF || !packed) {
                        // columns [c_first, c_last) of this thread's, relative to its first: the row's own
                        // example (SELF, packed) or the tokens below T; a product left out, not
                        // multiplied by zero, so that another example's infinity stays its own
                        const int c_first = SELF && packed ? own - c_lo : 0;
                        const int c_last = packed ? c_first + T : T - tj * kTN - c_lo;
                        float s0 = 0.f, s1 = 0.f;
#pragma unroll
                        for (int c0 = 0; c0 < kCols; c0 += 16) {
                            float v[16];
                            tmem_ld16(tb + c0, v);
                            if (c_first <= c0 && c_last >= c0 + 16) {
#pragma unroll
                                for (int i = 0; i < 16; i += 2) {
                                    s0 = fmaf(x[c0 + i], v[i], s0);
                                    s1 = fmaf(x[c0 + i + 1], v[i + 1], s1);
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    if (c0 + i >= c_first && c0 + i < c_last) s0 = fmaf(x[c0 + i], v[i], s0);
                            }
                        }
                        if (packed || ti * kTM + row < T) tile += s0 + s1;
                    } else if (brief) {
                        const bool first = blk == nbx;
                        switch (T) {
#define TDA_SHORT(t) case t: y_block_short<t, kCols>(x, tb, myred, first); break;
                            TDA_SHORT(1) TDA_SHORT(2) TDA_SHORT(3) TDA_SHORT(4) TDA_SHORT(5) TDA_SHORT(6) TDA_SHORT(7)
                            TDA_SHORT(8) TDA_SHORT(9) TDA_SHORT(10) TDA_SHORT(11) TDA_SHORT(12) TDA_SHORT(13)
                            TDA_SHORT(14) TDA_SHORT(15)
#undef TDA_SHORT
                        }
                    } else {
                        // packed, T >= 16: one sum per train example; left = columns to the end of the
                        // current one, at most one end inside 16 columns
                        const bool first = blk == nbx;
                        float s0 = 0.f, s1 = 0.f;
                        int left = (g_lo + 1) * T - c_lo;
                        float* dst = myred;
#pragma unroll
                        for (int c0 = 0; c0 < kCols; c0 += 16) {
                            float v[16];
                            tmem_ld16(tb + c0, v);
                            if (left > 16) {
#pragma unroll
                                for (int i = 0; i < 16; i += 2) {
                                    s0 = fmaf(x[c0 + i], v[i], s0);
                                    s1 = fmaf(x[c0 + i + 1], v[i + 1], s1);
                                }
                                left -= 16;
                            } else {
                                float n0 = 0.f;
#pragma unroll
                                for (int i = 0; i < 16; ++i) {
                                    if (i < left)
                                        s0 = fmaf(x[c0 + i], v[i], s0);
                                    else
                                        n0 = fmaf(x[c0 + i], v[i], n0);
                                }
                                *dst = first ? s0 + s1 : *dst + (s0 + s1);
                                ++dst;
                                s0 = n0;
                                s1 = 0.f;
                                left += T - 16;
                            }
                        }
                        if (left < T) *dst = first ? s0 + s1 : *dst + (s0 + s1);  // ends in the next half
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader<PAIR>(smem_u32(&tempty[b]));
                }
                if (!ok) break;
                tot = SELF && ti != tj ? fmaf(2.f, tile, tot) : tot + tile;  // (i, j) stands for (j, i) too
                if (++tj == p.tiles_t) tj = SELF ? ++ti : (++ti, 0);
            }
            if (!packed) {
                const float v = warp_sum(tot);
                if (lane == 0) wsum[ew] = v;
            } else if (SELF) {
                myred[0] = tot;
            }
            stop = epi_or(!ok);
            if (!stop) {
                if (!packed) {
                    if (et == 0) {
                        float v = 0.f;
                        for (int w = 0; w < kEpiWarps; ++w) v += wsum[w];
                        if (SELF)
                            emit(p, 0, u, v);
                        else
                            emit(p, u % p.n_q, u / p.n_q, v);
                    }
                } else {
                    // output o = (query qi of the tile, train example g of the tile): T rows of partial
                    // sums from the one or two column halves that hold the example's columns
                    const int pt = SELF ? 1 : p.pt, nout = p.pq * pt;
                    const int lanes = T >= 16 ? 32 : 1;  // long columns of partials: one warp each
                    for (int o = et / lanes; o < nout; o += 32 * kEpiWarps / lanes) {
                        const int qi = o / pt, g = o - qi * pt;
                        // the column halves that hold example g, and the first example of each
                        const int per = kCols / T;  // T < 16: examples per half
                        const int h0 = SELF ? 0 : (brief ? g / per : g * T / kCols);
                        const int h1 = SELF ? 1 : (brief ? h0 : (g * T + T - 1) / kCols);
                        float v = 0.f;
                        for (int hh = h0; hh <= h1; ++hh) {
                            const int g0 = SELF ? 0 : (brief ? hh * per : hh * kCols / T);
                            const float* r = red + (size_t)(hh * kTM + qi * T) * p.ldr + (SELF ? 0 : g - g0);
                            for (int t = lanes > 1 ? lane : 0; t < T; t += lanes) v += r[(size_t)t * p.ldr];
                        }
                        if (lanes > 1) v = warp_sum(v);
                        const int64_t qq = qtile(u) * p.pq + qi;
                        const int64_t ii = SELF ? 0 : (u / p.n_qtiles) * p.pt + g;
                        if (lanes == 1 || lane == 0) {
                            if (SELF) {
                                if (qq < p.n_q) emit(p, 0, qq, v);
                            } else if (qq < p.n_q && ii < p.n_t) {
                                emit(p, qq, ii, v);
                            }
                        }
                    }
                }
            }
            epi_or(false);  // the partial sums are read: the next unit may write them
        }
    }

    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        if constexpr (PAIR)
            tmem_dealloc2(tmem, kTmemCols);
        else
            tmem_dealloc(tmem, kTmemCols);
    }
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

// 3-D map over X[n][rows][d] (bf16), box 64 (d) x box_rows x 1, 128B swizzle, zero fill.
bool make_map(CUtensorMap* tm, const void* X, int64_t n, int64_t rows, int64_t d, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)n};
    cuuint64_t strides[2] = {(cuuint64_t)(d * 2), (cuuint64_t)(rows * d * 2)};
    cuuint32_t box[3] = {kChunkK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(X), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Maps of one side's factors: packed rows [1][n*T][d], else [n][T][d].
bool make_side(CUtensorMap* mA, CUtensorMap* mB, const tda_layer_desc& L, const void* A, const void* B, int64_t n,
               bool packed, int box_rows) {
    return packed ? make_map(mA, A, 1, n * L.T, L.d_in, box_rows) && make_map(mB, B, 1, n * L.T, L.d_out, box_rows)
                  : make_map(mA, A, n, L.T, L.d_in, box_rows) && make_map(mB, B, n, L.T, L.d_out, box_rows);
}

// Most examples of one launch's side: 32-bit TMA row coordinates, strides below 2^40 bytes.
int64_t max_examples(const tda_layer_desc& L, bool packed) {
    const int64_t d_max = L.d_in > L.d_out ? L.d_in : L.d_out;
    if (!packed) return ((int64_t)1 << 30);
    const int64_t by_rows = ((int64_t)1 << 30) / L.T, by_stride = (((int64_t)1 << 40) - 1) / (L.T * d_max * 2);
    return by_rows < by_stride ? by_rows : by_stride;
}

int sm_count() {
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

template <bool SELF, bool PAIR>
cudaError_t launch_kernel(const tda_layer_desc& L, const void* Aq, const void* Bq, int64_t n_q, const void* At,
                          const void* Bt, int64_t n_t, GParams p, cudaStream_t s) {
    using C = Cfg<SELF, PAIR>;
    const bool packed = L.T <= kTM;
    CUtensorMap mAq, mAt, mBq, mBt;
    if (!make_side(&mAq, &mBq, L, Aq, Bq, n_q, packed, kTM) || !make_side(&mAt, &mBt, L, At, Bt, n_t, packed, C::kBRows))
        return cudaErrorInvalidValue;
    if (PAIR) p.n_qtiles = (p.n_qtiles + 1) / 2;
    if (SELF)
        p.n_units = packed ? p.n_qtiles : n_q;
    else
        p.n_units = packed ? p.n_qtiles * ((n_t + p.pt - 1) / p.pt) : n_q * n_t;
    // partial sums of a packed tile: rows of an odd stride (no bank conflicts)
    const int64_t T = L.T;
    p.ldr = !packed || SELF ? 1 : (int)(T < 16 ? C::kCols / T : (C::kCols - 1) / T + 2) | 1;
    const size_t red = packed ? 2 * (size_t)kTM * p.ldr * sizeof(float) : 0;
    const int64_t stages = ((int64_t)kSmemMax - 1024 - (int64_t)kTailBytes - (int64_t)red) / C::kStageBytes;
    if (stages < 2) return cudaErrorInvalidValue;
    p.stages = stages < kMaxStages ? (int)stages : kMaxStages;
    const size_t smem = 1024 + (size_t)p.stages * C::kStageBytes + kTailBytes + red;
    cudaError_t e = smem_attr_once<gram_tc_kernel<SELF, PAIR>>((int)kSmemMax);
    if (e != cudaSuccess) return e;
    const int64_t room = PAIR ? (sm_count() > 1 ? sm_count() / 2 : 1) : sm_count();
    const int64_t grid = (p.n_units < room ? p.n_units : room) * (PAIR ? 2 : 1);
    note_launches(1);
    if constexpr (PAIR) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)grid);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, gram_tc_kernel<SELF, PAIR>, mAq, mAt, mBq, mBt, p);
        if (e != cudaSuccess) return e;
    } else {
        gram_tc_kernel<SELF, PAIR><<<(unsigned)grid, kThreads, smem, s>>>(mAq, mAt, mBq, mBt, p);
    }
    return cudaGetLastError();
}

template <bool SELF>
cudaError_t launch(const tda_layer_desc& L, const void* Aq, const void* Bq, int64_t n_q, const void* At,
                   const void* Bt, int64_t n_t, GParams p, cudaStream_t s) {
    using C = Cfg<SELF>;
    const int64_t T = L.T, sms = sm_count();
    const bool packed = T <= kTM;
    p.n_q = n_q;
    p.n_t = n_t;
    p.T = T;
    p.nk_in = (int)((L.d_in + kChunkK - 1) / kChunkK);
    p.nk_out = (int)((L.d_out + kChunkK - 1) / kChunkK);
    // Block lengths that keep the accuracy of an fp32 FMA chain over d features (1.6e-7 at d = 256, 5.2e-7 at
    // 2048, 8.5e-7 at 4096): 64, 128 or 256 features (1.5e-7, 2.5e-7 at d = 1024, 4.5e-7; 2048 -> 2048, T = 50:
    // 183 -> 143 us from 128 to 256). T < 16 pays the most per Y block, but Y blocks of twice the length are off
    // by half as much again (T = 5, d = 2048: 6.6e-7; 64 x 8192 pairs, T = 8, d = 256: 56 us, and 66 us so;
    // 64 x 2048 pairs, d = 2048: 58 us either way).
    auto block = [](int nk) { return nk <= 8 ? 1 : (nk < 32 ? 2 : 4); };
    p.kbx = block(p.nk_in);
    p.kby = block(p.nk_out);
    p.pq = packed ? (int)(kTM / T) : 0;
    p.pt = !packed ? 0 : (int)(T < 16 ? C::kCols / T * 2 : C::kTN / T);
    p.tiles_q = packed ? 1 : (int)((T + kTM - 1) / kTM);
    p.tiles_t = packed ? 1 : (int)((T + C::kTN - 1) / C::kTN);
    p.n_qtiles = packed ? (n_q + p.pq - 1) / p.pq : 0;
    if constexpr (!SELF) {
        // Pairs of CTAs take two query tiles against one train tile: each has half of the train rows to
        // copy and to read (512 clocks of shared memory a chunk instead of 768). 8192 -> 8192, T = 32, 64 x
        // 512 examples: 682 us in single CTAs, 634 us in pairs. Not where an odd tile count makes more
        // rounds, nor for few features, where a pair's start costs more (256 -> 256: 19 and 21 us).
        const int64_t tt = packed ? (n_t + p.pt - 1) / p.pt : 0;
        const int64_t ones = (p.n_qtiles * tt + sms - 1) / sms, half = sms > 1 ? sms / 2 : 1;
        const int64_t pairs = ((p.n_qtiles + 1) / 2 * tt + half - 1) / half;
        if (packed && p.n_qtiles >= 2 && pairs <= ones && p.nk_in + p.nk_out >= 48) return launch_kernel<false, true>(L, Aq, Bq, n_q, At, Bt, n_t, p, s);
    }
    return launch_kernel<SELF, false>(L, Aq, Bq, n_q, At, Bt, n_t, p, s);
}

}  // namespace

bool gram_tc_supported(const tda_layer_desc& L, tda_dtype dt, const void* Aq, const void* Bq, const void* At,
                       const void* Bt) {
    static int sm103 = -1;
    if (sm103 < 0) {
        int dev = 0, major = 0, minor = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
        sm103 = (major == 10 && minor == 3) ? 1 : 0;
    }
    if (!sm103 || !encode_fn() || dt != TDA_BF16) return false;
    if (L.T < 1 || L.T > (1 << 20) || L.d_in % 8 || L.d_out % 8 || L.d_in > (1LL << 30) || L.d_out > (1LL << 30))
        return false;
    if (max_examples(L, L.T <= kTM) < kTM) return false;
    for (const void* x : {Aq, Bq, At, Bt})
        if ((uintptr_t)x & 15) return false;
    return true;
}

// Few pairs of short, narrow examples: a tile's epilogue sums all of its pq x pt outputs, of which such a job uses a
// few, while the CUDA-core kernel has a CTA for every pair. Times of both in us, d both widths together. T = 3, 64 ->
// 64, 1 x 8 pairs: 5 us on the CUDA cores and 15 us here; T = 1, one pair: 4.5 and 73 us; T = 5, 128 -> 128, 4 x 16: 8.8 and
// 10.9 us, 256 -> 256: 14.5 and 13.8 us; norms, T = 3, 64 -> 64: 4.7 and 5.7 us, 128 -> 128: 7.6 and 7.1 us. Jobs of more
// pairs than two an SM stay here, whose time does not grow with them.
bool gram_short(const tda_layer_desc& L, int64_t n_q, int64_t n_t, bool norms) {
    const int64_t most = 2 * (int64_t)sm_count();
    if (L.T >= 16 || n_q > most || n_t > most || (norms ? n_q : n_q * n_t) > most) return false;
    const double T = (double)L.T, d = (double)(L.d_in + L.d_out), chain = (0.018 + 0.0009 * T) * d;
    if (norms) return 2.2 + chain < 4.0 + 0.09 * T + 0.0105 * d;
    const int64_t outputs = (int64_t)(kTM / L.T) * (Cfg<false>::kCols / L.T * 2);
    return 2.6 + chain < 5.6 + 0.0022 * (double)outputs + 0.0085 * d;
}

// S[q][i] = beta * S[q][i] + alpha * <DW_q, DW_i>_F for bf16 factors. A side with more examples
// than one launch addresses goes in pieces, each its own block of S.
cudaError_t launch_gram_tc(const tda_layer_desc& L, const void* Aq, const void* Bq, int64_t n_q, const void* At,
                           const void* Bt, int64_t n_t, float* S, int64_t ld_S, float beta, float alpha,
                           unsigned int* err, cudaStream_t s) {
    const int64_t most = max_examples(L, L.T <= kTM);
    const size_t a_ex = (size_t)L.T * L.d_in * 2, b_ex = (size_t)L.T * L.d_out * 2;
    GParams p = {};
    p.alpha = alpha;
    p.beta = beta;
    p.ld_S = ld_S;
    p.err = err;
    for (int64_t q0 = 0; q0 < n_q; q0 += most)
        for (int64_t i0 = 0; i0 < n_t; i0 += most) {
            p.S = S + q0 * ld_S + i0;
            cudaError_t e = launch<false>(L, (const char*)Aq + q0 * a_ex, (const char*)Bq + q0 * b_ex,
                                          n_q - q0 < most ? n_q - q0 : most, (const char*)At + i0 * a_ex,
                                          (const char*)Bt + i0 * b_ex, n_t - i0 < most ? n_t - i0 : most, p, s);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

// out[i] = ||DW_i||_F^2 for bf16 factors.
cudaError_t launch_gram_self_tc(const tda_layer_desc& L, const void* A, const void* B, int64_t n, float* out,
                                unsigned int* err, cudaStream_t s) {
    const int64_t most = max_examples(L, L.T <= kTM);
    const size_t a_ex = (size_t)L.T * L.d_in * 2, b_ex = (size_t)L.T * L.d_out * 2;
    GParams p = {};
    p.alpha = 1.f;
    p.err = err;
    for (int64_t i0 = 0; i0 < n; i0 += most) {
        const char *a = (const char*)A + i0 * a_ex, *b = (const char*)B + i0 * b_ex;
        const int64_t c = n - i0 < most ? n - i0 : most;
        p.S = out + i0;
        cudaError_t e = launch<true>(L, a, b, c, a, b, c, p, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tda
