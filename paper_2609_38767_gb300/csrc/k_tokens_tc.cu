// k_tokens_tc.cu -- token-level scores on the tcgen05 tensor cores (3xTF32):
//   out[q][t] = beta * out[q][t] + scale * g~_t^T R_q a~_t
// for k_in in 17 .. 64 (a multiple of 4) and k_out in {16, 32, 64} (the token-level
// decomposition of the score: summed over t it gives <Phi_i, R_q>). k_in up to 16
// stays on the CUDA cores: half of every 32-wide MMA chunk would be padding.
//
// As a contraction: X[t][(q, r)] = sum_c a~_t[c] R_q[r][c] is a GEMM with
// M = 128 tokens, N rows (q, r) of the stacked query matrices, K = k_in; the
// epilogue weights X by g~_t[r] and sums over r, one output per (t, q).
//
// fp32 accuracy from TF32: x = hi + lo, both rounded to nearest (truncated halves
// lose 2^-22 of every product on the same side), products hi*hi + hi*lo + lo*hi.
// The two small products of all k come first: the tensor pipe truncates its
// running sum, and while that sum is small so is the loss (k = 32: 3.0e-7 off, 8.2e-7
// with truncated halves and interleaved products). KC = 2 (below) keeps the two chunks'
// hi*hi in accumulators of their own, added with round-to-nearest.
//
// Shared memory: K in chunks of 32 (one 128-byte operand row each), KC of them.
// KC = 1: two token-tile buffers (hi and lo, 16 KiB each) and a ring of two query
// stages of N = 256 rows (hi and lo, 32 KiB each). KC = 2 has twice the bytes per
// row: one token-tile buffer, stages of N = 128. R's halves are split once per
// call into the workspace. k_in below a whole chunk is zero-filled by TMA.
//
// Measured: 16 examples of 1024 tokens, 16 queries, k = 64: 180 us on the CUDA
// cores (a thread per token, R_j broadcast from shared memory), 18 us here.
//
// Warp roles (256 threads, so that no SM sub-partition holds more than two
// warps and every thread may use up to 255 registers): warps 0 and 3 split the
// token tile (hi in place, lo to its own tile); warp 1 allocates TMEM, its lane 0
// issues the MMAs into two fp32 accumulators; lane 0 of warp 2 issues the TMA
// copies; warps 4-7 are the epilogue (TMEM lane quadrant warp % 4). Waits are
// bounded (about 1 s) and set kErrTimeout on expiry.
#include <cuda.h>

#include <mutex>

#include "tda_internal.cuh"

namespace tda {
namespace {

#include "tc_ptx.cuh"

constexpr int kThreads = 256;
constexpr int kTM = 128;                          // tokens per tile
constexpr int kKA = 32;                           // K chunk: one 128-byte operand row
constexpr uint32_t kATile = kTM * kKA * 4;        // 16 KiB
constexpr uint32_t kTmemCols = 512;

template <int KC>
struct Cfg {
    static constexpr int kTN = 256 / KC;                  // (query, r) rows per stage
    static constexpr int kABufs = 2 / KC;                 // token-tile buffers
    static constexpr int kBufCols = 256;                  // TMEM columns of a stage's KC accumulators
    static constexpr uint32_t kBTile = kTN * kKA * 4;     // one K chunk of a stage, hi or lo
    static constexpr uint32_t kABuf = 2 * KC * kATile;    // hi chunks, lo chunks
    static constexpr uint32_t kBBuf = 2 * KC * kBTile;
    static constexpr size_t kSmem = 1024 + kABufs * (size_t)kABuf + 2 * (size_t)kBBuf + 8 * 17 + 16;
    static_assert(kSmem <= 232448, "shared memory per CTA");
};

struct TParams {
    const float* Yb;   // g~ rows [NT][k_out]
    float* out;
    int64_t NT;        // tokens of this call
    int64_t tok0;      // global token index of token 0 (first example of the call times T)
    int64_t n_q, ld_q;
    int n_tt, n_nt;    // token tiles, query stages
    float scale, beta;
    unsigned int* err;
};

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
// x to TF32's 10 mantissa bits, nearest. From the value that would round past the largest on, the bits
// below are cut off; a NaN keeps its quiet bit (0x7FFFFFFF, the NaN of CUDA arithmetic and of the tensor pipe,
// would carry into the sign and become zero). An infinity's lo is a NaN, so its products are NaN.
__device__ __forceinline__ float round_tf32(float x) {
    const uint32_t u = __float_as_uint(x), mag = u & 0x7FFFFFFFu;
    const uint32_t r = mag >= 0x7F7FF000u ? u : u + 0x1000u;
    return __uint_as_float((r & 0xFFFFE000u) | (mag > 0x7F800000u ? 0x00400000u : 0u));
}
__device__ __forceinline__ void split_tf32(float x, float& hi, float& lo) {
    hi = round_tf32(x);
    lo = round_tf32(x - hi);
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
// bounded wait on the phase `parity` of `bar` without an abort flag (teardown drains)
__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity, unsigned int* err) {
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > kTimeoutNs) {
            atomicOr(err, kErrTimeout);
            break;
        }
}

// hi/lo halves of R: row (q, r) of Rs = R[q * ld_R + r * k_in + c]
__global__ void split_r_kernel(const float* __restrict__ R, int64_t n_q, int64_t ld_R, int64_t per,
                               float* __restrict__ Rhi, float* __restrict__ Rlo) {
    const int64_t total = n_q * per;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = e / per, rc = e - q * per;
        float h, l;
        split_tf32(R[q * ld_R + rc], h, l);
        Rhi[e] = h;
        Rlo[e] = l;
    }
}

template <int KG, int KC>
__global__ void __launch_bounds__(kThreads, 1)
token_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmRh,
                const __grid_constant__ CUtensorMap tmRl, const TParams p) {
    using C = Cfg<KC>;
    constexpr int kTN = C::kTN, G = kTN / KG;  // G: queries per stage
    constexpr uint32_t kABufs = C::kABufs, kABuf = C::kABuf, kBBuf = C::kBBuf, kBTile = C::kBTile;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* abuf = smem;                  // [kABufs] a~ hi | lo
    uint8_t* bbuf = smem + kABufs * kABuf; // [2] R hi | lo
    uint64_t* bars = (uint64_t*)(bbuf + 2 * kBBuf);
    uint64_t* a_raw = bars;        // [2] TMA landed (1 + tx)
    uint64_t* a_full = bars + 2;   // [2] split done (2 warps)
    uint64_t* a_empty = bars + 4;  // [2] MMAs done with the token tile (commit)
    uint64_t* b_full = bars + 6;   // [2] (1 + tx)
    uint64_t* b_empty = bars + 8;  // [2] (commit)
    uint64_t* tfull = bars + 10;   // [2] accumulator ready (commit)
    uint64_t* tempty = bars + 12;  // [2] accumulator drained (4)
    uint64_t* mma_done = bars + 14;
    uint32_t* tmem_slot = (uint32_t*)(bars + 17);
    volatile int* abort = (volatile int*)(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&a_raw[i]), 1);
            mbar_init(smem_u32(&a_full[i]), 2);
            mbar_init(smem_u32(&a_empty[i]), 1);
            mbar_init(smem_u32(&b_full[i]), 1);
            mbar_init(smem_u32(&b_empty[i]), 1);
            mbar_init(smem_u32(&tfull[i]), 1);
            mbar_init(smem_u32(&tempty[i]), 4);
        }
        mbar_init(smem_u32(mma_done), 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 || warp == 3) {
        // ---------------- split warps: a~ tile raw (TMA) -> hi in place + lo
        const int pt = (warp == 0 ? 0 : 32) + lane;
        uint32_t it = 0;
        for (int u = blockIdx.x; u < p.n_tt; u += gridDim.x, ++it) {
            const uint32_t ab = it % kABufs, ph = (it / kABufs) & 1u;
            bool got = warp_wait(smem_u32(&a_raw[ab]), ph, abort, p.err);
            if (!got) break;
            uint8_t* hi = abuf + ab * kABuf;
            uint8_t* lo = hi + KC * kATile;
#pragma unroll 4
            for (uint32_t off = (uint32_t)pt * 16u; off < KC * kATile; off += 64u * 16u) {
                const float4 v = *reinterpret_cast<const float4*>(hi + off);
                float4 h, l;
                split_tf32(v.x, h.x, l.x);
                split_tf32(v.y, h.y, l.y);
                split_tf32(v.z, h.z, l.z);
                split_tf32(v.w, h.w, l.w);
                *reinterpret_cast<float4*>(hi + off) = h;
                *reinterpret_cast<float4*>(lo + off) = l;
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&a_full[ab]));
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the warp waits, one lane issues
        constexpr uint32_t idesc = idesc_tf32(kTM, kTN);
        uint32_t it = 0, rb = 0, tt = 0;
        bool ok = true;
        for (int u = blockIdx.x; ok && u < p.n_tt; u += gridDim.x, ++it) {
            const uint32_t ab = it % kABufs;
            if (!warp_wait(smem_u32(&a_full[ab]), (it / kABufs) & 1u, abort, p.err)) break;
            tc_fence_after();
            const uint32_t ahs = smem_u32(abuf + ab * kABuf);
            for (int j = 0; j < p.n_nt; ++j, ++rb, ++tt) {
                const uint32_t s = rb & 1u, b = tt & 1u;
                if (!warp_wait(smem_u32(&tempty[b]), ((tt >> 1) & 1u) ^ 1u, abort, p.err) ||
                    !warp_wait(smem_u32(&b_full[s]), (rb >> 1) & 1u, abort, p.err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t bhs = smem_u32(bbuf + s * kBBuf);
                const uint32_t d = tmem + b * C::kBufCols;
                // lo * hi and hi * lo of every k, then hi * hi (K = 8 tf32 = 32 bytes per instruction);
                // KC = 2: the first chunk's hi * hi in an accumulator of its own
                if (elect_one()) {
#pragma unroll
                    for (int pr = 0; pr < 3; ++pr)
#pragma unroll
                        for (int c = 0; c < KC; ++c) {
                            const uint64_t ad = sw128_desc(ahs + (pr == 0 ? KC + c : c) * kATile);
                            const uint64_t bd = sw128_desc(bhs + (pr == 1 ? KC + c : c) * kBTile);
#pragma unroll
                            for (int k = 0; k < kKA / 8; ++k)
                                if (KC > 1 && pr == 2 && c == 0)
                                    mma_tf32(d + kTN, ad + 2 * k, bd + 2 * k, idesc, k > 0 ? 1u : 0u);
                                else
                                    mma_tf32(d, ad + 2 * k, bd + 2 * k, idesc, (pr > 0 || c > 0 || k > 0) ? 1u : 0u);
                        }
                    mma_commit(smem_u32(&b_empty[s]));
                    mma_commit(smem_u32(&tfull[b]));
                }
                __syncwarp();
            }
            if (!ok) break;
            if (elect_one()) mma_commit(smem_u32(&a_empty[ab]));
            __syncwarp();
        }
        if (elect_one()) {
            mma_commit(smem_u32(mma_done));
            drain_wait(smem_u32(mma_done), 0, p.err);
        }
        __syncwarp();
    } else if (warp == 2) {
        if (lane == 0) {
            // ---------------- TMA producer
            uint32_t it = 0, rb = 0;
            uint32_t a_par[2], b_par[2];
            bool a_iss[2] = {false, false}, b_iss[2] = {false, false}, ok = true;
            for (int u = blockIdx.x; ok && u < p.n_tt; u += gridDim.x, ++it) {
                const uint32_t ab = it % kABufs, aph = (it / kABufs) & 1u;
                if (!wait_bounded(smem_u32(&a_empty[ab]), aph ^ 1u, abort, p.err)) break;
                mbar_arrive_tx(smem_u32(&a_raw[ab]), KC * kATile);
#pragma unroll
                for (int c = 0; c < KC; ++c)
                    tma_load_2d(smem_u32(abuf + ab * kABuf + c * kATile), &tmA, kKA * c, u * kTM, smem_u32(&a_raw[ab]));
                a_iss[ab] = true;
                a_par[ab] = aph;
                for (int j = 0; j < p.n_nt; ++j, ++rb) {
                    const uint32_t s = rb & 1u, ph = (rb >> 1) & 1u;
                    if (!wait_bounded(smem_u32(&b_empty[s]), ph ^ 1u, abort, p.err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t dst = smem_u32(bbuf + s * kBBuf), bar = smem_u32(&b_full[s]);
                    mbar_arrive_tx(bar, kBBuf);
#pragma unroll
                    for (int c = 0; c < KC; ++c) {
                        tma_load_2d(dst + c * kBTile, &tmRh, kKA * c, j * kTN, bar);
                        tma_load_2d(dst + (KC + c) * kBTile, &tmRl, kKA * c, j * kTN, bar);
                    }
                    b_iss[s] = true;
                    b_par[s] = ph;
                }
            }
            // copies still in flight when the consumers stopped early land before the CTA exits
            for (int i = 0; i < 2; ++i) {
                if (a_iss[i]) drain_wait(smem_u32(&a_raw[i]), a_par[i], p.err);
                if (b_iss[i]) drain_wait(smem_u32(&b_full[i]), b_par[i], p.err);
            }
        }
    } else {
        // ---------------- epilogue: TMEM -> weighted sums over r -> out
        const int q4 = warp & 3, row = q4 * 32 + lane;
        uint32_t tt = 0;
        bool stop = false;
        for (int u = blockIdx.x; !stop && u < p.n_tt; u += gridDim.x) {
            const int64_t tok = (int64_t)u * kTM + row;
            const bool valid = tok < p.NT;
            float g[KG];
#pragma unroll
            for (int c = 0; c < KG; c += 4) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (valid) v = *reinterpret_cast<const float4*>(p.Yb + tok * KG + c);
                g[c] = v.x, g[c + 1] = v.y, g[c + 2] = v.z, g[c + 3] = v.w;
            }
            // beta != 0: the previous values of a stage's outputs are loaded one stage ahead,
            // so that their latency hides behind the wait for the accumulator
            const bool rmw = p.beta != 0.f;
            float old[G];
            auto prefetch = [&](int j) {
#pragma unroll
                for (int gq = 0; gq < G; ++gq) {
                    const int64_t q = (int64_t)j * G + gq;
                    old[gq] = (rmw && valid && q < p.n_q) ? p.out[q * p.ld_q + p.tok0 + tok] : 0.f;
                }
            };
            prefetch(0);
            for (int j = 0; j < p.n_nt; ++j, ++tt) {
                const uint32_t b = tt & 1u;
                bool got = warp_wait(smem_u32(&tfull[b]), (tt >> 1) & 1u, abort, p.err);
                if (epi_any(!got)) {
                    stop = true;
                    break;
                }
                tc_fence_after();
                const uint32_t tb = tmem + ((uint32_t)(q4 * 32) << 16) + b * C::kBufCols;
                float acc[G];
#pragma unroll
                for (int gq = 0; gq < G; ++gq) {
                    float sum[4] = {0.f, 0.f, 0.f, 0.f};  // four chains: less rounding
#pragma unroll
                    for (int c = 0; c < KG; c += 16) {
                        float v[16];
                        tmem_ld16(tb + gq * KG + c, v);
                        if constexpr (KC > 1) {
                            float w[16];
                            tmem_ld16(tb + kTN + gq * KG + c, w);
#pragma unroll
                            for (int i = 0; i < 16; ++i) v[i] += w[i];
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) sum[i & 3] = fmaf(g[c + i], v[i], sum[i & 3]);
                    }
                    const float s = (sum[0] + sum[1]) + (sum[2] + sum[3]);
                    acc[gq] = rmw ? p.beta * old[gq] + p.scale * s : p.scale * s;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&tempty[b]));
                if (valid) {
#pragma unroll
                    for (int gq = 0; gq < G; ++gq) {
                        const int64_t q = (int64_t)j * G + gq;
                        if (q < p.n_q) p.out[q * p.ld_q + p.tok0 + tok] = acc[gq];
                    }
                }
                if (j + 1 < p.n_nt) prefetch(j + 1);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
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

// 2-D map over fp32 rows of ka elements: box 32 x box_rows, 128-byte swizzle, zero fill past ka and the last row.
bool make_rows_map(CUtensorMap* tm, const float* X, int64_t rows, int ka, int box_rows) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)ka, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ka * 4};
    cuuint32_t box[2] = {(cuuint32_t)kKA, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(X), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool is_sm103() {
    static int sm103 = -1;
    if (sm103 < 0) {
        int dev = 0, major = 0, minor = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
        sm103 = (major == 10 && minor == 3) ? 1 : 0;
    }
    return sm103 == 1;
}

}  // namespace

size_t token_tc_split_bytes(int ka, int kg, int64_t n_q) {
    return (2 * sizeof(float) * (size_t)n_q * (size_t)ka * (size_t)kg + 255) & ~(size_t)255;
}

bool token_tc_supported(int ka, int kg, int64_t n_q) {
    return is_sm103() && encode_fn() && ka > 16 && ka <= 64 && ka % 4 == 0 && (kg == 16 || kg == 32 || kg == 64) && n_q >= 1 &&
           n_q * kg < ((int64_t)1 << 31) && device_error_word() != nullptr;
}

// Rs: token_tc_split_bytes(ka, kg, n_q) of device scratch for R's hi and lo halves.
cudaError_t launch_token_scores_tc(const float* Ya, const float* Yb, int64_t n, int64_t T, int ka, int kg,
                                   const float* R, int64_t n_q, int64_t ld_R, float scale, float* out, int64_t ld_q,
                                   int64_t i0, float beta, float* Rs, cudaStream_t s) {
    const int64_t NT = n * T;
    if (NT == 0 || n_q == 0) return cudaSuccess;
    if (NT >= ((int64_t)1 << 31) || ((uintptr_t)Ya & 15) || ((uintptr_t)Yb & 15) || ((uintptr_t)Rs & 15))
        return cudaErrorInvalidValue;
    float* Rhi = Rs;
    float* Rlo = Rs + n_q * kg * ka;
    const int KC = ka > kKA ? 2 : 1, tn = 256 / KC;
    CUtensorMap mA, mRh, mRl;
    if (!make_rows_map(&mA, Ya, NT, ka, kTM) || !make_rows_map(&mRh, Rhi, n_q * kg, ka, tn) ||
        !make_rows_map(&mRl, Rlo, n_q * kg, ka, tn))
        return cudaErrorInvalidValue;
    note_launches(1);
    split_r_kernel<<<(unsigned)((n_q * kg * ka + 255) / 256 < 1024 ? (n_q * kg * ka + 255) / 256 : 1024), 256, 0, s>>>(
        R, n_q, ld_R, (int64_t)kg * ka, Rhi, Rlo);
    TParams p;
    p.Yb = Yb;
    p.out = out;
    p.NT = NT;
    p.tok0 = i0 * T;
    p.n_q = n_q;
    p.ld_q = ld_q;
    p.n_tt = (int)((NT + kTM - 1) / kTM);
    p.n_nt = (int)((n_q * kg + tn - 1) / tn);
    p.scale = scale;
    p.beta = beta;
    p.err = device_error_word();
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    const unsigned grid = (unsigned)(p.n_tt < sms ? p.n_tt : sms);
    note_launches(1);
#define TDA_TOKENS(kgv, kcv)                                                             \
    if (kg == kgv && KC == kcv) {                                                        \
        cudaError_t e = smem_attr_once<token_tc_kernel<kgv, kcv>>((int)Cfg<kcv>::kSmem); \
        if (e != cudaSuccess) return e;                                                  \
        token_tc_kernel<kgv, kcv><<<grid, kThreads, Cfg<kcv>::kSmem, s>>>(mA, mRh, mRl, p); \
    }
    TDA_TOKENS(16, 1) TDA_TOKENS(32, 1) TDA_TOKENS(64, 1) TDA_TOKENS(16, 2) TDA_TOKENS(32, 2) TDA_TOKENS(64, 2)
#undef TDA_TOKENS
    return cudaGetLastError();
}

}  // namespace tda
