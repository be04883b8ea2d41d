// k_project_simt.cu -- sign-matrix dump and the generic (CUDA-core) factored
// projection, for any layer shape, fp32 or bf16 factors.
//
// Factored projection, Eq. 2: for every example n,
//   At = A_n S_in (T x k_in), Bt = B_n S_out (T x k_out),
//   Phi_n = scale * Bt^T At (k_out x k_in), scale = 1/sqrt(k_in k_out),
// with S generated on chip from the counter hash (App. A.2) and never stored.
// The general kernel is the fallback for shapes the tensor-core kernels do not
// cover (identity maps, k above their blocks); project_small_kernel takes short
// fp32 jobs of narrow layers, with the general kernel's sums bit for bit.
#include <cuda_bf16.h>
#include <math.h>

#include "tda_internal.cuh"

namespace tda {
namespace {

constexpr int kTile = 64;      // Phi tile edge: rows i (k_out), columns j (k_in)
constexpr int kTokChunk = 16;  // tokens per contraction step
constexpr int kDChunk = 64;    // rows of S per sign word
constexpr int kThreads = 256;

__device__ __forceinline__ float load_elem(const float* p) { return __ldg(p); }
__device__ __forceinline__ float load_elem(const __nv_bfloat16* p) { return __bfloat162float(*p); }

__global__ void proj_entries_kernel(uint64_t key, int kind, int64_t rows, int32_t cols,
                                    int8_t* __restrict__ out) {
    const int64_t total = rows * (int64_t)cols;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / cols;
        const int32_t c = (int32_t)(e - r * cols);
        int8_t v;
        if (kind == TDA_PROJ_IDENTITY)
            v = (r == c) ? 1 : 0;
        else
            v = ((sign_word(key, (uint32_t)c, (uint64_t)(r >> 6)) >> (r & 63)) & 1u) ? -1 : 1;
        out[e] = v;
    }
}

// X[t][j] = sum_c src[t0+t][c] * S[c][c0+j] for a chunk of kTokChunk tokens
// and a kTile-wide column tile. Thread (t = tid/16, 4 columns at (tid%16)*4).
template <typename T>
__device__ __forceinline__ void project_chunk(const T* __restrict__ src, int64_t Tn, int64_t d,
                                              int64_t t0, uint64_t key, int kind, int c0,
                                              float (*Xs)[kTile], float (*Vs)[kDChunk + 1],
                                              uint64_t* Ws) {
    const int tid = threadIdx.x;
    const int t = tid / 16, jq = (tid % 16) * 4;
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    for (int64_t dc = 0; dc < d; dc += kDChunk) {
        __syncthreads();  // previous readers of Vs / Ws are done
        for (int e = tid; e < kTokChunk * kDChunk; e += kThreads) {
            const int tt = e / kDChunk, cc = e % kDChunk;
            const int64_t tg = t0 + tt, cg = dc + cc;
            Vs[tt][cc] = (tg < Tn && cg < d) ? load_elem(src + tg * d + cg) : 0.f;
        }
        if (kind == TDA_PROJ_RADEMACHER && tid < kTile)
            Ws[tid] = sign_word(key, (uint32_t)(c0 + tid), (uint64_t)(dc >> 6));
        __syncthreads();
        if (kind == TDA_PROJ_RADEMACHER) {
            const uint64_t w0 = Ws[jq], w1 = Ws[jq + 1], w2 = Ws[jq + 2], w3 = Ws[jq + 3];
#pragma unroll 8
            for (int r = 0; r < kDChunk; ++r) {
                const float v = Vs[t][r];
                o[0] += ((w0 >> r) & 1u) ? -v : v;
                o[1] += ((w1 >> r) & 1u) ? -v : v;
                o[2] += ((w2 >> r) & 1u) ? -v : v;
                o[3] += ((w3 >> r) & 1u) ? -v : v;
            }
        } else {  // identity map: S[c][j] = [c == j]
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t jg = c0 + jq + q;
                if (jg >= dc && jg < dc + kDChunk) o[q] += Vs[t][jg - dc];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) Xs[t][jq + q] = o[q];
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
project_simt_kernel(const T* __restrict__ A, const T* __restrict__ B, int64_t Tn, int64_t d_in,
                    int64_t d_out, int k_in, int k_out, uint64_t key_in, uint64_t key_out,
                    int kind, float scale, float* __restrict__ phi, int64_t ld_phi) {
    __shared__ float Xs[kTokChunk][kTile];       // At chunk, column tile j0
    __shared__ float Ys[kTokChunk][kTile];       // Bt chunk, column tile i0
    __shared__ float Vs[kTokChunk][kDChunk + 1]; // staged factor rows
    __shared__ uint64_t Ws[kTile];               // sign words of the current 64-row block

    const int64_t n = blockIdx.x;
    const int i0 = blockIdx.y * kTile;
    const int j0 = blockIdx.z * kTile;
    const T* An = A + n * Tn * d_in;
    const T* Bn = B + n * Tn * d_out;
    const int tid = threadIdx.x;
    const int ri = (tid / 16) * 4, cj = (tid % 16) * 4;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;

    for (int64_t t0 = 0; t0 < Tn; t0 += kTokChunk) {
        project_chunk(An, Tn, d_in, t0, key_in, kind, j0, Xs, Vs, Ws);
        project_chunk(Bn, Tn, d_out, t0, key_out, kind, i0, Ys, Vs, Ws);
        __syncthreads();
#pragma unroll 4
        for (int t = 0; t < kTokChunk; ++t) {
            float y[4], x[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) y[a] = Ys[t][ri + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) x[b] = Xs[t][cj + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(y[a], x[b], acc[a][b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ri + a, j = j0 + cj + b;
            if (i < k_out && j < k_in) phi[n * ld_phi + (int64_t)i * k_in + j] = acc[a][b] * scale;
        }
}

// Few tokens of a narrow fp32 layer (T <= 64, d <= 512, k <= 16): one CTA per example, half its
// threads on each side. Bound by latency: a (token, column) sum is a chain of d dependent adds.
// A thread runs CPT such chains of one token (CPT = 4, 2, 1 for T <= 64, 32, 16, so that a side's
// 256 threads cover T x 16 columns), with 64-feature chunks of the factors staged in shared
// memory one chunk ahead in registers. The adds of a chain, and of an entry of Phi over the
// tokens, run in the general kernel's order, so the features are the same bit for bit (an fp64
// preconditioner state behind them sees no change). 64 examples, 256 -> 256, T = 32, k = 16:
// 63 us in the general kernel, which computes 64 columns whatever k is, 16 tokens at a time;
// 8 us here.
constexpr int kSmallT = 64, kSmallD = 512, kSmallK = 16;
constexpr int kSmallLd = kDChunk + 4;  // padded row: 16-byte loads of different tokens miss each other's banks

template <int CPT>
__global__ void __launch_bounds__(512)
project_small_kernel(const float* __restrict__ A, const float* __restrict__ B, int Tn, int d_in, int d_out, int k_in,
                     int k_out, uint64_t key_in, uint64_t key_out, float scale, float* __restrict__ phi,
                     int64_t ld_phi) {
    constexpr int kTok = 16 * CPT;            // tokens the threads of a side cover
    constexpr int kLoads = kTok * kDChunk / 4 / 256;  // 16-byte groups per thread and chunk
    __shared__ __align__(16) float Vs[2][kTok][kSmallLd];
    __shared__ float Xs[2][kTok][kSmallK + 1];
    const int side = threadIdx.x >> 8, tid = threadIdx.x & 255;
    const int d = side ? d_out : d_in;
    const uint64_t key = side ? key_out : key_in;
    const float* src = side ? B + (int64_t)blockIdx.x * Tn * d_out : A + (int64_t)blockIdx.x * Tn * d_in;
    const int t = tid / (16 / CPT), c0 = tid % (16 / CPT) * CPT;
    const int dmax = d_in > d_out ? d_in : d_out;
    float4 next[kLoads];
    auto load = [&](int dc) {
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int e = tid + 256 * i, tt = e / (kDChunk / 4), cc = dc + e % (kDChunk / 4) * 4;
            next[i] = tt < Tn && cc < d ? __ldg(reinterpret_cast<const float4*>(src + (int64_t)tt * d + cc))
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float o[CPT];
#pragma unroll
    for (int q = 0; q < CPT; ++q) o[q] = 0.f;
    load(0);
    for (int dc = 0; dc < dmax; dc += kDChunk) {
        __syncthreads();  // the previous chunk is read
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int e = tid + 256 * i;
            *reinterpret_cast<float4*>(&Vs[side][e / (kDChunk / 4)][e % (kDChunk / 4) * 4]) = next[i];
        }
        if (dc + kDChunk < dmax) load(dc + kDChunk);
        uint32_t w[CPT][2];
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const uint64_t x = sign_word(key, (uint32_t)(c0 + q), (uint64_t)(dc >> 6));
            w[q][0] = (uint32_t)x;
            w[q][1] = (uint32_t)(x >> 32);
        }
        __syncthreads();
        if (dc < d) {
#pragma unroll
            for (int half = 0; half < 2; ++half)
#pragma unroll
                for (int r = 0; r < 32; r += 4) {
                    const float4 v4 = *reinterpret_cast<const float4*>(&Vs[side][t][32 * half + r]);
                    const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int q = 0; q < CPT; ++q)
                            o[q] += __uint_as_float(__float_as_uint(v[i]) ^
                                                    ((w[q][half] << (31 - r - i)) & 0x80000000u));
                }
        }
    }
#pragma unroll
    for (int q = 0; q < CPT; ++q) Xs[side][t][c0 + q] = o[q];
    __syncthreads();
    const int e = threadIdx.x, i = e / kSmallK, j = e % kSmallK;  // Phi entry (i, j): i < 16 for half the threads
    if (i < k_out && j < k_in) {
        float acc = 0.f;
#pragma unroll 8
        for (int tt = 0; tt < Tn; ++tt) acc = fmaf(Xs[1][tt][i], Xs[0][tt][j], acc);
        phi[blockIdx.x * ld_phi + (int64_t)i * k_in + j] = acc * scale;
    }
}

}  // namespace

// The line is not where the tensor-core kernel (k_project_flex.cu) becomes faster but where a job is no longer
// small: below it features stay, bit for bit, what an fp64 preconditioner has seen before. d = 256, T = 32, k = 16,
// 8 or 64 examples: 6.6 us here, 9.5 us there; d = 512, T = 64: 16 to 128 examples 19.9 and 15.8 us, 256 examples
// 36.7 and 17.8 us; 16384 examples of one token, d = 512: 506 and 39 us. These sums are fp32 chains in order
// (T = 64, d = 512: 6.8e-7 off), the other kernel is closer (1.8e-7).
bool project_small_supported(const tda_layer_desc& L, const void* A, const void* B, int64_t N) {
    return L.kind == TDA_PROJ_RADEMACHER && L.T >= 1 && L.T <= kSmallT && L.d_in <= kSmallD && L.d_out <= kSmallD &&
           L.k_in <= kSmallK && L.k_out <= kSmallK && L.d_in % 4 == 0 && L.d_out % 4 == 0 && N <= 16384 / L.T &&
           !((uintptr_t)A & 15) && !((uintptr_t)B & 15);
}

// bf16 factors, the larger k in 65 .. 127 or unequal: whether the general kernel beats the tensor-core one, which
// computes tiles of 128 tokens x 128 + 128 columns whatever the job is (28.5 us a tile and 8.3 ns a feature of both
// widths). The general kernel takes 16 tokens and 64 x 64 features a CTA at a time, 1.2 us and 40 ns a feature, about
// 240 CTAs at once. T = 8, k = 100 x 96, measured here and there: 16 examples d = 64 8.7 and 30 us, d = 256 22 and
// 33 us, d = 1024 76 and 46 us; 152 examples d = 64 20 and 32 us, d = 256 63 and 36 us; 3000 examples d = 64 329 and
// 561 us; T = 64, 16 examples, d = 64 26 and 30 us. Within 15 % of the line either may be the faster one.
bool project_short_supported(const tda_layer_desc& L, int64_t N) {
    if (L.T > 128) return false;
    const double d = (double)(L.d_in + L.d_out), sms = (double)project_tc_max_grid();
    const double ctas = (double)N * (double)((L.k_in + 63) / 64) * (double)((L.k_out + 63) / 64);
    const double general = fmax(1.0, ctas / (240.0 / 152.0 * sms)) * ((double)((L.T + 15) / 16) * (1.2 + 0.04 * d) + 2.0);
    return general < ceil((double)N / sms) * (28.5 + 0.0083 * d);
}

cudaError_t launch_project_small(const tda_layer_desc& L, const void* A, const void* B, int64_t N, float* phi,
                                 int64_t ld_phi, cudaStream_t s) {
    if (N == 0) return cudaSuccess;
    const uint64_t key_in = side_key(L.seed, L.layer, 0), key_out = side_key(L.seed, L.layer, 1);
    auto launch = [&](auto kernel) {
        note_launches(1);
        kernel<<<(unsigned)N, 512, 0, s>>>((const float*)A, (const float*)B, (int)L.T, (int)L.d_in, (int)L.d_out,
                                           L.k_in, L.k_out, key_in, key_out, projection_scale(L), phi, ld_phi);
    };
    if (L.T > 32)
        launch(project_small_kernel<4>);
    else if (L.T > 16)
        launch(project_small_kernel<2>);
    else
        launch(project_small_kernel<1>);
    return cudaGetLastError();
}

cudaError_t launch_proj_entries(uint64_t key, int kind, int64_t rows, int32_t cols, int8_t* out,
                                cudaStream_t s) {
    const int64_t total = rows * (int64_t)cols;
    if (total == 0) return cudaSuccess;
    int64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    note_launches(1);
    proj_entries_kernel<<<(unsigned)blocks, 256, 0, s>>>(key, kind, rows, cols, out);
    return cudaGetLastError();
}

float projection_scale(const tda_layer_desc& L) {
    if (L.kind == TDA_PROJ_IDENTITY) return 1.0f;
    return (float)(1.0 / (sqrt((double)L.k_in) * sqrt((double)L.k_out)));
}

cudaError_t launch_project_simt(const tda_layer_desc& L, tda_dtype dt, const void* A, const void* B,
                                int64_t N, float* phi, int64_t ld_phi, cudaStream_t s) {
    if (N == 0) return cudaSuccess;
    const uint64_t key_in = side_key(L.seed, L.layer, 0);
    const uint64_t key_out = side_key(L.seed, L.layer, 1);
    dim3 grid((unsigned)N, (unsigned)((L.k_out + kTile - 1) / kTile),
              (unsigned)((L.k_in + kTile - 1) / kTile));
    const float scale = projection_scale(L);
    note_launches(1);
    if (dt == TDA_BF16)
        project_simt_kernel<__nv_bfloat16><<<grid, kThreads, 0, s>>>(
            (const __nv_bfloat16*)A, (const __nv_bfloat16*)B, L.T, L.d_in, L.d_out, L.k_in,
            L.k_out, key_in, key_out, L.kind, scale, phi, ld_phi);
    else
        project_simt_kernel<float><<<grid, kThreads, 0, s>>>(
            (const float*)A, (const float*)B, L.T, L.d_in, L.d_out, L.k_in, L.k_out, key_in,
            key_out, L.kind, scale, phi, ld_phi);
    return cudaGetLastError();
}

}  // namespace tda
