// k_precond.cu -- damped Fisher preconditioner of the queries, for a batch of
// layers with the same feature count D.
//
// App. B.3: curvature-based methods fit a curvature matrix over the training
// gradients and precondition the queries layer by layer; App. B.2: damping is
// a multiple of the layer's mean eigenvalue. On projected features phi (D per
// example and layer) the fit is the empirical Fisher F = (1/N) sum_i phi_i
// phi_i^T, and a query q becomes qhat = (F + lambda I)^{-1} q.
//
// Per-layer state (caller-owned, tda_precondition_state_bytes each, layers
// back to back): 64-byte header | M (D x D) | Dinv (ceil(D/32) blocks of
// 32 x 32), elements float or double. After FACTOR, M holds L strictly below
// its 32 x 32 diagonal blocks; each diagonal block of L is held as its inverse
// in Dinv.
//   FIT     M += Phi^T Phi (lower 128x128 tiles; register-blocked SYRK)
//   FACTOR  M <- L, L L^T = M/n_total + lambda I: right-looking Cholesky in
//           32-column steps; each step factors the diagonal block inside every
//           panel CTA (so it needs no launch of its own), solves the panel, then
//           updates the trailing lower triangle. The inverse of every diagonal
//           block is kept in Dinv.
//   APPLY   forward and backward block substitution; with Dinv each 32-row
//           block step is a small matrix product instead of a serial chain.
// Every launch covers all layers of the call (grid z or y = layer).
//
// Blocked path (fp32 state, D a multiple of 64 and at least 256): the same
// right-looking Cholesky in 256-column panels. Per panel: the 256 x 256 diagonal
// block is factored in shared memory by one CTA (diag_panel_kernel), the rows
// below it are solved against it (solve_kernel, x L_BB^T = a), and the trailing
// lower triangle takes the rank-256 update M -= P P^T on the tensor cores (3xTF32,
// launch_gemm_nt_tc_batched). After the last panel, L^T is copied into M's upper triangle.
// APPLY then solves the query rows panel by panel: a 256-wide triangular solve, and
// the rest of every row updated by a tensor-core product with L's panel (forward)
// or with L^T's panel from the upper triangle (backward).
#include <math.h>

#include "tda_internal.cuh"

namespace tda {
namespace {

constexpr int kNB = 32;  // Cholesky / substitution block

template <typename TS>
struct St {
    char* base;
    int64_t D;
    size_t bytes;
    __device__ __forceinline__ double* header(int l) const { return (double*)(base + (size_t)l * bytes); }
    __device__ __forceinline__ TS* M(int l) const { return (TS*)(base + (size_t)l * bytes + 64); }
    __device__ __forceinline__ TS* Dinv(int l) const { return M(l) + D * D; }
};

template <typename TS>
St<TS> state_of(void* state, int64_t D) {
    St<TS> s;
    s.base = (char*)state;
    s.D = D;
    s.bytes = tda_precondition_state_bytes(D, sizeof(TS) == 8 ? TDA_F64 : TDA_F32);
    return s;
}

// ---------------------------------------------------------------- FIT (fp32)
// Tile 128 x 128 of M for rows a0.., cols b0.. (b-tile <= a-tile), K = rows of
// Phi in chunks of 16. Thread (ty, tx) of 16 x 16 owns rows {ty*4+u, 64+ty*4+u}
// and columns {tx*4+v, 64+tx*4+v}: 8 x 8 accumulators, float4 shared reads.
constexpr int kFT = 128, kFK = 16;

__global__ void __launch_bounds__(256, 2)
fit_f32_kernel(St<float> st, const float* __restrict__ phi, int64_t n, int64_t ld) {
    if (blockIdx.x > blockIdx.y) return;  // upper tile: M is used through its lower triangle
    __shared__ __align__(16) float Xa[kFK][kFT];
    __shared__ __align__(16) float Xb[kFK][kFT];
    const int l = blockIdx.z;
    const int64_t D = st.D;
    const float* ph = phi + (int64_t)l * D;
    const int64_t a0 = (int64_t)blockIdx.y * kFT, b0 = (int64_t)blockIdx.x * kFT;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    float acc[8][8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
    const bool vec = ((ld & 3) == 0) && ((D & 3) == 0) && (((uintptr_t)ph & 15) == 0);
    for (int64_t r0 = 0; r0 < n; r0 += kFK) {
        // 16 rows x 128 columns per operand: 512 float4 each, 2 per thread
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = tid + h * 256;
            const int rr = e >> 5, c4 = (e & 31) * 4;
            const int64_t r = r0 + rr;
            float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
            if (r < n) {
                const float* row = ph + r * ld;
                if (vec && a0 + c4 + 3 < D) {
                    va = *reinterpret_cast<const float4*>(row + a0 + c4);
                } else {
                    float t[4];
                    for (int i = 0; i < 4; ++i) t[i] = (a0 + c4 + i < D) ? row[a0 + c4 + i] : 0.f;
                    va = make_float4(t[0], t[1], t[2], t[3]);
                }
                if (vec && b0 + c4 + 3 < D) {
                    vb = *reinterpret_cast<const float4*>(row + b0 + c4);
                } else {
                    float t[4];
                    for (int i = 0; i < 4; ++i) t[i] = (b0 + c4 + i < D) ? row[b0 + c4 + i] : 0.f;
                    vb = make_float4(t[0], t[1], t[2], t[3]);
                }
            }
            *reinterpret_cast<float4*>(&Xa[rr][c4]) = va;
            *reinterpret_cast<float4*>(&Xb[rr][c4]) = vb;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kFK; ++k) {
            const float4 x0 = *reinterpret_cast<const float4*>(&Xa[k][ty * 4]);
            const float4 x1 = *reinterpret_cast<const float4*>(&Xa[k][64 + ty * 4]);
            const float4 y0 = *reinterpret_cast<const float4*>(&Xb[k][tx * 4]);
            const float4 y1 = *reinterpret_cast<const float4*>(&Xb[k][64 + tx * 4]);
            const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
            const float y[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(x[u], y[v], acc[u][v]);
        }
        __syncthreads();
    }
    float* M = st.M(l);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int64_t a = a0 + (u < 4 ? ty * 4 + u : 64 + ty * 4 + (u - 4));
        if (a >= D) continue;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int64_t b = b0 + (v < 4 ? tx * 4 + v : 64 + tx * 4 + (v - 4));
            if (b < D) M[a * D + b] += acc[u][v];
        }
    }
}

// ---------------------------------------------------------------- FIT (fp64)
// fp64 runs at two multiply-adds a clock and SM here, so what counts is that every SM has work:
// T x T tiles with T = 64, or 16 when 64 would leave SMs idle (D = 256: 10 tiles, 75 us for 64
// rows; 136 tiles of 16). An entry's sum runs over the rows in order whatever T is.
template <int T>
__global__ void __launch_bounds__(256)
fit_f64_kernel(St<double> st, const float* __restrict__ phi, int64_t n, int64_t ld) {
    if (blockIdx.x > blockIdx.y) return;
    constexpr int K = 32, R = T / 16;
    __shared__ double Xa[K][T + 1];
    __shared__ double Xb[K][T + 1];
    const int l = blockIdx.z;
    const int64_t D = st.D;
    const float* ph = phi + (int64_t)l * D;
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const int64_t a0 = (int64_t)blockIdx.y * T, b0 = (int64_t)blockIdx.x * T;
    double acc[R][R] = {};
    for (int64_t r0 = 0; r0 < n; r0 += K) {
        for (int e = tid; e < K * T; e += 256) {
            const int rr = e / T, cc = e % T;
            const int64_t r = r0 + rr;
            Xa[rr][cc] = (r < n && a0 + cc < D) ? (double)ph[r * ld + a0 + cc] : 0.0;
            Xb[rr][cc] = (r < n && b0 + cc < D) ? (double)ph[r * ld + b0 + cc] : 0.0;
        }
        __syncthreads();
        for (int rr = 0; rr < K; ++rr)
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int v = 0; v < R; ++v) acc[u][v] += Xa[rr][ty * R + u] * Xb[rr][tx * R + v];
        __syncthreads();
    }
    double* M = st.M(l);
    for (int u = 0; u < R; ++u)
        for (int v = 0; v < R; ++v) {
            const int64_t a = a0 + ty * R + u, b = b0 + tx * R + v;
            if (a < D && b < D) M[a * D + b] += acc[u][v];
        }
}

// ---------------------------------------------------------------- FACTOR
// Header: mean eigenvalue of F = M/n_total is tr(M)/(n_total D); lambda.
template <typename TS>
__global__ void prepare_kernel(St<TS> st, int64_t n_total, double lambda_abs, double lambda_rel) {
    __shared__ double part[256];
    const int l = blockIdx.x;
    const int64_t D = st.D;
    const TS* M = st.M(l);
    double s = 0.0;
    for (int64_t a = threadIdx.x; a < D; a += blockDim.x) s += (double)M[a * D + a];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double* h = st.header(l);
        const double mean_eig = part[0] / (double)n_total / (double)D;
        h[kPcLambda] = lambda_abs + lambda_rel * mean_eig;
        h[kPcMeanEig] = mean_eig;
        h[kPcFailedPivot] = 0.0;
        h[kPcNTotal] = (double)n_total;
    }
}

// Lower triangle of M <- M / n_total + lambda I.
template <typename TS>
__global__ void scale_kernel(St<TS> st, int n_layers) {
    const int64_t D = st.D, per = D * D;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < per * n_layers;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int l = (int)(e / per);
        const int64_t r = e - (int64_t)l * per, a = r / D, b = r - a * D;
        if (b > a) continue;
        const double* h = st.header(l);
        TS* M = st.M(l);
        TS v = M[r] * (TS)(1.0 / h[kPcNTotal]);
        if (a == b) v += (TS)h[kPcLambda];
        M[r] = v;
    }
}

// One 32-column step at k0, grid (layer, row chunk): every CTA factors the
// diagonal block in shared memory (one warp), then solves x L_kk^T = a for 256
// panel rows. Row chunk 0 also writes L_kk and its inverse (into Dinv).
template <typename TS>
__global__ void __launch_bounds__(256) panel_kernel(St<TS> st, int64_t k0) {
    __shared__ TS Lk[kNB][kNB + 1];
    const int l = blockIdx.x;
    const int64_t D = st.D;
    TS* M = st.M(l);
    const int nb = (int)((D - k0) < kNB ? (D - k0) : kNB);
    const int tid = threadIdx.x, lane = tid & 31;
    for (int e = tid; e < kNB * kNB; e += blockDim.x) {
        const int i = e / kNB, j = e % kNB;
        TS v;
        if (i < nb && j < nb)
            v = (j <= i) ? M[(k0 + i) * D + k0 + j] : (TS)0;
        else
            v = (i == j) ? (TS)1 : (TS)0;  // identity padding of a ragged last block
        Lk[i][j] = v;
    }
    __syncthreads();
    if (tid < 32) {
        // Lane i holds row i of the block in registers; step j broadcasts the
        // pivot and the scaled column j with warp shuffles (right-looking).
        TS r[kNB];
#pragma unroll
        for (int c = 0; c < kNB; ++c) r[c] = Lk[lane][c];
        int bad = -1;
#pragma unroll
        for (int j = 0; j < kNB; ++j) {
            const TS p = __shfl_sync(0xffffffffu, r[j], j);
            const bool ok = p > (TS)0;
            if (!ok && bad < 0) bad = j;
            const TS piv = ok ? sqrt(p) : (TS)NAN;  // sqrtf for a float state
            if (lane == j) r[j] = piv;
            if (lane > j) r[j] /= piv;
#pragma unroll
            for (int c = j + 1; c < kNB; ++c) {
                const TS v = __shfl_sync(0xffffffffu, r[j], c);  // L[c][j]
                if (lane >= c) r[c] -= r[j] * v;
            }
        }
#pragma unroll
        for (int c = 0; c < kNB; ++c) Lk[lane][c] = (c <= lane) ? r[c] : (TS)0;
        if (blockIdx.y == 0 && lane == 0 && bad >= 0 && bad < nb) {
            double* h = st.header(l);
            if (h[kPcFailedPivot] == 0.0) h[kPcFailedPivot] = (double)(k0 + bad + 1);
        }
    }
    __syncthreads();
    // The diagonal block of M is left as it is: other CTAs of this launch read
    // it, and later steps use the block only through its inverse in Dinv.
    if (blockIdx.y == 0) {
        // inverse of the (padded) diagonal block: lane c solves L X[:, c] = e_c
        if (tid < 32) {
            TS* Di = st.Dinv(l) + (k0 / kNB) * (kNB * kNB);
            const int c = lane;
            TS x[kNB];
#pragma unroll
            for (int i = 0; i < kNB; ++i) {
                TS s = (i == c) ? (TS)1 : (TS)0;
#pragma unroll
                for (int m = 0; m < i; ++m) s -= Lk[i][m] * x[m];
                x[i] = (i < c) ? (TS)0 : s / Lk[i][i];
            }
#pragma unroll
            for (int i = 0; i < kNB; ++i) Di[i * kNB + c] = x[i];
        }
    }
    const int64_t i = k0 + nb + (int64_t)blockIdx.y * blockDim.x + tid;
    if (i >= D) return;
    TS x[kNB];
#pragma unroll
    for (int j = 0; j < kNB; ++j) x[j] = (j < nb) ? M[i * D + k0 + j] : (TS)0;
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
        TS s = x[j];
#pragma unroll
        for (int m = 0; m < j; ++m) s -= x[m] * Lk[j][m];
        x[j] = s / Lk[j][j];
    }
#pragma unroll
    for (int j = 0; j < kNB; ++j)
        if (j < nb) M[i * D + k0 + j] = x[j];
}

// Trailing update of the lower triangle: M[i][j] -= sum_m L[i][m] L[j][m] over
// the panel columns m in [k0, k0+nb), i >= j >= k0+nb. 64x64 tiles, grid z = layer.
template <typename TS>
__global__ void __launch_bounds__(256) update_kernel(St<TS> st, int64_t k0) {
    if (blockIdx.x > blockIdx.y) return;
    constexpr int T = 64;
    __shared__ TS Pi[kNB][T + 1];
    __shared__ TS Pj[kNB][T + 1];
    const int l = blockIdx.z;
    const int64_t D = st.D;
    TS* M = st.M(l);
    const int nb = (int)((D - k0) < kNB ? (D - k0) : kNB);
    const int64_t s0 = k0 + nb;
    const int64_t i0 = s0 + (int64_t)blockIdx.y * T, j0 = s0 + (int64_t)blockIdx.x * T;
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    for (int e = tid; e < kNB * T; e += 256) {
        const int r = e / kNB, m = e % kNB;
        Pi[m][r] = (i0 + r < D && m < nb) ? M[(i0 + r) * D + k0 + m] : (TS)0;
        Pj[m][r] = (j0 + r < D && m < nb) ? M[(j0 + r) * D + k0 + m] : (TS)0;
    }
    __syncthreads();
    TS acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = (TS)0;
#pragma unroll 8
    for (int m = 0; m < kNB; ++m) {
        TS a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = Pi[m][ty * 4 + u];
#pragma unroll
        for (int v = 0; v < 4; ++v) b[v] = Pj[m][tx * 4 + v];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] += a[u] * b[v];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t i = i0 + ty * 4 + u, j = j0 + tx * 4 + v;
            if (i < D && j < D && j <= i) M[i * D + j] -= acc[u][v];
        }
}

// ---------------------------------------------------------------- FACTOR (fp64)
// The same right-looking steps for an fp64 state, laid out for the fp64 pipe (two
// multiply-adds a clock and SM, so a warp-wide one holds its pipe for tens of clocks): no
// square root, division or triangular solve row by row on the serial path, work spread over
// as many CTAs as there is, and nothing done twice but the 32 x 32 diagonal block.
//
// Panel step at k0, grid (row chunk, layer), 128 threads: a CTA eliminates the diagonal block
// together with its 8 panel rows, A_ic -= (A_ij w_j) A_cj with w_j = 1 / A_jj, and scales column j
// by 1/sqrt(A_jj) at the end, all columns at once. The serial chain is one pivot after the other,
// so warp 0 does nothing else: it brings A_jj of the next column up to date and inverts it (a 20-bit
// guess and one cubic step) while warps 1-3 update the rest with the current column; one barrier a
// column. Chunk 0 leaves L_kk in the block's slot of Dinv; f64_inverse_kernel replaces it by its
// inverse after the last step. D = 256: 150 us a step in panel_kernel (one CTA: two warps of
// serial chains), 26 us here.
constexpr int kF64Rows = 8;

// 1/p on the pivots' serial chain, for p between kRcpMin and kRcpMax: the hardware's 20-bit guess of a
// double's reciprocal, and one step of Householder's third-order iteration takes it past 2^-59 before rounding.
constexpr double kRcpMin = 9.4e-302, kRcpMax = 1.07e301;
__device__ __forceinline__ double rcp_chain(double p) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
    const double e = fma(-p, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// What the updates by a pivot p multiply with: w = 1/p, or near the ends of the exponent range, where 1/p
// may overflow or lose bits, w = 1/sqrt(p) to be multiplied with twice (twice: true).
__device__ __forceinline__ double pivot_factor(double p, bool& twice) {
    twice = !(p > kRcpMin && p < kRcpMax);
    if (!twice) return rcp_chain(p);
    return p > 0.0 ? rsqrt(p) : NAN;
}

__global__ void __launch_bounds__(128) panel_f64_kernel(St<double> st, int64_t k0) {
    constexpr int R = kNB + kF64Rows;
    __shared__ double A[R][kNB + 1];
    __shared__ double inv[kNB];
    const int l = blockIdx.y;
    const int64_t D = st.D;
    double* M = st.M(l);
    const int nb = (int)((D - k0) < kNB ? (D - k0) : kNB);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t i0 = k0 + nb + (int64_t)blockIdx.x * kF64Rows;  // this CTA's panel rows
    for (int e = tid; e < R * kNB; e += 128) {
        const int i = e / kNB, j = e % kNB;
        double v;
        if (i < kNB)  // identity padding of a ragged last block
            v = (i < nb && j < nb) ? (j <= i ? M[(k0 + i) * D + k0 + j] : 0.0) : (i == j ? 1.0 : 0.0);
        else
            v = (i0 + i - kNB < D && j < nb) ? M[(i0 + i - kNB) * D + k0 + j] : 0.0;
        A[i][j] = v;
    }
    __syncthreads();
    __shared__ double wj[2];  // pivot_factor of the current and the next column
    __shared__ int wtwice[2];
    int bad = -1;             // warp 0: first non-positive pivot
    bool twice = false;
    if (warp == 0) {
        const double p = A[0][0];
        if (!(p > 0.0)) bad = 0;
        const double w = pivot_factor(p, twice);
        if (lane == 0) wj[0] = w, wtwice[0] = twice;
    }
    __syncthreads();
    for (int j = 0; j < kNB - 1; ++j) {
        const double w = wj[j & 1];
        if (warp == 0) {
            const double a = A[j + 1][j], aw = a * w, p = A[j + 1][j + 1] - (twice ? aw * aw : aw * a);
            if (!(p > 0.0) && bad < 0) bad = j + 1;
            const double wn = pivot_factor(p, twice);
            if (lane == 0) {
                A[j + 1][j + 1] = p;
                wj[(j + 1) & 1] = wn;
                wtwice[(j + 1) & 1] = twice;
            }
        } else {
            const int u = warp - 1;
            auto update = [&](auto&& col) {  // col(c): the column's entry c, times w where that is due twice
                // the diagonal block's rows below j + 1: column c of row `lane`
                if (lane > j + 1) {
                    const double t = A[lane][j] * w;
                    for (int c = j + 1 + u; c <= lane; c += 3) A[lane][c] -= t * col(c);
                }
                // the panel rows: 8 rows x the columns after j, 12 columns at a time
                const int pr = kNB + (lane & 7);
                const double tp = A[pr][j] * w;
                for (int c = j + 1 + u * 4 + (lane >> 3); c < kNB; c += 12) A[pr][c] -= tp * col(c);
            };
            if (wtwice[j & 1])
                update([&](int c) { return A[c][j] * w; });
            else
                update([&](int c) { return A[c][j]; });
        }
        __syncthreads();
    }
    if (warp == 0) {
        const double p = A[lane][lane];
        inv[lane] = p > 0.0 ? rsqrt(p) : NAN;
        if (blockIdx.x == 0 && lane == 0 && bad >= 0 && bad < nb) {
            double* h = st.header(l);
            if (h[kPcFailedPivot] == 0.0) h[kPcFailedPivot] = (double)(k0 + bad + 1);
        }
    }
    __syncthreads();
    // the diagonal block of M is left as it is: other CTAs of this launch read it
    if (blockIdx.x == 0) {
        double* Lk = st.Dinv(l) + (k0 / kNB) * (kNB * kNB);
        for (int e = tid; e < kNB * kNB; e += 128) {
            const int i = e / kNB, j = e % kNB;
            Lk[e] = j <= i ? A[i][j] * inv[j] : 0.0;
        }
    }
    for (int e = tid; e < kF64Rows * kNB; e += 128) {
        const int r = e / kNB, j = e % kNB;
        if (i0 + r < D && j < nb) M[(i0 + r) * D + k0 + j] = A[kNB + r][j] * inv[j];
    }
}

// Trailing update in 16 x 16 tiles, two entries a thread (D = 256: up to 105 tiles instead of 10).
__global__ void __launch_bounds__(128) update_f64_kernel(St<double> st, int64_t k0) {
    if (blockIdx.x > blockIdx.y) return;
    constexpr int T = 16;
    __shared__ double Pi[T][kNB + 1];
    __shared__ double Pj[T][kNB + 1];
    const int l = blockIdx.z;
    const int64_t D = st.D;
    double* M = st.M(l);
    const int64_t s0 = k0 + kNB;
    const int64_t i0 = s0 + (int64_t)blockIdx.y * T, j0 = s0 + (int64_t)blockIdx.x * T;
    const int tid = threadIdx.x;
    for (int e = tid; e < kNB * T; e += 128) {
        const int r = e / kNB, m = e % kNB;
        Pi[r][m] = i0 + r < D ? M[(i0 + r) * D + k0 + m] : 0.0;
        Pj[r][m] = j0 + r < D ? M[(j0 + r) * D + k0 + m] : 0.0;
    }
    __syncthreads();
    const int ty = tid / T, tx = tid % T;
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
    for (int m = 0; m < kNB; ++m) {
        a0 += Pi[ty][m] * Pj[tx][m];
        a1 += Pi[ty + 8][m] * Pj[tx][m];
    }
    const int64_t i = i0 + ty, j = j0 + tx;
    if (i < D && j <= i) M[i * D + j] -= a0;
    if (i + 8 < D && j <= i + 8) M[(i + 8) * D + j] -= a1;
}

// Dinv's slots from L_kk to its inverse, grid (block, layer): lane c of every warp holds column c
// of X, L X = I, eliminated column by column; the four warps take every fourth row.
__global__ void __launch_bounds__(128) f64_inverse_kernel(St<double> st) {
    __shared__ double L[kNB][kNB + 1];
    __shared__ double X[kNB][kNB + 1];
    double* Di = st.Dinv(blockIdx.y) + (int64_t)blockIdx.x * (kNB * kNB);
    const int tid = threadIdx.x, c = tid & 31, warp = tid >> 5;
    for (int e = tid; e < kNB * kNB; e += 128) {
        L[e / kNB][e % kNB] = Di[e];
        X[e / kNB][e % kNB] = e / kNB == e % kNB ? 1.0 : 0.0;
    }
    __syncthreads();
    __shared__ double inv[kNB];
    if (tid < kNB) inv[tid] = 1.0 / L[tid][tid];
    __syncthreads();
    for (int i = 0; i < kNB; ++i) {
        const double x = X[i][c] * inv[i];
        for (int m = i + 1 + warp; m < kNB; m += 4) X[m][c] -= L[m][i] * x;
        __syncthreads();
    }
    for (int e = tid; e < kNB * kNB; e += 128) {
        const int i = e / kNB, j = e % kNB;
        Di[e] = j <= i ? X[i][j] * inv[i] : 0.0;
    }
}

// ---------------------------------------------------------------- APPLY
// grid (query group, layer). G query rows per CTA; y[G][D] in shared memory.
// Forward, block b:  r = q_b - L_{b,<b} y_<b ;  y_b = Dinv_b r
// Backward, block b: r = y_b - L_{>b,b}^T x_>b ;  x_b = Dinv_b^T r
// part[0..7][g][i] added in pairs: three dependent fp64 adds instead of eight
template <typename TS, int G>
__device__ __forceinline__ TS sum8(const TS (&part)[8][G][kNB], int g, int i) {
    return ((part[0][g][i] + part[1][g][i]) + (part[2][g][i] + part[3][g][i])) +
           ((part[4][g][i] + part[5][g][i]) + (part[6][g][i] + part[7][g][i]));
}

template <typename TS, int G>
__global__ void __launch_bounds__(256)
apply_kernel(St<TS> st, const float* __restrict__ q, int64_t n_q, int64_t ld_q, TS* __restrict__ out,
             int64_t ld_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TS* y = (TS*)smem_raw;  // [G][D]
    __shared__ TS part[8][G][kNB];
    __shared__ TS r[G][kNB];
    __shared__ TS Dsm[kNB][kNB + 1];  // inverse of the current diagonal block
    const int l = blockIdx.y;
    const int64_t D = st.D;
    const TS* L = st.M(l);
    const TS* Dv = st.Dinv(l);
    const double* h = st.header(l);
    const int64_t g0 = (int64_t)blockIdx.x * G;
    const int gn = (int)((n_q - g0) < G ? (n_q - g0) : G);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (h[kPcFailedPivot] != 0.0) {
        for (int g = 0; g < gn; ++g)
            for (int64_t i = tid; i < D; i += blockDim.x) out[(g0 + g) * ld_out + (int64_t)l * D + i] = (TS)NAN;
        return;
    }
    const int64_t nblk = (D + kNB - 1) / kNB;
    // forward
    for (int64_t bi = 0; bi < nblk; ++bi) {
        const int64_t b0 = bi * kNB;
        const int nb = (int)((D - b0) < kNB ? (D - b0) : kNB);
        for (int e = tid; e < kNB * kNB; e += blockDim.x) Dsm[e / kNB][e % kNB] = Dv[bi * kNB * kNB + e];
        if constexpr (sizeof(TS) == 8) {
            // fp64: lane = row, the warps share the columns (an fp64 add per shuffle of a row sum
            // would cost more than the row), partial sums meet in shared memory
            TS acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = (TS)0;
            if (lane < nb)
#pragma unroll 8
                for (int64_t m = warp; m < b0; m += 8) {
                    const TS lv = L[(b0 + lane) * D + m];
#pragma unroll
                    for (int g = 0; g < G; ++g) acc[g] += lv * y[g * D + m];
                }
#pragma unroll
            for (int g = 0; g < G; ++g) part[warp][g][lane] = acc[g];
            __syncthreads();
            for (int e = tid; e < G * kNB; e += blockDim.x) {
                const int g = e / kNB, i = e % kNB;
                const TS t = sum8(part, g, i);
                r[g][i] = (i < nb && g < gn) ? (TS)q[(g0 + g) * ld_q + (int64_t)l * D + b0 + i] - t : (TS)0;
            }
            __syncthreads();
            // y_b = Dinv_b r: warp w takes columns 4w .. 4w + 3
#pragma unroll
            for (int g = 0; g < G; ++g) {
                TS t = (TS)0;
#pragma unroll
                for (int j = 4 * warp; j < 4 * warp + 4; ++j) t += Dsm[lane][j] * r[g][j];
                part[warp][g][lane] = t;
            }
            __syncthreads();
            for (int e = tid; e < G * kNB; e += blockDim.x) {
                const int g = e / kNB, i = e % kNB;
                const TS t = sum8(part, g, i);
                if (i < nb) y[g * D + b0 + i] = t;
            }
            __syncthreads();
            continue;
        }
        for (int ii = warp; ii < kNB; ii += 8) {
            TS acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = (TS)0;
            if (ii < nb)
#pragma unroll 8
                for (int64_t m = lane; m < b0; m += 32) {
                    const TS lv = L[(b0 + ii) * D + m];
#pragma unroll
                    for (int g = 0; g < G; ++g) acc[g] += lv * y[g * D + m];
                }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                TS s = acc[g];
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0)
                    r[g][ii] = (ii < nb && g < gn) ? (TS)q[(g0 + g) * ld_q + (int64_t)l * D + b0 + ii] - s : (TS)0;
            }
        }
        __syncthreads();
        for (int e = tid; e < G * kNB; e += blockDim.x) {
            const int g = e / kNB, i = e % kNB;
            TS s = (TS)0;
            for (int j = 0; j <= i; ++j) s += Dsm[i][j] * r[g][j];
            if (i < nb) y[g * D + b0 + i] = s;
        }
        __syncthreads();
    }
    // backward (x overwrites y)
    for (int64_t bi = nblk - 1; bi >= 0; --bi) {
        const int64_t b0 = bi * kNB;
        const int nb = (int)((D - b0) < kNB ? (D - b0) : kNB);
        const int64_t e0 = b0 + nb;
        for (int e = tid; e < kNB * kNB; e += blockDim.x) Dsm[e / kNB][e % kNB] = Dv[bi * kNB * kNB + e];
        TS acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = (TS)0;
        if (lane < nb)
#pragma unroll 8
            for (int64_t m = e0 + warp; m < D; m += 8) {
                const TS lv = L[m * D + b0 + lane];
#pragma unroll
                for (int g = 0; g < G; ++g) acc[g] += lv * y[g * D + m];
            }
#pragma unroll
        for (int g = 0; g < G; ++g) part[warp][g][lane] = acc[g];
        __syncthreads();
        for (int e = tid; e < G * kNB; e += blockDim.x) {
            const int g = e / kNB, i = e % kNB;
            TS t = (TS)0;
            if constexpr (sizeof(TS) == 8)
                t = sum8(part, g, i);
            else
                for (int w = 0; w < 8; ++w) t += part[w][g][i];
            r[g][i] = (i < nb) ? y[g * D + b0 + i] - t : (TS)0;
        }
        __syncthreads();
        if constexpr (sizeof(TS) == 8) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                TS t = (TS)0;
#pragma unroll
                for (int j = 4 * warp; j < 4 * warp + 4; ++j) t += Dsm[j][lane] * r[g][j];
                part[warp][g][lane] = t;
            }
            __syncthreads();
        }
        for (int e = tid; e < G * kNB; e += blockDim.x) {
            const int g = e / kNB, i = e % kNB;
            TS s = (TS)0;
            if constexpr (sizeof(TS) == 8)
                s = sum8(part, g, i);
            else
                for (int j = i; j < kNB; ++j) s += Dsm[j][i] * r[g][j];
            if (i < nb) y[g * D + b0 + i] = s;
        }
        __syncthreads();
    }
    for (int g = 0; g < gn; ++g)
        for (int64_t i = tid; i < D; i += blockDim.x) out[(g0 + g) * ld_out + (int64_t)l * D + i] = y[g * D + i];
}

// ---------------------------------------------------------------- FACTOR in one launch (fp32)
// The same right-looking Cholesky in 32-column steps, with one thread-block
// cluster of CS CTAs per layer instead of two launches per step: every CTA
// factors the diagonal block, the CTAs share the panel rows and the trailing
// 64 x 64 tiles, and cluster barriers separate the phases. M is read through
// L2 (ld.global.cg): other CTAs of the cluster wrote it. Each step does the
// arithmetic of prepare/scale/panel/update_kernel in the same order; the
// factored diagonal blocks are kept in M's diagonal blocks and inverted into
// Dinv after the last step, one warp per block.
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// release / acquire at cluster scope order every earlier global and shared access of
// the arriving threads before every later access of the waiting ones: the data the CTAs
// exchange through M (read back with ld.global.cg) needs no separate device-wide fence
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Cholesky of a 32 x 32 block by one warp. Lane i holds row i of the block
// in registers, shifted so that r[0] is always the column being eliminated:
// the step loop stays rolled (compact code; every array index is static).
// Column j of L goes to row j of LkT (LkT[j][i] = L[i][j], zero above the
// diagonal), 1 / L_jj to dinv[j]. Returns the first non-positive pivot's
// column or -1.
__device__ __forceinline__ int warp_cholesky32(const float (*A)[kNB + 1], float (*LkT)[2 * kNB + 1],
                                               float* dinv, int lane) {
    float r[kNB];
#pragma unroll
    for (int c = 0; c < kNB; ++c) r[c] = A[lane][c];
    int bad = -1;
#pragma unroll 1
    for (int j = 0; j < kNB; ++j) {
        const float p = __shfl_sync(0xffffffffu, r[0], j);
        const bool ok = p > 0.f;
        if (!ok && bad < 0) bad = j;
        // L_jj = p * rsqrt(p) and 1 / L_jj = rsqrt(p): one special-function op on the
        // serial path instead of a rounded square root and a division
        const float inv = ok ? rsqrtf(p) : NAN;
        const float piv = p * inv;
        if (lane == j) r[0] = piv;
        else if (lane > j) r[0] *= inv;
        LkT[j][lane] = (lane >= j) ? r[0] : 0.f;
        if (lane == 0) dinv[j] = inv;
        // A[i][j + idx] -= L[i][j] L[j + idx][j] below the diagonal
#pragma unroll
        for (int idx = 1; idx < kNB; ++idx) {
            const float v = __shfl_sync(0xffffffffu, r[0], (j + idx) & (kNB - 1));
            if (lane >= j + idx) r[idx] -= r[0] * v;
        }
#pragma unroll
        for (int idx = 0; idx < kNB - 1; ++idx) r[idx] = r[idx + 1];
        r[kNB - 1] = 0.f;
    }
    return bad;
}

// Queries solved inside the factorisation (FACTOR_APPLY): the query rows ride
// along as extra rows below M -- solved against each diagonal block and updated
// by each panel, which is the forward substitution L y = q -- and a second sweep
// from the last block to the first does the backward substitution L^T x = y.
// CTA r of the cluster keeps the query columns of the 64-wide tiles t with
// t % CS == r in shared memory for the whole call; the owner of a block's
// columns solves that block for all queries and the others read the result
// through distributed shared memory (two buffers, alternating by step).
constexpr int kQT = 64, kQP = kQT + 4;  // query column tile and its padded row
constexpr int kXS = kNB + 4;            // row stride of a solved block: 16-byte rows
// 16 bytes of CTA `rank`'s shared memory at the address of p in this CTA
__device__ __forceinline__ float4 ld_peer4(const float* p, uint32_t rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(r));
    return v;
}
// this CTA's copy of the solved block [n_q][kNB] (stride kXS) that CTA `rank` holds at Xo
__device__ __forceinline__ void copy_peer_block(float* XL, const float* Xo, int64_t n_q, uint32_t rank, int tid) {
    const int64_t n4 = n_q * (kNB / 4);
    for (int64_t e0 = tid; e0 < n4; e0 += 4 * 256) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {  // four loads in flight before the first store
            const int64_t e = e0 + u * 256;
            if (e < n4) v[u] = ld_peer4(Xo + (e / (kNB / 4)) * kXS + (e % (kNB / 4)) * 4, rank);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t e = e0 + u * 256;
            if (e < n4) *reinterpret_cast<float4*>(XL + (e / (kNB / 4)) * kXS + (e % (kNB / 4)) * 4) = v[u];
        }
    }
}
__host__ __device__ inline int64_t query_tiles_per_cta(int64_t D, int cs) {
    return ((D + kQT - 1) / kQT + cs - 1) / cs;
}
__host__ __device__ inline size_t solve_smem_bytes(int64_t D, int64_t n_q, int cs) {
    return sizeof(float) * ((size_t)query_tiles_per_cta(D, cs) * n_q * kQP + 3 * (size_t)n_q * kXS);
}
struct QArgs {
    const float* q;   // layer 0's column 0 of query row 0
    float* qhat;
    int64_t n_q, ld_q, ld_qhat;
};

template <int CS, bool SOLVE>
__global__ void __launch_bounds__(256, 1) factor_cluster_kernel(St<float> st, int64_t n_total, double lambda_abs,
                                                              double lambda_rel, QArgs qa) {
    __shared__ float Lk[kNB][kNB + 1];        // the diagonal block before factoring
    __shared__ float LkT[kNB][2 * kNB + 1];   // L transposed; columns 32..63 stay zero
    __shared__ float dinv[kNB];               // 1 / L_jj of the current block
    __shared__ double part[256];
    constexpr int T = 64;
    __shared__ __align__(16) float Pi[kNB][T + 4];  // 16-byte rows: the products read float4
    __shared__ __align__(16) float Pj[kNB][T + 4];
    const int rank = (int)cluster_ctarank();
    const int l = blockIdx.x / CS;
    const int64_t D = st.D;
    float* M = st.M(l);
    double* h = st.header(l);
    const int tid = threadIdx.x, lane = tid & 31, ty = tid / 16, tx = tid % 16;
    const int64_t n_q = SOLVE ? qa.n_q : 0;
    extern __shared__ __align__(16) float qsm[];
    const int64_t nown = SOLVE ? query_tiles_per_cta(D, CS) : 0;
    float* Qs = qsm;                                 // [nown][n_q][kQP]: owned query column tiles
    float* XB = Qs + nown * n_q * kQP;               // [2][n_q][kXS]: a solved block, for the others
    float* XL = XB + 2 * n_q * kXS;                  // [n_q][kXS]: the owner's block, copied here
    for (int e = tid; e < kNB * (2 * kNB + 1); e += blockDim.x) (&LkT[0][0])[e] = 0.f;
    // damping from the mean eigenvalue tr(M)/(n_total D), summed like prepare_kernel
    double s = 0.0;
    for (int64_t a = tid; a < D; a += blockDim.x) s += (double)__ldcg(M + a * D + a);
    part[tid] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (tid < w) part[tid] += part[tid + w];
        __syncthreads();
    }
    const double mean_eig = part[0] / (double)n_total / (double)D;
    const double lambda = lambda_abs + lambda_rel * mean_eig;
    if (rank == 0 && tid == 0) {
        h[kPcLambda] = lambda;
        h[kPcMeanEig] = mean_eig;
        h[kPcFailedPivot] = 0.0;
        h[kPcNTotal] = (double)n_total;
    }
    cluster_barrier();  // every CTA has read the diagonal before it is scaled
    {
        const float inv_n = (float)(1.0 / (double)n_total), lam = (float)lambda;
        for (int64_t i = rank; i < D; i += CS)
            for (int64_t j = tid; j <= i; j += blockDim.x) {
                float v = __ldcg(M + i * D + j) * inv_n;
                if (i == j) v += lam;
                M[i * D + j] = v;
            }
        if (SOLVE)
            for (int64_t o = 0; o < nown; ++o) {
                const int64_t c0 = (rank + o * CS) * kQT;
                for (int64_t e = tid; e < n_q * kQT; e += blockDim.x) {
                    const int64_t qi = e / kQT, c = c0 + e % kQT;
                    Qs[(o * n_q + qi) * kQP + e % kQT] = c < D ? qa.q[qi * qa.ld_q + (int64_t)l * D + c] : 0.f;
                }
            }
    }
    cluster_barrier();
    static_assert(CS >= 2, "rank 0 factors the next diagonal block while the others update");
    for (int64_t k0 = 0; k0 < D; k0 += kNB) {
        // ---- diagonal block. The first is factored in registers by warp 0 of every CTA; each
        // later one was factored by rank 0 during the previous step's trailing update (look-
        // ahead: it lies in that update's first tile), which rank 0 keeps in LkT / dinv and the
        // others read back from M's diagonal block and the block's slot of Dinv
        if (k0 == 0) {
            for (int e = tid; e < kNB * kNB; e += blockDim.x) {
                const int i = e / kNB, j = e % kNB;
                Lk[i][j] = (j <= i) ? __ldcg(M + (k0 + i) * D + k0 + j) : 0.f;
            }
            __syncthreads();
            if (tid < 32) {
                const int bad = warp_cholesky32(Lk, LkT, dinv, lane);
                if (rank == 0 && lane == 0 && bad >= 0 && h[kPcFailedPivot] == 0.0) h[kPcFailedPivot] = (double)(k0 + bad + 1);
            }
        } else if (rank != 0) {
            for (int e = tid; e < kNB * kNB; e += blockDim.x) {
                const int i = e / kNB, j = e % kNB;
                LkT[j][i] = (j <= i) ? __ldcg(M + (k0 + i) * D + k0 + j) : 0.f;
            }
            if (tid < kNB) dinv[tid] = __ldcg(st.Dinv(l) + (k0 / kNB) * (kNB * kNB) + tid);
        }
        __syncthreads();
        // ---- panel rows below the block (and the query rows): x L_kk^T = a, every CS-th row
        // to each CTA of the cluster. Column order with the same register shift: once x_j is
        // known it leaves every later entry
        for (int64_t i = k0 + kNB + (int64_t)tid * CS + rank; i < D; i += (int64_t)CS * blockDim.x) {
            float* row = M + i * D + k0;
            float x[kNB];
#pragma unroll
            for (int j = 0; j < kNB; ++j) x[j] = __ldcg(row + j);
#pragma unroll 1
            for (int j = 0; j < kNB; ++j) {
                const float xj = x[0] * dinv[j];
                row[j] = xj;
#pragma unroll
                for (int idx = 1; idx < kNB; ++idx) x[idx] -= xj * LkT[j][j + idx];
#pragma unroll
                for (int idx = 0; idx < kNB - 1; ++idx) x[idx] = x[idx + 1];
                x[kNB - 1] = 0.f;
            }
        }
        const int blk = (int)(k0 / kNB), own = (blk / 2) % CS;  // the block's columns: tile blk / 2
        if (SOLVE && rank == own) {
            // y_b = q~_b L_bb^-T for every query, the same column-order solve as a panel row
            float* Qb = Qs + ((blk / 2) / CS) * n_q * kQP + (blk % 2) * kNB;
            float* Xo = XB + (blk & 1) * n_q * kXS;
            // query rows start at thread 128: the panel rows above keep at most the first
            // ceil((D - 32) / CS) threads busy, so both chains run side by side
            for (int64_t qi = (tid + blockDim.x / 2) % blockDim.x; qi < n_q; qi += blockDim.x) {
                float* row = Qb + qi * kQP;
                float x[kNB];
#pragma unroll
                for (int j = 0; j < kNB; ++j) x[j] = row[j];
#pragma unroll 1
                for (int j = 0; j < kNB; ++j) {
                    const float xj = x[0] * dinv[j];
                    row[j] = xj;
                    Xo[qi * kXS + j] = xj;
#pragma unroll
                    for (int idx = 1; idx < kNB; ++idx) x[idx] -= xj * LkT[j][j + idx];
#pragma unroll
                    for (int idx = 0; idx < kNB - 1; ++idx) x[idx] = x[idx + 1];
                    x[kNB - 1] = 0.f;
                }
            }
        }
        cluster_barrier();
        if (SOLVE && k0 + kNB < D) {
            // q~[:, c] -= y_b L[c][k0..k0+31]^T for the owned columns c >= k0 + 32
            copy_peer_block(XL, XB + (blk & 1) * n_q * kXS, n_q, (uint32_t)own, tid);
            __syncthreads();
            for (int64_t o = 0; o < nown; ++o) {
                const int64_t c0 = (rank + o * CS) * kQT;
                if (c0 + kQT <= k0 + kNB || c0 >= D) continue;
                for (int e = tid; e < kNB * kQT; e += blockDim.x) {
                    const int cc = e / kNB, m = e % kNB;
                    const int64_t c = c0 + cc;
                    Pj[m][cc] = (c >= k0 + kNB && c < D) ? __ldcg(M + c * D + k0 + m) : 0.f;
                }
                __syncthreads();
                for (int64_t q0 = 0; q0 < n_q; q0 += kQT) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int64_t qi = q0 + ty * 4 + r;
                        if (qi >= n_q) break;
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                        for (int m = 0; m < kNB; ++m) {
                            const float xv = XL[qi * kXS + m];
                            const float4 b4 = *reinterpret_cast<const float4*>(&Pj[m][tx * 4]);
                            acc[0] += xv * b4.x, acc[1] += xv * b4.y, acc[2] += xv * b4.z, acc[3] += xv * b4.w;
                        }
                        float4* dst = reinterpret_cast<float4*>(Qs + (o * n_q + qi) * kQP + tx * 4);
                        float4 v = *dst;
                        v.x -= acc[0], v.y -= acc[1], v.z -= acc[2], v.w -= acc[3];
                        *dst = v;
                    }
                }
                __syncthreads();
            }
        }
        // the factored block goes back into M's diagonal block once every CTA has read the
        // unfactored one (no later step reads that block); the inverses of all diagonal
        // blocks are formed after the last step
        if (k0 == 0 && rank == 0)
            for (int e = tid; e < kNB * kNB; e += blockDim.x) {
                const int i = e / kNB, j = e % kNB;
                if (j <= i) M[(k0 + i) * D + k0 + j] = LkT[j][i];
            }
        // ---- trailing update of the lower triangle (and of the query rows' remaining
        // columns), 64 x 64 tiles shared by the cluster
        const int64_t s0 = k0 + kNB;
        const int64_t rest = D - s0;
        if (rest > 0) {
            const int64_t t = (rest + T - 1) / T, lower = t * (t + 1) / 2;
            const int64_t tiles = lower;
            // tile u: lower-triangle tile (bi, bj), bj <= bi, row-major; then query tiles (qb, bj)
            struct Tile {
                float* rows;  // M or the query rows
                int64_t ld, lim, i0, j0;
                bool tri;     // lower triangle of M: only j <= i
            };
            auto tile_of = [&](int64_t u) {
                Tile tl;
                {
                    // fp32 estimate (fp64 is a slow pipe here), corrected in integers
                    int64_t bi = (int64_t)((sqrtf(8.f * (float)u + 1.f) - 1.f) * 0.5f);
                    while (bi * (bi + 1) / 2 > u) --bi;
                    while ((bi + 1) * (bi + 2) / 2 <= u) ++bi;
                    tl.rows = M, tl.ld = D, tl.lim = D, tl.tri = true;
                    tl.i0 = s0 + bi * T;
                    tl.j0 = s0 + (u - bi * (bi + 1) / 2) * T;
                }
                return tl;
            };
            // software pipeline: while tile u is multiplied, the panel rows and the current
            // values of this CTA's next tile are on their way (each thread: 8 + 8 panel values,
            // row e/32, column e%32, and its 4 x 4 outputs)
            float ra[8], rb[8], mv[4][4];
            auto load_tile = [&](int64_t u) {
                const Tile tl = tile_of(u);
#pragma unroll
                for (int hh = 0; hh < 8; ++hh) {
                    const int e = tid + hh * 256, r = e / kNB, m = e % kNB;
                    ra[hh] = (tl.i0 + r < tl.lim) ? __ldcg(tl.rows + (tl.i0 + r) * tl.ld + k0 + m) : 0.f;
                    rb[hh] = (tl.j0 + r < D) ? __ldcg(M + (tl.j0 + r) * D + k0 + m) : 0.f;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int64_t i = tl.i0 + ty * 4 + q, j = tl.j0 + tx * 4 + v;
                        mv[q][v] = (i < tl.lim && j < D && (!tl.tri || j <= i)) ? __ldcg(tl.rows + i * tl.ld + j)
                                                                                 : 0.f;
                    }
            };
            // rank 0 takes tile 0 alone (it holds the next diagonal block, factored right after);
            // ranks 1 .. CS-1 share the others
            const int64_t ustep = rank == 0 ? tiles : CS - 1;
            int64_t u = rank;
            if (u < tiles) load_tile(u);
            for (; u < tiles; u += ustep) {
                const Tile tl = tile_of(u);
#pragma unroll
                for (int hh = 0; hh < 8; ++hh) {
                    const int e = tid + hh * 256, r = e / kNB, m = e % kNB;
                    Pi[m][r] = ra[hh];
                    Pj[m][r] = rb[hh];
                }
                float acc[4][4];
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) acc[a][b] = mv[a][b];
                __syncthreads();
                if (u + ustep < tiles) load_tile(u + ustep);
#pragma unroll 8
                for (int m = 0; m < kNB; ++m) {
                    const float4 a4 = *reinterpret_cast<const float4*>(&Pi[m][ty * 4]);
                    const float4 b4 = *reinterpret_cast<const float4*>(&Pj[m][tx * 4]);
                    const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int v = 0; v < 4; ++v) acc[q][v] -= a[q] * b[v];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int64_t i = tl.i0 + ty * 4 + q, j = tl.j0 + tx * 4 + v;
                        if (i < tl.lim && j < D && (!tl.tri || j <= i)) tl.rows[i * tl.ld + j] = acc[q][v];
                        // tile 0's top-left 32 x 32: the next diagonal block, updated (D - s0 >= 32)
                        if (u == 0 && ty * 4 + q < kNB && tx * 4 + v < kNB)
                            Lk[ty * 4 + q][tx * 4 + v] = (tx * 4 + v <= ty * 4 + q) ? acc[q][v] : 0.f;
                    }
                __syncthreads();
            }
            if (rank == 0) {
                // look-ahead: factor the next diagonal block now; the others read it after the barrier
                if (tid < 32) {
                    const int bad = warp_cholesky32(Lk, LkT, dinv, lane);
                    if (lane == 0 && bad >= 0 && h[kPcFailedPivot] == 0.0) h[kPcFailedPivot] = (double)(s0 + bad + 1);
                }
                __syncthreads();
                for (int e = tid; e < kNB * kNB; e += blockDim.x) {
                    const int i = e / kNB, j = e % kNB;
                    if (j <= i) M[(s0 + i) * D + s0 + j] = LkT[j][i];
                }
                if (tid < kNB) st.Dinv(l)[(s0 / kNB) * (kNB * kNB) + tid] = dinv[tid];
            }
        }
        cluster_barrier();
    }
    // inverses of the factored diagonal blocks: a CTA stages a block in shared
    // memory and lane c of warp 0 solves L X[:, c] = e_c in column order
    const int nblk = (int)(D / kNB);
    for (int b = rank; b < nblk; b += CS) {
        const float* Lb = M + (int64_t)b * kNB * D + (int64_t)b * kNB;
        for (int e = tid; e < kNB * kNB; e += blockDim.x) {
            const int i = e / kNB, j = e % kNB;
            Lk[i][j] = (j <= i) ? __ldcg(Lb + (int64_t)i * D + j) : 0.f;
        }
        __syncthreads();
        if (tid < kNB) {
            const int c = lane;
            float x[kNB];
#pragma unroll
            for (int i = 0; i < kNB; ++i) x[i] = (i == c) ? 1.f : 0.f;
#pragma unroll
            for (int j = 0; j < kNB; ++j) {
                x[j] = (j < c) ? 0.f : x[j] / Lk[j][j];
#pragma unroll
                for (int i = j + 1; i < kNB; ++i) x[i] -= Lk[i][j] * x[j];
            }
            float* Di = st.Dinv(l) + (int64_t)b * (kNB * kNB);
#pragma unroll
            for (int i = 0; i < kNB; ++i) Di[i * kNB + c] = x[i];
        }
        __syncthreads();
    }
    if constexpr (SOLVE) {
        // ---- backward substitution L^T x = y from the last block: the owner of block b forms
        // x_b = Dinv_b^T y~_b for every query; then each CTA removes x_b L[b0..b0+31][c] from
        // its owned columns c < b0
        cluster_barrier();  // Dinv complete
        const int64_t ldh = qa.ld_qhat;
        float* Qh = qa.qhat + (int64_t)l * D;
        if (__ldcg(&h[kPcFailedPivot]) != 0.0) {
            for (int64_t o = 0; o < nown; ++o) {
                const int64_t c0 = (rank + o * CS) * kQT;
                for (int64_t e = tid; e < n_q * kQT; e += blockDim.x)
                    if (c0 + e % kQT < D) Qh[(e / kQT) * ldh + c0 + e % kQT] = NAN;
            }
            return;
        }
        for (int b = nblk - 1; b >= 0; --b) {
            const int64_t b0 = (int64_t)b * kNB;
            const int own = (b / 2) % CS;
            // L[b0..b0+31][c] of this CTA's first owned tile left of the block does not depend
            // on x_b: staged while the owner solves
            const bool pre = nown > 0 && (int64_t)rank * kQT < b0;
            if (pre)
                for (int e = tid; e < kNB * kQT; e += blockDim.x) {
                    const int m = e / kQT, cc = e % kQT;
                    const int64_t c = (int64_t)rank * kQT + cc;
                    Pj[m][cc] = (c < b0) ? __ldcg(M + (b0 + m) * D + c) : 0.f;
                }
            if (rank == own) {
                const float* Di = st.Dinv(l) + (int64_t)b * (kNB * kNB);
                for (int e = tid; e < kNB * kNB; e += blockDim.x) Lk[e / kNB][e % kNB] = __ldcg(Di + e);
                __syncthreads();
                float* Qb = Qs + ((b / 2) / CS) * n_q * kQP + (b % 2) * kNB;
                float* Xo = XB + (b & 1) * n_q * kXS;
                for (int64_t e = tid; e < n_q * kNB; e += blockDim.x) {
                    const int64_t qi = e / kNB;
                    const int c = (int)(e % kNB);
                    float acc = 0.f;  // Dinv_b is lower triangular: entries above the diagonal are 0
#pragma unroll
                    for (int i = 0; i < kNB; ++i) acc += Lk[i][c] * Qb[qi * kQP + i];
                    Xo[qi * kXS + c] = acc;
                }
                __syncthreads();
                for (int64_t e = tid; e < n_q * kNB; e += blockDim.x)
                    Qb[(e / kNB) * kQP + e % kNB] = Xo[(e / kNB) * kXS + e % kNB];
            }
            cluster_barrier();
            if (b0 == 0) break;
            copy_peer_block(XL, XB + (b & 1) * n_q * kXS, n_q, (uint32_t)own, tid);
            __syncthreads();
            for (int64_t o = 0; o < nown; ++o) {
                const int64_t c0 = (rank + o * CS) * kQT;
                if (c0 >= b0) continue;
                if (o > 0) {
                    for (int e = tid; e < kNB * kQT; e += blockDim.x) {
                        const int m = e / kQT, cc = e % kQT;
                        Pj[m][cc] = (c0 + cc < b0) ? __ldcg(M + (b0 + m) * D + c0 + cc) : 0.f;
                    }
                }
                __syncthreads();
                for (int64_t q0 = 0; q0 < n_q; q0 += kQT) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const int64_t qi = q0 + ty * 4 + r;
                        if (qi >= n_q) break;
                        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
                        for (int m = 0; m < kNB; ++m) {
                            const float xv = XL[qi * kXS + m];
                            const float4 b4 = *reinterpret_cast<const float4*>(&Pj[m][tx * 4]);
                            acc[0] += xv * b4.x, acc[1] += xv * b4.y, acc[2] += xv * b4.z, acc[3] += xv * b4.w;
                        }
                        float4* dst = reinterpret_cast<float4*>(Qs + (o * n_q + qi) * kQP + tx * 4);
                        float4 v = *dst;
                        v.x -= acc[0], v.y -= acc[1], v.z -= acc[2], v.w -= acc[3];
                        *dst = v;
                    }
                }
                __syncthreads();
            }
        }
        // the owned columns now hold x: out to qhat
        for (int64_t o = 0; o < nown; ++o) {
            const int64_t c0 = (rank + o * CS) * kQT;
            for (int64_t e = tid; e < n_q * kQT; e += blockDim.x)
                if (c0 + e % kQT < D) Qh[(e / kQT) * ldh + c0 + e % kQT] = Qs[(o * n_q + e / kQT) * kQP + e % kQT];
        }
        cluster_barrier();  // peers may still read this CTA's exchange buffer
    }
}

template <int CS, bool SOLVE>
cudaError_t factor_cluster(int n_layers, int64_t D, void* state, int64_t n_total, double la, double lr,
                           const QArgs& qa, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (CS > 8)
        e = cudaFuncSetAttribute(factor_cluster_kernel<CS, SOLVE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const size_t smem = SOLVE ? solve_smem_bytes(D, qa.n_q, CS) : 0;
    if (smem > 190 * 1024) return cudaErrorNotSupported;
    if (SOLVE &&
        (e = cudaFuncSetAttribute(factor_cluster_kernel<CS, SOLVE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem)) != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_layers * CS));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int max_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&max_clusters, factor_cluster_kernel<CS, SOLVE>, &cfg) != cudaSuccess ||
        max_clusters < 1) {
        cudaGetLastError();
        return cudaErrorNotSupported;
    }
    note_launches(1);
    e = cudaLaunchKernelEx(&cfg, factor_cluster_kernel<CS, SOLVE>, state_of<float>(state, D), n_total, la, lr, qa);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <typename TS>
cudaError_t factor_impl(int n_layers, int64_t D, void* state, int64_t n_total, double la, double lr,
                        cudaStream_t s) {
    if constexpr (sizeof(TS) == 4) {
        // fp32 state, whole 32-column blocks: one launch, a cluster of 16 (else 8) CTAs per layer
        if (D % kNB == 0 && D >= 2 * kNB) {
            const QArgs none{nullptr, nullptr, 0, 0, 0};
            cudaError_t e = factor_cluster<16, false>(n_layers, D, state, n_total, la, lr, none, s);
            if (e == cudaErrorNotSupported) e = factor_cluster<8, false>(n_layers, D, state, n_total, la, lr, none, s);
            if (e != cudaErrorNotSupported) return e;
        }
    }
    St<TS> st = state_of<TS>(state, D);
    note_launches(2);
    prepare_kernel<TS><<<n_layers, 256, 0, s>>>(st, n_total, la, lr);
    int64_t blocks = (D * D * n_layers + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    scale_kernel<TS><<<(unsigned)blocks, 256, 0, s>>>(st, n_layers);
    if constexpr (sizeof(TS) == 8) {
        for (int64_t k0 = 0; k0 < D; k0 += kNB) {
            const int64_t rest = D - k0 - kNB;
            note_launches(1);
            panel_f64_kernel<<<dim3((unsigned)(rest > 0 ? (rest + kF64Rows - 1) / kF64Rows : 1), n_layers), 128, 0, s>>>(
                st, k0);
            if (rest <= 0) continue;
            // 64 x 64 tiles (a quarter of the loads per entry) once they fill the chip
            const unsigned t64 = (unsigned)((rest + 63) / 64), t16 = (unsigned)((rest + 15) / 16);
            note_launches(1);
            if ((int64_t)t64 * (t64 + 1) / 2 * n_layers >= 304)
                update_kernel<TS><<<dim3(t64, t64, n_layers), 256, 0, s>>>(st, k0);
            else
                update_f64_kernel<<<dim3(t16, t16, n_layers), 128, 0, s>>>(st, k0);
        }
        note_launches(1);
        f64_inverse_kernel<<<dim3((unsigned)((D + kNB - 1) / kNB), n_layers), 128, 0, s>>>(st);
    } else {
        for (int64_t k0 = 0; k0 < D; k0 += kNB) {
            const int64_t rest = D - k0 - kNB;
            const unsigned chunks = (unsigned)(rest > 0 ? (rest + 255) / 256 : 1);
            note_launches(1);
            panel_kernel<TS><<<dim3(n_layers, chunks), 256, 0, s>>>(st, k0);
            if (rest > 0) {
                const unsigned t = (unsigned)((rest + 63) / 64);
                note_launches(1);
                update_kernel<TS><<<dim3(t, t, n_layers), 256, 0, s>>>(st, k0);
            }
        }
    }
    return cudaGetLastError();
}

template <typename TS, int G>
cudaError_t apply_impl(int n_layers, int64_t D, const void* state, const float* q, int64_t n_q, int64_t ld_q,
                       void* qhat, int64_t ld_qhat, cudaStream_t s) {
    St<TS> st = state_of<TS>(const_cast<void*>(state), D);
    const size_t smem = (size_t)G * D * sizeof(TS);
    cudaError_t e = cudaFuncSetAttribute(apply_kernel<TS, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    note_launches(1);
    apply_kernel<TS, G><<<dim3((unsigned)((n_q + G - 1) / G), n_layers), 256, smem, s>>>(st, q, n_q, ld_q,
                                                                                     (TS*)qhat, ld_qhat);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- blocked path (fp32)
constexpr int kBB = 128;                // panel width
// FACTOR and FACTOR_APPLY of layers of whole 64-column blocks, against the one-launch cluster kernel,
// seven layers and 64 queries: D = 256 129 us here and 190 us there (one layer: 125 and 170 us),
// D = 512 316 and 448 us, D = 1024 690 and 1110 us. At D = 128 the difference is the
// launches' (77 and 110 us) and the cluster kernel's smaller inverses are as accurate, so it stays.
constexpr int64_t kBlockedMinD = 256;
// APPLY by itself: states of other sizes may come from the cluster kernel, which leaves no L^T (earlier
// versions factored them so)
bool blocked_states(int64_t D) { return D >= 2048 && D % kBB == 0; }

// ---- diagonal panels. A panel is 256 columns (64, 128 or 192 at the end of other D): the rows and
// columns [lo, lo + 256) of a layer, factored by one CTA with everything in shared memory, since
// the pivots are a serial chain and the next panel waits for them. Per 128-column half:
//   factor128   16 columns at a time: four warps, a thread per row with the 16 values in registers,
//               one barrier per pivot (the pivot column's 16 entries pass through shared memory);
//               then all 512 threads take the rank-16 update from the transposed columns;
//   invert64    the inverse W of each 64 x 64 diagonal block (32 x 32 inverses by one warp each,
//               then W10 = -W11 L10 W00), kept transposed in the block's strict upper triangle;
// the second half's rows are solved against the first (64 columns at a time with W) and its
// diagonal block takes L21 L21^T before its own factorisation. L goes to M's lower triangle, W^T
// above the diagonal inside each 64 x 64 diagonal block (solve_kernel reads it), the 32 x 32
// inverses to Dinv (APPLY's other path). D = 4096, seven layers: 85 us a 128-column block as a
// column-by-column left-looking factorisation, plus 49 us and 33 us for the second half's solve
// and update as launches of their own; 73 us the 256 columns here.
constexpr int kDiagThreads = 512;
constexpr int kLdS = kBB + 4;  // 16-byte rows, four banks apart
struct DiagSmem {
    float S[2][kBB][kLdS];  // the halves' diagonal blocks
    float S21[kBB][kLdS];
    float P[16][kLdS];      // a 16-column panel, transposed; invert64's scratch
    float inv[2][kBB];      // 1 / L_jj of both halves
    float col[2][16];       // the pivot column's entries in the panel's diagonal rows
};
static_assert(sizeof(DiagSmem) <= 232448 - 1024, "shared memory per CTA");
static_assert(sizeof(float) * 2 * 32 * 33 <= sizeof(float) * 16 * kLdS, "invert64 scratch");

__device__ __forceinline__ void bar_rows() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

__device__ __forceinline__ void factor128(DiagSmem& sm, int half, int64_t col0, double* h) {
    const int tid = threadIdx.x;
    float(*S)[kLdS] = sm.S[half];
    float* inv = sm.inv[half];
    for (int c0 = 0; c0 < kBB; c0 += 16) {
        if (tid < kBB) {
            const int r = tid;
            float a[16];
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&S[r][c0 + c]);
                a[c] = v.x, a[c + 1] = v.y, a[c + 2] = v.z, a[c + 3] = v.w;
            }
            const bool own = r >= c0 && r < c0 + 16;
            float cj[16];
            auto column = [&](int j) {  // the panel's diagonal rows of column j, to every row
                if (own) sm.col[j & 1][r - c0] = a[j];
                bar_rows();
#pragma unroll
                for (int c = 0; c < 16; c += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(&sm.col[j & 1][c]);
                    cj[c] = v.x, cj[c + 1] = v.y, cj[c + 2] = v.z, cj[c + 3] = v.w;
                }
            };
            column(0);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const float p = cj[j], iv = p > 0.f ? rsqrtf(p) : NAN;
                const float lr = a[j] * iv;  // L_rj (rows above the pivot: unused)
                float lc[16];                // L_cj
#pragma unroll
                for (int c = j + 1; c < 16; ++c) lc[c] = cj[c] * iv;
                a[j] = lr;
                if (j < 15) {  // the next pivot's column first: its way to the other rows is the chain
                    a[j + 1 < 16 ? j + 1 : 15] -= lr * lc[j < 15 ? j + 1 : 15];
                    column(j < 15 ? j + 1 : 15);
                }
#pragma unroll
                for (int c = j + 2; c < 16; ++c) a[c] -= lr * lc[c];
                if (r == c0 + j) {
                    inv[c0 + j] = iv;
                    if (!(p > 0.f) && h[kPcFailedPivot] == 0.0) h[kPcFailedPivot] = (double)(col0 + c0 + j + 1);
                }
            }
            if (r >= c0) {
#pragma unroll
                for (int c = 0; c < 16; c += 4)
                    *reinterpret_cast<float4*>(&S[r][c0 + c]) = make_float4(a[c], a[c + 1], a[c + 2], a[c + 3]);
            }
#pragma unroll
            for (int c = 0; c < 16; ++c) sm.P[c][r] = a[c];
        }
        __syncthreads();
        // rank-16 update of the 4 x 4 tiles on and below the diagonal, one tile a thread
        const int s0 = c0 + 16, nt = (kBB - s0) / 4;
        if (tid < nt * (nt + 1) / 2) {
            int ti = (int)((sqrtf(8.f * (float)tid + 1.f) - 1.f) * 0.5f);
            while (ti * (ti + 1) / 2 > tid) --ti;
            while ((ti + 1) * (ti + 2) / 2 <= tid) ++ti;
            const int i0 = s0 + 4 * ti, j0 = s0 + 4 * (tid - ti * (ti + 1) / 2);
            float acc[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 v = *reinterpret_cast<const float4*>(&S[i0 + u][j0]);
                acc[u][0] = v.x, acc[u][1] = v.y, acc[u][2] = v.z, acc[u][3] = v.w;
            }
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                const float4 x = *reinterpret_cast<const float4*>(&sm.P[m][i0]);
                const float4 y = *reinterpret_cast<const float4*>(&sm.P[m][j0]);
                const float xa[4] = {x.x, x.y, x.z, x.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] -= xa[u] * ya[v];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<float4*>(&S[i0 + u][j0]) = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
        }
        __syncthreads();
    }
}

// W^T of both 64 x 64 diagonal blocks into their strict upper triangles (W's diagonal is inv).
__device__ __forceinline__ void invert64(DiagSmem& sm, int half) {
    float(*S)[kLdS] = sm.S[half];
    const float* inv = sm.inv[half];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp < 4) {  // 32 x 32 block `warp`: lane c solves L X[:, c] = e_c, column order
        const int b0 = warp * kNB, c = lane;
        float x[kNB];
#pragma unroll
        for (int r = 0; r < kNB; ++r) x[r] = r == c ? 1.f : 0.f;
#pragma unroll
        for (int j = 0; j < kNB; ++j) {
            x[j] = j < c ? 0.f : x[j] * inv[b0 + j];
#pragma unroll
            for (int r = j + 1; r < kNB; ++r) x[r] -= S[b0 + r][b0 + j] * x[j];
        }
#pragma unroll
        for (int r = 1; r < kNB; ++r)
            if (r > c) S[b0 + c][b0 + r] = x[r];
    }
    __syncthreads();
    // W10 = -W11 (L10 W00) for the two 64-blocks: thread (block, row i, four columns)
    float(*T)[kNB][kNB + 1] = reinterpret_cast<float(*)[kNB][kNB + 1]>(&sm.P[0][0]);
    // (columns kq, kq + 8, ...: neighbouring lanes on neighbouring rows of W00, no bank conflicts)
    const int blk = tid >> 8, i = (tid >> 3) & 31, kq = tid & 7, lo = 64 * blk, hi = lo + kNB;
    float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int m = 0; m < kNB; m += 4) {  // (L10 W00)[i][k] = sum_{m >= k} L10[i][m] W00[m][k]
        const float4 l4 = *reinterpret_cast<const float4*>(&S[hi + i][lo + m]);
        const float l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int k = kq + 8 * v;
            const float4 w4 = *reinterpret_cast<const float4*>(&S[lo + k][lo + m]);
            const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
                t[v] = fmaf(l[u], m + u > k ? w[u] : (m + u == k ? inv[lo + k] : 0.f), t[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) T[blk][i][kq + 8 * v] = t[v];
    __syncthreads();
    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int m = 0; m < kNB; ++m) {  // W11[i][m], m <= i
        const float w = m < i ? S[hi + m][hi + i] : (m == i ? inv[hi + i] : 0.f);
#pragma unroll
        for (int v = 0; v < 4; ++v) o[v] = fmaf(w, T[blk][m][kq + 8 * v], o[v]);
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 4; ++v) S[lo + kq + 8 * v][hi + i] = -o[v];
    __syncthreads();
}

// Rows of S21 solved against the first block, S11: X L11^T = A, 64 columns at a time with W. A thread has four rows
// and columns ci, ci + 16, ci + 32, ci + 48 (16 lanes on 16 neighbouring rows or columns of S11).
__device__ __forceinline__ void solve_half(DiagSmem& sm) {
    const int tid = threadIdx.x, r0 = (tid >> 4) * 4, ci = tid & 15;
    for (int b = 0; b < 2; ++b) {
        const int c0 = 64 * b;
        float acc[4][4];
        auto store = [&]() {  // a row's 16 threads are half a warp: they alone read and write it
            __syncwarp();
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) sm.S21[r0 + u][c0 + ci + 16 * v] = acc[u][v];
            __syncwarp();
        };
        if (b == 1) {  // columns 64..127 less the solved columns' share
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = sm.S21[r0 + u][c0 + ci + 16 * v];
#pragma unroll 2
            for (int k = 0; k < 64; k += 4) {
                float4 x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    x[u] = *reinterpret_cast<const float4*>(&sm.S21[r0 + u][k]);
                    y[u] = *reinterpret_cast<const float4*>(&sm.S[0][c0 + ci + 16 * u][k]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        acc[u][v] -= x[u].x * y[v].x + x[u].y * y[v].y + x[u].z * y[v].z + x[u].w * y[v].w;
            }
            store();
        }
        float iv[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) iv[v] = sm.inv[0][c0 + ci + 16 * v];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
        // out[r][i] = sum_{k <= i} x[r][k] W[i][k], W[i][k] = S[0][c0 + k][c0 + i] for k < i
#pragma unroll
        for (int k = 0; k < 64; k += 4) {
            float x[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 q = *reinterpret_cast<const float4*>(&sm.S21[r0 + u][c0 + k]);
                x[u][0] = q.x, x[u][1] = q.y, x[u][2] = q.z, x[u][3] = q.w;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                if (k >= 16 * v + 16) continue;  // W is lower triangular
                const int i = ci + 16 * v;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float s = sm.S[0][c0 + k + t][c0 + i];
                    const float w = k + t < i ? s : (k + t == i ? iv[v] : 0.f);
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc[u][v] = fmaf(x[u][t], w, acc[u][v]);
                }
            }
        }
        store();
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kDiagThreads) diag_panel_kernel(St<float> st, int64_t lo) {
    extern __shared__ __align__(16) unsigned char dsm[];
    DiagSmem& sm = *reinterpret_cast<DiagSmem*>(dsm);
    const int l = blockIdx.x;
    const int64_t D = st.D;
    float* M = st.M(l);
    double* h = st.header(l);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = D - lo < 2 * kBB ? (int)(D - lo) : 2 * kBB;  // the panel's rows, a multiple of 64
    const bool two = n > kBB;
    if (tid == 0) h[kPcW64] = 64.0;  // solve_kernel: the 64 x 64 inverses are there
    // a warp per row, 16 bytes a lane, nothing above the diagonal (one SM draws 17 bytes a clock)
#pragma unroll 4
    for (int r = warp; r < kBB; r += kDiagThreads / 32) {
        const int c = 4 * lane;
        auto diagonal = [&](int half) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const int row = half * kBB + r;
            if (c <= r && row < n) v = *reinterpret_cast<const float4*>(M + (lo + row) * D + lo + half * kBB + c);
            v = make_float4(v.x, c + 1 <= r ? v.y : 0.f, c + 2 <= r ? v.z : 0.f, c + 3 <= r ? v.w : 0.f);
            if (row >= n) {  // past the last block: identity
                v.x = c == r ? 1.f : 0.f, v.y = c + 1 == r ? 1.f : 0.f;
                v.z = c + 2 == r ? 1.f : 0.f, v.w = c + 3 == r ? 1.f : 0.f;
            }
            *reinterpret_cast<float4*>(&sm.S[half][r][c]) = v;
        };
        diagonal(0);
        if (two) {
            *reinterpret_cast<float4*>(&sm.S21[r][c]) =
                kBB + r < n ? *reinterpret_cast<const float4*>(M + (lo + kBB + r) * D + lo + c)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
            diagonal(1);
        }
    }
    __syncthreads();
    // a loop and not two copies: every launch starts with a cold instruction cache
#pragma unroll 1
    for (int half = 0; half < (two ? 2 : 1); ++half) {
        factor128(sm, half, lo + half * kBB, h);
        invert64(sm, half);
        if (half == 1 || !two) break;
        solve_half(sm);
        // S22 -= L21 L21^T on and below the diagonal: tiles of 8 rows by 4 columns, the
        // columns 2 (ti + 1) apart so that neighbouring lanes read neighbouring rows of S21 (no bank conflicts)
        for (int u = tid; u < 16 * 17; u += kDiagThreads) {
            // tile row ti has 2 (ti + 1) tiles
            int ti = (int)((sqrtf(4.f * (float)u + 1.f) - 1.f) * 0.5f);
            while (ti * (ti + 1) > u) --ti;
            while ((ti + 1) * (ti + 2) <= u) ++ti;
            const int i0 = 8 * ti, j0 = u - ti * (ti + 1), js = 2 * (ti + 1);  // columns j0 + js v
            float acc[8][4];
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[a][v] = sm.S[1][i0 + a][j0 + js * v];
#pragma unroll 2
            for (int k = 0; k < kBB; k += 4) {
                float4 y[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) y[v] = *reinterpret_cast<const float4*>(&sm.S21[j0 + js * v][k]);
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const float4 x = *reinterpret_cast<const float4*>(&sm.S21[i0 + a][k]);
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        acc[a][v] -= x.x * y[v].x + x.y * y[v].y + x.z * y[v].z + x.w * y[v].w;
                }
            }
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int v = 0; v < 4; ++v) sm.S[1][i0 + a][j0 + js * v] = acc[a][v];
        }
        __syncthreads();
    }
    // L on and below the diagonal, W^T above it inside the 64 x 64 diagonal blocks (the rest of a
    // half's upper triangle is the other 64-block's, written by upper_from_lower_kernel)
    for (int r = warp; r < kBB; r += kDiagThreads / 32) {
        const int c = 4 * lane;
        for (int half = 0; half < (two ? 2 : 1); ++half) {
            const float* src = &sm.S[half][r][c];
            float* dst = M + (lo + half * kBB + r) * D + lo + half * kBB + c;
            if (c / 64 <= r / 64 && half * kBB + r < n)
                *reinterpret_cast<float4*>(dst) = *reinterpret_cast<const float4*>(src);
        }
        if (kBB + r < n)
            *reinterpret_cast<float4*>(M + (lo + kBB + r) * D + lo + c) = *reinterpret_cast<const float4*>(&sm.S21[r][c]);
    }
    float* Dg = st.Dinv(l) + (lo / kNB) * (kNB * kNB);
    for (int e = tid; e < n / kNB * kNB * kNB; e += kDiagThreads) {
        const int b = e >> 10, r = (e >> 5) & 31, c = e & 31, half = b >> 2, o = (b & 3) * kNB;
        const float(*S)[kLdS] = sm.S[half];
        Dg[e] = c < r ? S[o + c][o + r] : (c == r ? sm.inv[half][o + r] : 0.f);
    }
}

// Row vectors solved against the panel's diagonal block B = [lo, lo + nb) of layer l (grid y),
// nb = 64 to 256: FWD x <- L_BB^{-1} x, else x <- L_BB^{-T} x, for rows of nb values at column lo of
// two sets of rows (the first blocks_a CTAs of a layer have rows_a). Used for the rows of M below a
// panel (FWD) and for the query rows of APPLY (both directions).
// R rows a CTA, their nb values in shared memory; 64 columns at a time: the solved columns' share
// is taken off with L, then the 64 x 64 inverse applied, both from one slab S[k][i] of
// coefficients (k: solved or own column, i: column of the block). A thread has RT x 4 entries, so
// a slab value read from shared memory serves RT products. R = 128 for many rows, 16 where few
// rows would leave SMs idle. Seven layers, 256 columns: 3840 rows each 131 us as two 128-column
// solves (a warp per row) and a product between them, 91 us here; 256 rows each 26 us.
template <int R>
struct SolveCfg {
    static constexpr int NT = R >= 96 ? 512 : 256;          // threads (R = 96: 99 us with 256, 91 with 512)
    static constexpr int RT = R / (NT / 16);                // NT / 16 row groups x 16 column groups
    static constexpr int kLdX = 2 * kBB + 4;
    static constexpr size_t kSmem = sizeof(float) * ((size_t)R * kLdX + (size_t)2 * kBB * 64 + kNB * (kNB + 1));
};
struct SolveRows {
    char* base;          // layer l's rows at byte l * layer_bytes
    size_t layer_bytes;
    int64_t ldx, n_rows;
};
template <int R, bool FWD>
__global__ void __launch_bounds__(SolveCfg<R>::NT) solve_kernel(St<float> st, int64_t lo, int nb, SolveRows rows_a, SolveRows rows_b,
                                                    int blocks_a) {
    using C = SolveCfg<R>;
    constexpr int RT = C::RT, NT = C::NT, kPl = 12 * 256 / NT, kPw = 4 * 256 / NT;
    extern __shared__ __align__(16) float ssm[];
    float(*xs)[C::kLdX] = reinterpret_cast<float(*)[C::kLdX]>(ssm);
    float(*S)[64] = reinterpret_cast<float(*)[64]>(ssm + R * C::kLdX);  // [k][i ^ 4 (k & 7)]
    float(*T)[kNB + 1] = reinterpret_cast<float(*)[kNB + 1]>(ssm + R * C::kLdX + 2 * kBB * 64);
    const int l = blockIdx.y;
    const int64_t D = st.D;
    const float* M = st.M(l) + lo * D + lo;
    const bool w64 = st.header(l)[kPcW64] == 64.0;
    const int tid = threadIdx.x, rg = tid >> 4, i0 = (tid & 15) * 4;
    const bool second = (int)blockIdx.x >= blocks_a;
    const SolveRows w = second ? rows_b : rows_a;
    const int64_t row0 = (int64_t)(second ? blockIdx.x - blocks_a : blockIdx.x) * R, n_rows = w.n_rows, ldx = w.ldx;
    float* X = (float*)(w.base + (size_t)l * w.layer_bytes) + lo;
    // n 16-byte loads, eight of a thread's in flight together: ld(e) loads item e, st(e, value) stores it
    auto copy = [&](int n, auto&& ld, auto&& st) {
        for (int e0 = tid; e0 < n; e0 += 8 * NT) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (e0 + NT * u < n) v[u] = ld(e0 + NT * u);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (e0 + NT * u < n) st(e0 + NT * u, v[u]);
        }
    };
    const int q4 = nb / 4;
    copy(R * q4,
         [&](int e) {
             const int r = e / q4, c = e % q4 * 4;
             return row0 + r < n_rows ? *reinterpret_cast<const float4*>(X + (row0 + r) * ldx + c)
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
         },
         [&](int e, const float4& v) { *reinterpret_cast<float4*>(&xs[e / q4][e % q4 * 4]) = v; });
    // Block b's coefficients: the solved columns' (4 nblk x 64 items of 16 bytes at most) and W's, one to
    // four of the thread's items each. They are loaded into registers beside the previous block's
    // products and stored behind them.
    const int nblk = nb / 64;
    float4 pl[kPl], pw[kPw];
    auto block = [&](int s, int& c0, int& k0, int& nk) {  // its columns and the solved ones
        const int b = FWD ? s : nblk - 1 - s;
        c0 = 64 * b;
        k0 = FWD ? 0 : c0 + 64;
        nk = FWD ? c0 : nb - c0 - 64;
    };
    auto load = [&](int s) {
        int c0, k0, nk;
        block(s, c0, k0, nk);
#pragma unroll
        for (int u = 0; u < kPl; ++u) {
            const int e = tid + NT * u;
            if (NT / 16 * u < nk)  // FWD: L[c0 + e % 64][e / 64 * 4 ..]; else L[k0 + e / 16][c0 + e % 16 * 4 ..]
                pl[u] = *reinterpret_cast<const float4*>(FWD ? M + (int64_t)(c0 + e % 64) * D + e / 64 * 4
                                                             : M + (int64_t)(k0 + e / 16) * D + c0 + e % 16 * 4);
        }
        if (w64)
#pragma unroll
            for (int u = 0; u < kPw; ++u) {
                const int e = tid + NT * u;
                pw[u] = *reinterpret_cast<const float4*>(M + (int64_t)(c0 + e / 16) * D + c0 + e % 16 * 4);
            }
    };
    load(0);
    for (int s = 0; s < nblk; ++s) {
        int c0, k0, nk;
        block(s, c0, k0, nk);
        __syncthreads();  // the previous block's slab is read
        // slab rows 0 .. nk-1: L between the block's columns and the solved ones; rows nk .. nk+63: W
#pragma unroll
        for (int u = 0; u < kPl; ++u) {
            const int e = tid + NT * u;
            if (NT / 16 * u >= nk) continue;
            const float4 v = pl[u];
            if (FWD) {  // S[k][i] = L[c0 + i][k], a warp's lanes along i: every store hits 32 banks
                const int i = e % 64, k = e / 64 * 4;
                S[k][i ^ ((k & 7) << 2)] = v.x;
                S[k + 1][i ^ (((k + 1) & 7) << 2)] = v.y;
                S[k + 2][i ^ (((k + 2) & 7) << 2)] = v.z;
                S[k + 3][i ^ (((k + 3) & 7) << 2)] = v.w;
            } else {    // S[k][i] = L[k0 + k][c0 + i]
                const int k = e / 16;
                *reinterpret_cast<float4*>(&S[k][(e % 16 * 4) ^ ((k & 7) << 2)]) = v;
            }
        }
        if (w64) {
            // the block as stored: L left of the diagonal, W^T right of it. FWD: S[k][i] = W[i][k] =
            // stored[k][i] for k < i; else S[k][i] = W[k][i] = stored[i][k] for k > i
#pragma unroll
            for (int u = 0; u < kPw; ++u) {
                const int e = tid + NT * u, a = e / 16, c = e % 16 * 4;
                const float v[4] = {pw[u].x, pw[u].y, pw[u].z, pw[u].w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int i = FWD ? c + t : a, k = FWD ? a : c + t, kr = nk + k;
                    S[kr][i ^ ((kr & 7) << 2)] = (FWD ? k < i : k > i) ? v[t] : (k == i ? 1.f / v[t] : 0.f);
                }
            }
        } else {
            // a state factored before these inverses were kept: from the 32 x 32 ones,
            // W = [W00 0; -W11 (L10 W00) W11]
            const float *D0 = st.Dinv(l) + (lo + c0) / kNB * (kNB * kNB), *D1 = D0 + kNB * kNB;
            for (int e = tid; e < kNB * kNB; e += NT) {
                const int i = e / kNB, k = e % kNB;
                float t = 0.f;
                for (int m = k; m < kNB; ++m) t = fmaf(M[(int64_t)(c0 + kNB + i) * D + c0 + m], D0[m * kNB + k], t);
                T[i][k] = t;
            }
            __syncthreads();
            for (int e = tid; e < 64 * 64; e += NT) {
                const int r = e / 64, c = e % 64;
                float w = 0.f;
                if (c <= r && r < kNB)
                    w = D0[r * kNB + c];
                else if (c <= r && c >= kNB)
                    w = D1[(r - kNB) * kNB + c - kNB];
                else if (c <= r)
                    for (int m = 0; m <= r - kNB; ++m) w = fmaf(-D1[(r - kNB) * kNB + m], T[m][c], w);
                const int i = FWD ? r : c, kr = nk + (FWD ? c : r);
                S[kr][i ^ ((kr & 7) << 2)] = w;
            }
        }
        __syncthreads();
        if (s + 1 < nblk) load(s + 1);
        float acc[RT][4];  // the solved columns' share less x, so that both products add
#pragma unroll
        for (int u = 0; u < RT; ++u) {
            const float4 v = *reinterpret_cast<const float4*>(&xs[rg * RT + u][c0 + i0]);
            acc[u][0] = -v.x, acc[u][1] = -v.y, acc[u][2] = -v.z, acc[u][3] = -v.w;
        }
        auto products = [&](int ks, int xc, int n) {  // acc += x[:, xc + k] S[ks + k][:]
#pragma unroll 2
            for (int k = 0; k < n; k += 4) {
                float w[4][4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float4 v = *reinterpret_cast<const float4*>(&S[ks + k + t][i0 ^ (((ks + k + t) & 7) << 2)]);
                    w[t][0] = v.x, w[t][1] = v.y, w[t][2] = v.z, w[t][3] = v.w;
                }
#pragma unroll
                for (int u = 0; u < RT; ++u) {
                    const float4 x = *reinterpret_cast<const float4*>(&xs[rg * RT + u][xc + k]);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        acc[u][v] = fmaf(x.x, w[0][v], acc[u][v]);
                        acc[u][v] = fmaf(x.y, w[1][v], acc[u][v]);
                        acc[u][v] = fmaf(x.z, w[2][v], acc[u][v]);
                        acc[u][v] = fmaf(x.w, w[3][v], acc[u][v]);
                    }
                }
            }
        };
        auto store = [&](float sign) {  // a row group's 16 threads are half a warp: they alone read its rows
            __syncwarp();
#pragma unroll
            for (int u = 0; u < RT; ++u)
                *reinterpret_cast<float4*>(&xs[rg * RT + u][c0 + i0]) =
                    make_float4(sign * acc[u][0], sign * acc[u][1], sign * acc[u][2], sign * acc[u][3]);
            __syncwarp();
        };
        if (nk > 0) {
            products(0, k0, nk);
            store(-1.f);
        }
#pragma unroll
        for (int u = 0; u < RT; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
        products(nk, c0, 64);
        store(1.f);
    }
    __syncthreads();
    for (int e = tid; e < R * q4; e += NT) {
        const int r = e / q4, c = e % q4 * 4;
        if (row0 + r < n_rows)
            *reinterpret_cast<float4*>(X + (row0 + r) * ldx + c) = *reinterpret_cast<const float4*>(&xs[r][c]);
    }
}

// Lower triangle of M <- M / n_total + lambda I for the blocked path: a warp per row, 16 bytes a lane
// (which scales up to three entries right of the diagonal too: they are overwritten later).
// grid (row groups, layer).
__global__ void __launch_bounds__(256) scale_lower_kernel(St<float> st) {
    const int l = blockIdx.y, lane = threadIdx.x & 31;
    const int64_t D = st.D;
    const double* h = st.header(l);
    const float inv_n = (float)(1.0 / h[kPcNTotal]), lam = (float)h[kPcLambda];
    float* M = st.M(l);
    for (int64_t a = blockIdx.x * 8 + (threadIdx.x >> 5); a < D; a += gridDim.x * 8) {
        float* row = M + a * D;
        for (int64_t b0 = 4 * lane; b0 <= a; b0 += 4 * 128) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (b0 + 128 * u <= a) v[u] = *reinterpret_cast<const float4*>(row + b0 + 128 * u);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t b = b0 + 128 * u;
                if (b > a) break;
                float4 w = make_float4(v[u].x * inv_n, v[u].y * inv_n, v[u].z * inv_n, v[u].w * inv_n);
                if (b == a) w.x += lam;
                if (b + 1 == a) w.y += lam;
                if (b + 2 == a) w.z += lam;
                if (b + 3 == a) w.w += lam;
                *reinterpret_cast<float4*>(row + b) = w;
            }
        }
    }
}

// M[i][j] = M[j][i] for every 64 x 64 block strictly above the diagonal blocks (U = L^T, read by
// the backward solve's tensor-core products; the diagonal blocks hold W^T there). Each thread has
// four 16-byte loads in flight and the block index comes from an fp32 estimate corrected in
// integers: with 32 x 32 blocks, scalar loads and an fp64 square root per block this took 417 us
// for seven layers of D = 4096, 73 us here.
__global__ void __launch_bounds__(256) upper_from_lower_kernel(St<float> st, int n_layers) {
    __shared__ float t[64][65];
    const int64_t D = st.D, nb = D / 64, pairs = nb * (nb - 1) / 2;
    const int r = threadIdx.x >> 4, c = (threadIdx.x & 15) * 4;
    for (int64_t w = blockIdx.x; w < pairs * n_layers; w += gridDim.x) {
        const int l = (int)(w / pairs);
        const int64_t p = w - (int64_t)l * pairs;
        int64_t bj = (int64_t)((1.f + sqrtf(1.f + 8.f * (float)p)) * 0.5f);  // p = bj(bj-1)/2 + bi, bi < bj
        while (bj * (bj - 1) / 2 > p) --bj;
        while ((bj + 1) * bj / 2 <= p) ++bj;
        const int64_t bi = p - bj * (bj - 1) / 2;
        float* M = st.M(l);
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            v[u] = *reinterpret_cast<const float4*>(M + (bj * 64 + r + 16 * u) * D + bi * 64 + c);
        __syncthreads();  // the previous block is read
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float* d = &t[r + 16 * u][c];
            d[0] = v[u].x, d[1] = v[u].y, d[2] = v[u].z, d[3] = v[u].w;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = r + 16 * u;
            *reinterpret_cast<float4*>(M + (bi * 64 + i) * D + bj * 64 + c) =
                make_float4(t[c][i], t[c + 1][i], t[c + 2][i], t[c + 3][i]);
        }
    }
}

// Query rows of a layer whose factorisation failed become NaN.
__global__ void nan_failed_kernel(St<float> st, float* qhat, int64_t ld, int64_t n_q) {
    const int l = blockIdx.y;
    if (st.header(l)[kPcFailedPivot] == 0.0) return;
    const int64_t D = st.D;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_q * D; e += (int64_t)gridDim.x * blockDim.x)
        qhat[(e / D) * ld + (int64_t)l * D + e % D] = NAN;
}

// (layers are a grid's y coordinate: the entry point takes 65535 at most)
bool blocked_pc(int64_t D, tda_dtype sdt) {
    return sdt == TDA_F32 && D % 64 == 0 && D >= kBlockedMinD && D < (1LL << 31) / kBB && gemm_tc_available();
}

template <int R, bool FWD>
cudaError_t launch_solve_r(St<float> st, int n_layers, int64_t lo, int nb, const SolveRows& a, const SolveRows& b,
                           cudaStream_t s) {
    cudaError_t e = smem_attr_once<solve_kernel<R, FWD>>((int)SolveCfg<R>::kSmem);
    if (e != cudaSuccess) return e;
    const int64_t na = (a.n_rows + R - 1) / R, nb_b = (b.n_rows + R - 1) / R;
    if (na + nb_b == 0) return cudaSuccess;
    note_launches(1);
    solve_kernel<R, FWD><<<dim3((unsigned)(na + nb_b), n_layers), SolveCfg<R>::NT, SolveCfg<R>::kSmem, s>>>(st, lo, nb, a, b, (int)na);
    return cudaGetLastError();
}

// Rows a CTA: the fewest microseconds over the rounds of 152 CTAs (measured, 256 columns: 26 us for the
// slabs and the chain, 0.26 us a row).
template <bool FWD>
cudaError_t launch_solve(St<float> st, int n_layers, int64_t lo, int nb, const SolveRows& a, const SolveRows& b,
                         cudaStream_t s) {
    int best = 0;
    double least = 0.0;
    for (int r : {128, 96, 64, 32, 16}) {
        const int64_t ctas = ((a.n_rows + r - 1) / r + (b.n_rows + r - 1) / r) * n_layers;
        const double us = (double)((ctas + 151) / 152) * (26.0 + 0.26 * r);
        if (!best || us < least) best = r, least = us;
    }
    switch (best) {
        case 128: return launch_solve_r<128, FWD>(st, n_layers, lo, nb, a, b, s);
        case 96: return launch_solve_r<96, FWD>(st, n_layers, lo, nb, a, b, s);
        case 64: return launch_solve_r<64, FWD>(st, n_layers, lo, nb, a, b, s);
        case 32: return launch_solve_r<32, FWD>(st, n_layers, lo, nb, a, b, s);
        default: return launch_solve_r<16, FWD>(st, n_layers, lo, nb, a, b, s);
    }
}

// Factorisation in panels of 256 columns: the diagonal block, the rows below it, then the trailing
// lower triangle of all layers in one launch, M -= P P^T, P = L[hi:D, lo:hi]. With queries (qhat,
// n_q > 0) their rows ride along: x L^T = q is one more set of rows below each panel, so that the
// forward substitution needs no launches of its own (seven layers of D = 4096, 256 queries: 1.0 ms
// as 32 launches).
cudaError_t factor_blocked(int n_layers, int64_t D, void* state, int64_t n_total, double la, double lr, float* qhat,
                           int64_t n_q, int64_t ld_qhat, cudaStream_t s) {
    cudaError_t e = smem_attr_once<diag_panel_kernel>((int)sizeof(DiagSmem));
    if (e != cudaSuccess) return e;
    unsigned int* err = device_error_word();
    if (!err) return cudaErrorUnknown;
    St<float> st = state_of<float>(state, D);
    note_launches(2);
    prepare_kernel<float><<<n_layers, 256, 0, s>>>(st, n_total, la, lr);
    const int64_t per = (D + 7) / 8, most = 152 * 8 / n_layers > 1 ? 152 * 8 / n_layers : 1;
    scale_lower_kernel<<<dim3((unsigned)(per < most ? per : most), n_layers), 256, 0, s>>>(st);
    float* M0 = (float*)((char*)state + 64);  // layer l's M is st.bytes further on
    const int64_t cz = (int64_t)(st.bytes / 4);
    const size_t lb = (size_t)D * 4;
    for (int64_t lo = 0; lo < D; lo += 2 * kBB) {
        note_launches(1);
        diag_panel_kernel<<<n_layers, kDiagThreads, sizeof(DiagSmem), s>>>(st, lo);
        const int64_t hi = lo + 2 * kBB < D ? lo + 2 * kBB : D, rest = D - hi;
        e = launch_solve<true>(st, n_layers, lo, (int)(hi - lo), SolveRows{(char*)M0 + (size_t)hi * D * 4, st.bytes, D, rest},
                               SolveRows{(char*)qhat, lb, ld_qhat, n_q}, s);
        if (e != cudaSuccess) return e;
        if (rest <= 0) break;
        const float* P = M0 + hi * D + lo;
        const GemmSecond q2{qhat + lo, n_q, ld_qhat, lb, qhat + hi, ld_qhat, D};
        e = launch_gemm_nt_tc_batched(P, rest, D, st.bytes, P, rest, D, st.bytes, 2 * kBB, M0 + hi * D + hi, D, cz,
                                      n_layers, -1.f, 1.f, true, err, s, n_q > 0 ? &q2 : nullptr);
        if (e != cudaSuccess) return e;
    }
    const int64_t nb = D / 64;
    int64_t g = nb * (nb - 1) / 2 * n_layers;
    if (g > 152 * 8) g = 152 * 8;
    note_launches(1);
    upper_from_lower_kernel<<<(unsigned)g, 256, 0, s>>>(st, n_layers);
    return cudaGetLastError();
}

// (D >= kBlockedMinD suffices where the state is factored in the same call)
bool apply_blocked_ok(int64_t D, tda_dtype sdt, int64_t ld_q, const void* qhat, int64_t ld_qhat,
                      int64_t n_q) {
    // 2-D copies: row strides below 2^31 bytes
    return blocked_pc(D, sdt) && ((uintptr_t)qhat & 15) == 0 && (ld_qhat & 3) == 0 && n_q < (1LL << 24) &&
           ld_q < (1LL << 29) && ld_qhat < (1LL << 29);
}

cudaError_t copy_queries(int n_layers, int64_t D, const float* q, int64_t n_q, int64_t ld_q, float* qhat,
                         int64_t ld_qhat, cudaStream_t s) {
    if (q == qhat && ld_q == ld_qhat) return cudaSuccess;
    return cudaMemcpy2DAsync(qhat, (size_t)ld_qhat * 4, q, (size_t)ld_q * 4, (size_t)n_layers * D * 4, (size_t)n_q,
                             cudaMemcpyDeviceToDevice, s);
}

// Both substitutions of the rows of qhat in place, or (forward = false) the backward one alone.
cudaError_t apply_blocked(int n_layers, int64_t D, const void* state, int64_t n_q, float* qhat, int64_t ld_qhat,
                          bool forward, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    unsigned int* err = device_error_word();
    if (!err) return cudaErrorUnknown;
    St<float> st = state_of<float>(const_cast<void*>(state), D);
    const size_t lb = (size_t)D * 4;  // layer l's columns start l * D floats into each row
    const float* M0 = (const float*)((const char*)state + 64);  // layer l's M is st.bytes further on
    constexpr int64_t kPanel = 2 * kBB;
    const SolveRows rows{(char*)qhat, lb, ld_qhat, n_q}, none{};
    for (int64_t lo = 0; forward && lo < D; lo += kPanel) {
        const int64_t hi = lo + kPanel < D ? lo + kPanel : D;
        e = launch_solve<true>(st, n_layers, lo, (int)(hi - lo), rows, none, s);
        if (e != cudaSuccess) return e;
        if (hi == D) break;
        e = launch_gemm_nt_tc_batched(M0 + hi * D + lo, D - hi, D, st.bytes, qhat + lo, n_q, ld_qhat, lb, kPanel,
                                      qhat + hi, ld_qhat, D, n_layers, -1.f, 1.f, false, err, s);
        if (e != cudaSuccess) return e;
    }
    for (int64_t lo = (D - 1) / kPanel * kPanel; lo >= 0; lo -= kPanel) {
        const int64_t hi = lo + kPanel < D ? lo + kPanel : D;
        e = launch_solve<false>(st, n_layers, lo, (int)(hi - lo), rows, none, s);
        if (e != cudaSuccess) return e;
        if (lo == 0) break;
        // rows [0, lo) of U = L^T, columns [lo, hi): U[i][j] = L[j][i]
        e = launch_gemm_nt_tc_batched(M0 + lo, lo, D, st.bytes, qhat + lo, n_q, ld_qhat, lb, hi - lo, qhat, ld_qhat, D,
                                      n_layers, -1.f, 1.f, false, err, s);
        if (e != cudaSuccess) return e;
    }
    note_launches(1);
    nan_failed_kernel<<<dim3(64, n_layers), 256, 0, s>>>(st, qhat, ld_qhat, n_q);
    return cudaGetLastError();
}

}  // namespace

int64_t precondition_apply_max_d(tda_dtype sdt) {
    // one query row of D elements must fit the shared-memory budget of APPLY
    return (int64_t)(160 * 1024) / (sdt == TDA_F64 ? 8 : 4);
}

cudaError_t launch_pc_fit(int n_layers, int64_t D, tda_dtype sdt, void* state, const float* phi, int64_t n,
                          int64_t ld, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (sdt == TDA_F32 && fit_tc_supported(n_layers, D, phi, n, ld)) {
        unsigned int* err = device_error_word();
        if (err)
            return launch_fit_tc(n_layers, D, state, tda_precondition_state_bytes(D, TDA_F32), phi, n, ld, err, s);
    }
    note_launches(1);
    if (sdt == TDA_F64) {
        const unsigned t = (unsigned)((D + 63) / 64), t16 = (unsigned)((D + 15) / 16);
        if ((int64_t)t * (t + 1) / 2 * n_layers >= 304)
            fit_f64_kernel<64><<<dim3(t, t, n_layers), 256, 0, s>>>(state_of<double>(state, D), phi, n, ld);
        else
            fit_f64_kernel<16><<<dim3(t16, t16, n_layers), 256, 0, s>>>(state_of<double>(state, D), phi, n, ld);
    } else {
        const unsigned t = (unsigned)((D + kFT - 1) / kFT);
        fit_f32_kernel<<<dim3(t, t, n_layers), 256, 0, s>>>(state_of<float>(state, D), phi, n, ld);
    }
    return cudaGetLastError();
}

cudaError_t launch_pc_factor(int n_layers, int64_t D, tda_dtype sdt, void* state, int64_t n_total,
                             double lambda_abs, double lambda_rel, cudaStream_t s) {
    if (blocked_pc(D, sdt))
        return factor_blocked(n_layers, D, state, n_total, lambda_abs, lambda_rel, nullptr, 0, 0, s);
    if (sdt == TDA_F64) return factor_impl<double>(n_layers, D, state, n_total, lambda_abs, lambda_rel, s);
    return factor_impl<float>(n_layers, D, state, n_total, lambda_abs, lambda_rel, s);
}

cudaError_t launch_pc_factor_apply(int n_layers, int64_t D, tda_dtype sdt, void* state, int64_t n_total,
                                   double lambda_abs, double lambda_rel, const float* q, int64_t n_q, int64_t ld_q,
                                   void* qhat, int64_t ld_qhat, cudaStream_t s) {
    cudaError_t e;
    if (n_q >= 1 && apply_blocked_ok(D, sdt, ld_q, qhat, ld_qhat, n_q)) {
        if ((e = copy_queries(n_layers, D, q, n_q, ld_q, (float*)qhat, ld_qhat, s)) != cudaSuccess) return e;
        e = factor_blocked(n_layers, D, state, n_total, lambda_abs, lambda_rel, (float*)qhat, n_q, ld_qhat, s);
        if (e != cudaSuccess) return e;
        return apply_blocked(n_layers, D, state, n_q, (float*)qhat, ld_qhat, false, s);
    }
    // fp32 state, whole 32-column blocks, up to 256 queries: factorisation and both
    // substitutions in one cluster launch per call;
    // otherwise FACTOR, then APPLY
    if (sdt == TDA_F32 && !(blocked_states(D) && blocked_pc(D, sdt)) && D % kNB == 0 && D >= 2 * kNB &&
        n_q >= 1 && n_q <= 256) {
        const QArgs qa{q, (float*)qhat, n_q, ld_q, ld_qhat};
        e = factor_cluster<16, true>(n_layers, D, state, n_total, lambda_abs, lambda_rel, qa, s);
        if (e == cudaErrorNotSupported)
            e = factor_cluster<8, true>(n_layers, D, state, n_total, lambda_abs, lambda_rel, qa, s);
        if (e != cudaErrorNotSupported) return e;
    }
    e = launch_pc_factor(n_layers, D, sdt, state, n_total, lambda_abs, lambda_rel, s);
    if (e != cudaSuccess) return e;
    return launch_pc_apply(n_layers, D, sdt, state, q, n_q, ld_q, qhat, ld_qhat, s);
}

cudaError_t launch_pc_apply(int n_layers, int64_t D, tda_dtype sdt, const void* state, const float* q,
                            int64_t n_q, int64_t ld_q, void* qhat, int64_t ld_qhat, cudaStream_t s) {
    if (n_q == 0) return cudaSuccess;
    // a blocked factorisation left L^T in M's upper triangle: tensor-core substitutions
    if (blocked_states(D) && apply_blocked_ok(D, sdt, ld_q, qhat, ld_qhat, n_q)) {
        const cudaError_t e = copy_queries(n_layers, D, q, n_q, ld_q, (float*)qhat, ld_qhat, s);
        return e != cudaSuccess ? e : apply_blocked(n_layers, D, state, n_q, (float*)qhat, ld_qhat, true, s);
    }
    const size_t el = sdt == TDA_F64 ? 8 : 4;
    const size_t budget = 160 * 1024;
    if (sdt == TDA_F64) {
        // fewer queries per CTA while CTAs are what is missing (the fp64 pipe is per SM)
        if ((size_t)D * el * 8 <= budget && (n_q + 1) / 2 * n_layers >= 152)
            return apply_impl<double, 8>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
        if ((size_t)D * el * 2 <= budget && n_q * n_layers >= 152)
            return apply_impl<double, 2>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
        return apply_impl<double, 1>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
    }
    if ((size_t)D * el * 4 <= budget) return apply_impl<float, 4>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
    if ((size_t)D * el * 2 <= budget) return apply_impl<float, 2>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
    return apply_impl<float, 1>(n_layers, D, state, q, n_q, ld_q, qhat, ld_qhat, s);
}

}  // namespace tda
