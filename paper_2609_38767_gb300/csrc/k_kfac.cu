// k_kfac.cu -- K-FAC and EK-FAC on projected factors (the paper applies both
// Kronecker-factored curvature methods to the projected pair (a~, g~)
// unchanged, App. A.2, and damps by a multiple of the mean eigenvalue,
// App. B.2):
//   factor covariances  C_a = (1/M) sum a~ a~^T, C_g = (1/M) sum g~ g~^T,
//   eigenbases          C = U diag(w) U^T (parallel cyclic Jacobi, fp64),
//   EK-FAC eigenvalues  Lam = (1/N) sum_i (U_g^T Phi_i U_a)^2,
//   preconditioning     Qhat = U_g [(U_g^T Q U_a) / (Lam + lambda)] U_a^T.
// Sums over examples go through per-CTA partials reduced in a fixed order, so
// results do not depend on scheduling.
#include "tda_internal.cuh"

namespace tda {

// fp64 state of one layer, offsets in doubles
struct KfLayout {
    int64_t ka, kg, Sa, Sg, Ua, wa, Ug, wg, Le, total;
    __host__ __device__ explicit KfLayout(int64_t k_in, int64_t k_out) : ka(k_in), kg(k_out) {
        Sa = 8;  // header: [0] M token positions, [1] N examples (EK-FAC), [2] Jacobi sweeps a, [3] sweeps g
        Sg = Sa + ka * ka;
        Ua = Sg + kg * kg;
        wa = Ua + ka * ka;
        Ug = wa + ka;
        wg = Ug + kg * kg;
        Le = wg + kg;
        total = Le + ka * kg;
    }
};

size_t kfac_state_bytes(int64_t k_in, int64_t k_out) {
    const KfLayout l(k_in, k_out);
    return ((size_t)l.total * 8 + 255) & ~(size_t)255;
}

namespace {

constexpr int kKfThreads = 256;

// part[b][i*k+j] = sum over the rows of block b of Y[r][i] * Y[r][j] (fp32)
__global__ void __launch_bounds__(kKfThreads)
cov_partial_kernel(const float* __restrict__ Y, int64_t rows, int k, int64_t rows_per_block, float* __restrict__ part) {
    extern __shared__ float ys[];  // [64][k]
    const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
    int64_t r1 = r0 + rows_per_block;
    if (r1 > rows) r1 = rows;
    const int kk = k * k;
    constexpr int kMaxPer = 64;  // k <= 128: k*k / 256 <= 64 entries per thread
    float acc[kMaxPer];
#pragma unroll
    for (int m = 0; m < kMaxPer; ++m) acc[m] = 0.f;
    for (int64_t b0 = r0; b0 < r1; b0 += 64) {
        const int nr = (int)((r1 - b0) < 64 ? (r1 - b0) : 64);
        __syncthreads();
        for (int x = threadIdx.x; x < nr * k; x += blockDim.x) ys[x] = Y[b0 * k + x];
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kMaxPer; ++m) {
            const int e = threadIdx.x + m * kKfThreads;
            if (e < kk) {
                const int i = e / k, j = e - (e / k) * k;
                float a = acc[m];
                for (int r = 0; r < nr; ++r) a = fmaf(ys[r * k + i], ys[r * k + j], a);
                acc[m] = a;
            }
        }
    }
    float* out = part + (int64_t)blockIdx.x * kk;
#pragma unroll
    for (int m = 0; m < kMaxPer; ++m) {
        const int e = threadIdx.x + m * kKfThreads;
        if (e < kk) out[e] = acc[m];
    }
}

// S[e] += scale * sum_b part[b * stride + e] in fp64, n entries: the first n0 to S0, the others to
// S1; header[slot] += add. A CTA has 32 entries: each of its 8 warps adds an eighth of the blocks in
// order, then the eighths are added in order. (One thread per entry is a chain of loads and of fp64
// adds on four SMs: 35 us for the 152 blocks of a k = 32 projection, twice per linear; 6 now.)
__global__ void __launch_bounds__(256)
sum_partials_kernel(const float* __restrict__ part, int nblk, int64_t stride, int64_t n, int64_t n0,
                    double* __restrict__ S0, double* __restrict__ S1, double scale, double* __restrict__ header,
                    int slot, double add) {
    __shared__ double sub[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (nblk + 7) / 8, b0 = warp * per, b1 = b0 + per < nblk ? b0 + per : nblk;
    const int64_t e = (int64_t)blockIdx.x * 32 + lane;
    double v = 0.0;
    if (e < n)
#pragma unroll 8
        for (int b = b0; b < b1; ++b) v += (double)part[(int64_t)b * stride + e];
    sub[warp][lane] = v;
    __syncthreads();
    if (warp == 0 && e < n) {
        for (int w = 1; w < 8; ++w) v += sub[w][lane];
        double* dst = e < n0 ? S0 + e : S1 + (e - n0);
        *dst += scale * v;
    }
    if (header && blockIdx.x == 0 && threadIdx.x == 0) header[slot] += add;
}

__device__ __forceinline__ float j_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double j_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float j_abs(float x) { return fabsf(x); }
__device__ __forceinline__ double j_abs(double x) { return fabs(x); }

// Parallel cyclic Jacobi (round-robin pair ordering) by one CTA on the
// symmetric n x n matrix A in shared memory (row stride lda), accumulating
// V <- V J (row stride ldv). Each round rotates floor(m/2) disjoint pairs at
// once: angles from the round's starting matrix, then all row updates, then
// all column updates, which is J^T A J for the product J of the round's
// rotations. Stops when the off-diagonal squared norm is <= tol * fro (fro =
// squared norm of A at entry); returns the sweep count, or -1 after
// max_sweeps. Shared matrices use an odd row stride (n + 1) so that the column
// updates, whose threads walk down a column, hit distinct banks.
template <typename T>
__device__ int jacobi_sweeps(T* A, int lda, T* V, int ldv, int n, T* cs, T* sn, int* P, int* Q, double* red, int* done,
                             double tol, int max_sweeps) {
    const int m = (n + 1) & ~1;  // even number of players; index n is a dummy when n is odd
    double f = 0.0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const double a = (double)A[(e / n) * lda + e % n];
        f += a * a;
    }
    red[threadIdx.x] = f;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    const double fro = red[0];
    __syncthreads();
    const int W = n <= 32 ? 32 : (n <= 64 ? 64 : 128);
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        double off = 0.0;
        for (int e = threadIdx.x; e < n * n; e += blockDim.x)
            if (e / n != e % n) {
                const double a = (double)A[(e / n) * lda + e % n];
                off += a * a;
            }
        red[threadIdx.x] = off;
        __syncthreads();
        for (int h = blockDim.x / 2; h > 0; h >>= 1) {
            if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
            __syncthreads();
        }
        if (threadIdx.x == 0) *done = (red[0] <= tol * fro) ? 1 : 0;
        __syncthreads();
        if (*done) return sweep;
        for (int r = 0; r < m - 1; ++r) {
            for (int i = threadIdx.x; i < m / 2; i += blockDim.x) {
                int p = i == 0 ? r : (r + i) % (m - 1);
                int q = i == 0 ? m - 1 : (r - i + m - 1) % (m - 1);
                if (p > q) {
                    const int t = p;
                    p = q;
                    q = t;
                }
                T c = 1, sv = 0;
                if (q < n) {
                    const T apq = A[p * lda + q];
                    if (apq != T(0)) {
                        const T tau = (A[q * lda + q] - A[p * lda + p]) / (T(2) * apq);
                        const T t = (tau >= T(0) ? T(1) : T(-1)) / (j_abs(tau) + j_sqrt(T(1) + tau * tau));
                        c = T(1) / j_sqrt(T(1) + t * t);
                        sv = t * c;
                    }
                }
                cs[i] = c;
                sn[i] = sv;
                P[i] = p;
                Q[i] = q < n ? q : -1;
            }
            __syncthreads();
            // threads walk (pair, k) with k along a power of two of at least n (no divisions)
            const int half = m / 2, k = threadIdx.x & (W - 1), step = blockDim.x / W;
            if (k < n)
                for (int i = threadIdx.x / W; i < half; i += step) {  // rows p, q: A <- J^T A; V <- V J
                    const int p = P[i], q = Q[i];
                    const T c = cs[i], sv = sn[i];
                    if (q < 0 || sv == T(0)) continue;
                    const T apk = A[p * lda + k], aqk = A[q * lda + k];
                    const T vkp = V[k * ldv + p], vkq = V[k * ldv + q];
                    A[p * lda + k] = c * apk - sv * aqk;
                    A[q * lda + k] = sv * apk + c * aqk;
                    V[k * ldv + p] = c * vkp - sv * vkq;
                    V[k * ldv + q] = sv * vkp + c * vkq;
                }
            __syncthreads();
            if (k < n)
                for (int i = threadIdx.x / W; i < half; i += step) {  // columns p, q: A <- A J
                    const int p = P[i], q = Q[i];
                    const T c = cs[i], sv = sn[i];
                    if (q < 0 || sv == T(0)) continue;
                    const T akp = A[k * lda + p], akq = A[k * lda + q];
                    A[k * lda + p] = c * akp - sv * akq;
                    A[k * lda + q] = sv * akp + c * akq;
                }
            __syncthreads();
        }
    }
    return -1;
}

// out = X^T Y (tx) or X Y, n x n fp64 in the shared memory of every CTA of a cluster of cs (the same
// X and Y in each, row stride ld): CTA r computes an equal share of the entries and writes them to
// all. fp64 runs at two multiply-adds a clock and SM, so eight SMs take an eighth of the time.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ void gemm_nn(double* out, const double* X, const double* Y, int n, int ld, bool tx, int cs, int rank) {
    cluster_barrier();  // every CTA is done with what `out` held
    const int total = n * n, per = (total + cs - 1) / cs;
    const int e1 = (rank + 1) * per < total ? (rank + 1) * per : total;
    for (int e = rank * per + threadIdx.x; e < e1; e += blockDim.x) {
        const int i = e / n, j = e - i * n;
        double acc = 0.0;
#pragma unroll 4
        for (int k = 0; k < n; ++k) acc += (tx ? X[k * ld + i] : X[i * ld + k]) * Y[k * ld + j];
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(out + i * ld + j);
        for (int r = 0; r < cs; ++r) {
            uint32_t dst;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(at), "r"(r));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst), "d"(acc) : "memory");
        }
    }
    cluster_barrier();  // the whole product is in every CTA
}
// V <- V (3I - V^T V) / 2: one Newton-Schulz step towards orthonormal columns (T1, T2: scratch). A
// deviation of d becomes n d^2 at most, so the step is not the last one if d was above 1e-9: returns whether
// it was (in every CTA alike: they hold the same V^T V).
__device__ bool orthonormalise(double* V, double* T1, double* T2, int n, int ld, int cs, int rank) {
    gemm_nn(T1, V, V, n, ld, true, cs, rank);
    // (the diagonal by two warps, the rest by their high words, 1e-9's is 0x3E112E0B: fp64 comparisons of
    // all entries took 6 us of a call)
    int far = (int)threadIdx.x < n && fabs(T1[threadIdx.x * ld + threadIdx.x] - 1.0) > 1e-9;
    __syncthreads();
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int i = e / n, j = e % n;
        const double t = T1[i * ld + j];
        far |= i != j && (__double2hiint(t) & 0x7FFFFFFF) > 0x3E112E0B;
        T1[i * ld + j] = ((i == j) ? 1.5 : 0.0) - 0.5 * t;
    }
    far = __syncthreads_or(far);
    gemm_nn(T2, V, T1, n, ld, false, cs, rank);
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) V[(e / n) * ld + e % n] = T2[(e / n) * ld + e % n];
    __syncthreads();
    return far;
}

// Eigenbases of C = S / M for the a side (blockIdx.x 0) and the g side (1) of
// layer blockIdx.y, C = U diag(w) U^T.
//   n <= 64 (MIXED): a cluster of cs CTAs per side and layer. The sweeps run in
//   fp32 (the fp64 pipe is a small fraction of the fp32 one here), the same in
//   every CTA, until the off-diagonal part is near fp32 rounding. Then, in fp64
//   and with products shared by the cluster: a Newton-Schulz step
//   V <- V (3I - V^T V) / 2, A = V^T C V afresh, and twice the first-order
//   rotation of all pairs at once, V <- V (I + E) with E_ij = A_ij / (A_jj - A_ii),
//   made orthonormal by Newton-Schulz steps, one mostly (errors of 1e-7 become 1e-14,
//   then rounding; pairs with a gap below 1000 |A_ij| are left out). fp64 sweeps
//   finish what is left: none, mostly, where two used to take most of the time
//   (three k = 32 layers: 576 us, 220 now). The header gets the fp64 sweep count.
//   n > 64, and up to 2: fp64 sweeps from the start, V (n > 64) in the state's U.
template <bool MIXED>
__global__ void __launch_bounds__(kKfThreads)
jacobi_kernel(double* __restrict__ st0, int64_t stride, int64_t ka, int64_t kg, int cs) {
    extern __shared__ double smd[];
    double* st = st0 + (int64_t)blockIdx.y * stride;
    const KfLayout l(ka, kg);
    const bool side_g = (int)blockIdx.x / cs == 1;
    const int rank = (int)blockIdx.x % cs;
    const int n = (int)(side_g ? kg : ka);
    const double* S = st + (side_g ? l.Sg : l.Sa);
    double* U = st + (side_g ? l.Ug : l.Ua);
    double* w = st + (side_g ? l.wg : l.wa);
    const int nmax = (int)(ka > kg ? ka : kg), mh = (nmax + 2) / 2, ld = n + 1, sq = nmax * (nmax + 1);
    __shared__ double red[kKfThreads];
    __shared__ int done;
    const double Mtok = st[0];
    const double inv = Mtok > 0 ? 1.0 / Mtok : 0.0;
    double* A = smd;  // [n][ld]
    int sweeps;
    // every CTA of the cluster reads the sums before rank 0 writes the results (the a side's rank 0
    // also clears the EK-FAC sums, which nothing here reads)
    if constexpr (MIXED) {
        double* V = A + sq;
        double* Tm = V + sq;  // fp64 scratch
        double* cs64 = Tm + sq;
        double* sn = cs64 + mh;
        float* A32 = (float*)(sn + mh);
        float* V32 = A32 + sq;
        float* cs32 = V32 + sq;
        float* sn32 = cs32 + mh;
        int* P = (int*)(sn32 + mh);
        int* Q = P + mh;
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const int i = e / n, j = e % n;
            A32[i * ld + j] = (float)(S[e] * inv);
            V32[i * ld + j] = (i == j) ? 1.f : 0.f;
        }
        __syncthreads();
        // fp32: the off-diagonal part down to about 1e-6 of ||C|| (near fp32 rounding; at most
        // 20 sweeps, since fp32 cannot go much further)
        jacobi_sweeps<float>(A32, ld, V32, ld, n, cs32, sn32, P, Q, red, &done, 1e-12, 20);
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const int i = e / n, j = e % n;
            V[i * ld + j] = (double)V32[i * ld + j];
        }
        __syncthreads();
        auto form_a = [&]() {  // A = V^T C V
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) A[(e / n) * ld + e % n] = S[e] * inv;
            __syncthreads();
            gemm_nn(Tm, A, V, n, ld, false, cs, rank);
            gemm_nn(A, V, Tm, n, ld, true, cs, rank);
        };
        orthonormalise(V, Tm, A, n, ld, cs, rank);
        form_a();
        for (int it = 0; it < 2; ++it) {
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
                const int i = e / n, j = e % n;
                const double gap = A[j * ld + j] - A[i * ld + i], a = A[i < j ? i * ld + j : j * ld + i];
                Tm[i * ld + j] = i == j ? 1.0 : (fabs(a) < 1e-3 * fabs(gap) ? a / gap : 0.0);
            }
            __syncthreads();
            gemm_nn(A, V, Tm, n, ld, false, cs, rank);
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) V[(e / n) * ld + e % n] = A[(e / n) * ld + e % n];
            __syncthreads();
            // many pairs just past the gap's limit turn V by up to 0.06: then one last step is not enough
            for (int r = 0; orthonormalise(V, Tm, A, n, ld, cs, rank) && it == 1 && r < 3; ++r) {
            }
            form_a();
        }
        sweeps = jacobi_sweeps<double>(A, ld, V, ld, n, cs64, sn, P, Q, red, &done, 1e-28, 60);
        if (rank == 0)
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) U[e] = V[(e / n) * ld + e % n];
        cluster_barrier();  // no CTA leaves while another may still write to it
        if (rank != 0) return;
    } else {
        const bool v_shared = nmax <= 64;
        double* V = v_shared ? A + sq : U;
        const int ldv = v_shared ? ld : n;
        double* c1 = A + (v_shared ? 2 : 1) * sq;
        double* sn = c1 + mh;
        int* P = (int*)(sn + mh);
        int* Q = P + mh;
        for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
            const int i = e / n, j = e % n;
            A[i * ld + j] = S[e] * inv;
            V[i * ldv + j] = (i == j) ? 1.0 : 0.0;
        }
        __syncthreads();
        sweeps = jacobi_sweeps<double>(A, ld, V, ldv, n, c1, sn, P, Q, red, &done, 1e-28, 60);
        if (v_shared)
            for (int e = threadIdx.x; e < n * n; e += blockDim.x) U[e] = V[(e / n) * ld + e % n];
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) w[i] = A[i * ld + i];
    if (threadIdx.x == 0) st[2 + (side_g ? 1 : 0)] = (double)sweeps;
    if (!side_g) {  // a new eigenbasis invalidates the EK-FAC sums
        for (int64_t e = threadIdx.x; e < ka * kg; e += blockDim.x) st[l.Le + e] = 0.0;
        if (threadIdx.x == 0) st[1] = 0.0;
    }
}

// Eigenbases of one layer as fp32 in shared memory (SU) or read from the fp64
// state (large k).
template <bool SU>
struct Bases {
    const float* ua;
    const float* ug;
    const double* uad;
    const double* ugd;
    __device__ __forceinline__ float a(int64_t i) const { return SU ? ua[i] : (float)uad[i]; }
    __device__ __forceinline__ float g(int64_t i) const { return SU ? ug[i] : (float)ugd[i]; }
};

// part[layer][b][r*ka+c] = sum over the examples of block b of ((U_g^T Phi_i U_a)[r][c])^2
template <bool SU>
__global__ void __launch_bounds__(kKfThreads)
ekfac_partial_kernel(const float* __restrict__ phi, int64_t n, int64_t ld, const double* __restrict__ st0,
                     int64_t stride, int64_t ka, int64_t kg, float* __restrict__ part) {
    extern __shared__ float sm[];  // [U_a, U_g if SU] Phi_i [kg][ka], Y [kg][ka]
    const int layer = blockIdx.y;
    const double* st = st0 + (int64_t)layer * stride;
    const KfLayout l(ka, kg);
    const int64_t D = ka * kg;
    float* F = sm + (SU ? ka * ka + kg * kg : 0);
    float* Y = F + D;
    Bases<SU> U{sm, sm + ka * ka, st + l.Ua, st + l.Ug};
    if (SU) {
        for (int64_t e = threadIdx.x; e < ka * ka; e += blockDim.x) sm[e] = (float)st[l.Ua + e];
        for (int64_t e = threadIdx.x; e < kg * kg; e += blockDim.x) sm[ka * ka + e] = (float)st[l.Ug + e];
    }
    const float* ph = phi + (int64_t)layer * D;
    constexpr int kMaxPer = 64;
    float acc[kMaxPer];
#pragma unroll
    for (int m = 0; m < kMaxPer; ++m) acc[m] = 0.f;
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        __syncthreads();
        for (int64_t e = threadIdx.x; e < D; e += blockDim.x) F[e] = ph[i * ld + e];
        __syncthreads();
        for (int64_t e = threadIdx.x; e < D; e += blockDim.x) {  // Y = Phi U_a
            const int64_t r = e / ka, c = e - (e / ka) * ka;
            float sacc = 0.f;
            for (int64_t j = 0; j < ka; ++j) sacc = fmaf(F[r * ka + j], U.a(j * ka + c), sacc);
            Y[e] = sacc;
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kMaxPer; ++m) {  // X = U_g^T Y, accumulate X^2
            const int64_t e = threadIdx.x + (int64_t)m * kKfThreads;
            if (e < D) {
                const int64_t r = e / ka, c = e - (e / ka) * ka;
                float sacc = 0.f;
                for (int64_t j = 0; j < kg; ++j) sacc = fmaf(U.g(j * kg + r), Y[j * ka + c], sacc);
                acc[m] = fmaf(sacc, sacc, acc[m]);
            }
        }
    }
    float* out = part + ((int64_t)layer * gridDim.x + blockIdx.x) * D;
#pragma unroll
    for (int m = 0; m < kMaxPer; ++m) {
        const int64_t e = threadIdx.x + (int64_t)m * kKfThreads;
        if (e < D) out[e] = acc[m];
    }
}

// Square k = 16, 32, 64: thread (column c, row group g) keeps U_a[:, c] and,
// per example, column c of Y = Phi U_a in registers; Phi and U_g^T rows are
// read from shared memory as warp broadcasts, so each multiply-add costs a
// quarter of a (vector) shared load.
template <int K>
__global__ void __launch_bounds__(256)
ekfac_reg_kernel(const float* __restrict__ phi, int64_t n, int64_t ld, const double* __restrict__ st0, int64_t stride,
                 float* __restrict__ part) {
    constexpr int RG = 256 / K;  // row groups
    constexpr int RPT = K / RG;  // rows per thread
    __shared__ __align__(16) float F[K * K];    // Phi_i [r][j]
    __shared__ __align__(16) float Y[K * K];    // Phi_i U_a [r][c]
    __shared__ __align__(16) float UgT[K * K];  // U_g^T [r][j]
    const int layer = blockIdx.y;
    const double* st = st0 + (int64_t)layer * stride;
    const KfLayout l(K, K);
    const int c = threadIdx.x % K, g = threadIdx.x / K;
    float ua[K];
#pragma unroll
    for (int j = 0; j < K; ++j) ua[j] = (float)st[l.Ua + j * K + c];
    for (int e = threadIdx.x; e < K * K; e += 256) UgT[e] = (float)st[l.Ug + (e % K) * K + e / K];
    float acc[RPT];
#pragma unroll
    for (int m = 0; m < RPT; ++m) acc[m] = 0.f;
    const float* ph = phi + (int64_t)layer * K * K;
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        __syncthreads();
        for (int e = threadIdx.x; e < K * K / 4; e += 256)
            reinterpret_cast<float4*>(F)[e] = reinterpret_cast<const float4*>(ph + i * ld)[e];
        __syncthreads();
#pragma unroll
        for (int m = 0; m < RPT; ++m) {  // Y[r][c] = sum_j Phi[r][j] U_a[j][c]
            const int r = g + RG * m;
            float sacc = 0.f;
#pragma unroll
            for (int j = 0; j < K; j += 4) {
                const float4 f = *reinterpret_cast<const float4*>(F + r * K + j);
                sacc = fmaf(f.x, ua[j], sacc);
                sacc = fmaf(f.y, ua[j + 1], sacc);
                sacc = fmaf(f.z, ua[j + 2], sacc);
                sacc = fmaf(f.w, ua[j + 3], sacc);
            }
            Y[r * K + c] = sacc;
        }
        __syncthreads();
        float yc[K];
#pragma unroll
        for (int j = 0; j < K; ++j) yc[j] = Y[j * K + c];
#pragma unroll
        for (int m = 0; m < RPT; ++m) {  // X[r][c] = sum_j U_g[j][r] Y[j][c]; accumulate X^2
            const int r = g + RG * m;
            float sacc = 0.f;
#pragma unroll
            for (int j = 0; j < K; j += 4) {
                const float4 u = *reinterpret_cast<const float4*>(UgT + r * K + j);
                sacc = fmaf(u.x, yc[j], sacc);
                sacc = fmaf(u.y, yc[j + 1], sacc);
                sacc = fmaf(u.z, yc[j + 2], sacc);
                sacc = fmaf(u.w, yc[j + 3], sacc);
            }
            acc[m] = fmaf(sacc, sacc, acc[m]);
        }
    }
    float* out = part + ((int64_t)layer * gridDim.x + blockIdx.x) * K * K;
#pragma unroll
    for (int m = 0; m < RPT; ++m) out[(g + RG * m) * K + c] = acc[m];
}

// Le of every layer += its block partials (in fixed order: eighths of the blocks as in
// sum_partials_kernel); N += n
__global__ void __launch_bounds__(256)
ekfac_reduce_kernel(const float* __restrict__ part, int nblk, double* __restrict__ st0, int64_t stride,
                    int64_t ka, int64_t kg, double n) {
    __shared__ double sub[8][32];
    const int layer = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* st = st0 + (int64_t)layer * stride;
    const KfLayout l(ka, kg);
    const int64_t D = ka * kg, e = (int64_t)blockIdx.x * 32 + lane;
    const float* pl = part + (int64_t)layer * nblk * D;
    const int per = (nblk + 7) / 8, b0 = warp * per, b1 = b0 + per < nblk ? b0 + per : nblk;
    double v = 0.0;
    if (e < D)
#pragma unroll 8
        for (int b = b0; b < b1; ++b) v += (double)pl[(int64_t)b * D + e];
    sub[warp][lane] = v;
    __syncthreads();
    if (warp == 0 && e < D) {
        for (int w = 1; w < 8; ++w) v += sub[w][lane];
        st[l.Le + e] += v;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) st[1] += n;
}

// One CTA per (query row, layer): Qhat = U_g [(U_g^T Q U_a) / (Lam + lambda)] U_a^T. U_a's rows are
// padded in shared memory: the last product but one walks down its columns (32 threads on one bank
// otherwise: 64 us for 64 queries of three k = 32 layers, 27 now).
template <bool SU>
__global__ void __launch_bounds__(kKfThreads)
kfac_apply_kernel(int kind, const double* __restrict__ st0, int64_t stride, int ka, int kg,
                  double lambda_abs, double lambda_rel, const float* __restrict__ q, int64_t ld_q,
                  float* __restrict__ qhat, int64_t ld_qhat) {
    extern __shared__ float sm[];  // [U_a (padded), U_g if SU] X [kg][ka], Y [kg][ka]
    const int layer = blockIdx.y;
    const double* st = st0 + (int64_t)layer * stride;
    const KfLayout l(ka, kg);
    const int D = ka * kg, lda = SU ? ka + 1 : ka;
    float* X = sm + (SU ? ka * lda + kg * kg : 0);
    float* Y = X + D;
    Bases<SU> U{sm, sm + ka * lda, st + l.Ua, st + l.Ug};
    if (SU) {
        for (int e = threadIdx.x; e < ka * ka; e += blockDim.x) sm[e / ka * lda + e % ka] = (float)st[l.Ua + e];
        for (int e = threadIdx.x; e < kg * kg; e += blockDim.x) sm[ka * lda + e] = (float)st[l.Ug + e];
    }
    __shared__ double red[kKfThreads];
    // Lam[e] = scale * raw(e): EK-FAC's sums are divided by the example count once
    const double nex = st[1], scale = kind == 0 ? 1.0 : (nex > 0 ? 1.0 / nex : 0.0);
    auto raw = [&](int e) -> double {
        return kind == 0 ? st[l.wg + e / ka] * st[l.wa + e % ka] : st[l.Le + e];
    };
    double sacc = 0.0;
    for (int e = threadIdx.x; e < D; e += blockDim.x) sacc += raw(e);
    red[threadIdx.x] = sacc;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    const double lambda = lambda_abs + lambda_rel * (scale * red[0]) / (double)D;
    const float* qi = q + (int64_t)blockIdx.x * ld_q + (int64_t)layer * D;
    for (int e = threadIdx.x; e < D; e += blockDim.x) X[e] = qi[e];
    __syncthreads();
    for (int e = threadIdx.x; e < D; e += blockDim.x) {  // Y = Q U_a
        const int r = e / ka, c = e - r * ka;
        float a = 0.f;
#pragma unroll 8
        for (int j = 0; j < ka; ++j) a = fmaf(X[r * ka + j], U.a(j * lda + c), a);
        Y[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < D; e += blockDim.x) {  // X = (U_g^T Y) / (Lam + lambda)
        const int r = e / ka, c = e - r * ka;
        float a = 0.f;
#pragma unroll 8
        for (int j = 0; j < kg; ++j) a = fmaf(U.g(j * kg + r), Y[j * ka + c], a);
        X[e] = (float)((double)a / (scale * raw(e) + lambda));
    }
    __syncthreads();
    for (int e = threadIdx.x; e < D; e += blockDim.x) {  // Y = X U_a^T
        const int r = e / ka, c = e - r * ka;
        float a = 0.f;
#pragma unroll 8
        for (int j = 0; j < ka; ++j) a = fmaf(X[r * ka + j], U.a(c * lda + j), a);
        Y[e] = a;
    }
    __syncthreads();
    float* out = qhat + (int64_t)blockIdx.x * ld_qhat + (int64_t)layer * D;
    for (int e = threadIdx.x; e < D; e += blockDim.x) {  // out = U_g Y
        const int r = e / ka, c = e - r * ka;
        float a = 0.f;
#pragma unroll 8
        for (int j = 0; j < kg; ++j) a = fmaf(U.g(r * kg + j), Y[j * ka + c], a);
        out[e] = a;
    }
}

}  // namespace

int kfac_partial_blocks(int64_t rows) {
    int64_t b = (rows + 255) / 256;
    if (b > 304) b = 304;
    return b < 1 ? 1 : (int)b;
}

// S += scale * Y^T Y for rows x k fp32 rows Y (deterministic), header M += add_m.
cudaError_t launch_kfac_cov(const float* Y, int64_t rows, int k, double* S, double scale, double* header,
                            double add_m, float* part, cudaStream_t s) {
    if (rows == 0) {
        if (header && add_m != 0) {
            note_launches(1);
            sum_partials_kernel<<<1, 256, 0, s>>>(part, 0, 0, 0, 0, S, nullptr, scale, header, 0, add_m);
        }
        return cudaGetLastError();
    }
    const int nb = kfac_partial_blocks(rows);
    int64_t per = (rows + nb - 1) / nb;
    per = (per + 63) / 64 * 64;
    const int nblk = (int)((rows + per - 1) / per);
    note_launches(2);
    cov_partial_kernel<<<nblk, kKfThreads, (size_t)64 * k * 4, s>>>(Y, rows, k, per, part);
    sum_partials_kernel<<<(unsigned)((k * k + 31) / 32), 256, 0, s>>>(part, nblk, (int64_t)k * k, (int64_t)k * k,
                                                                      (int64_t)k * k, S, nullptr, scale, header, 0,
                                                                      add_m);
    return cudaGetLastError();
}

// Sums of per-CTA partials written by another kernel (the fused projection): n0 entries to S0 and
// n - n0 to S1.
cudaError_t launch_kfac_sum_partials(const float* part, int nblk, int64_t stride, int64_t n, int64_t n0, double* S0,
                                     double* S1, double scale, double* header, int slot, double add, cudaStream_t s) {
    note_launches(1);
    sum_partials_kernel<<<(unsigned)(n > 0 ? (n + 31) / 32 : 1), 256, 0, s>>>(part, nblk, stride, n, n0, S0, S1, scale,
                                                                              header, slot, add);
    return cudaGetLastError();
}

cudaError_t launch_kfac_eigen(int n_layers, double* state, int64_t ka, int64_t kg, cudaStream_t s) {
    const int64_t nmax = ka > kg ? ka : kg;
    const int64_t mh = (nmax + 2) / 2, sq = nmax * (nmax + 1);
    const int64_t stride = (int64_t)kfac_state_bytes(ka, kg) / 8;
    cudaError_t e;
    note_launches(1);
    // up to 2 columns: the fp64 sweeps alone, without the refinement's cluster barriers (k = 1 6 us and 23 with them,
    // k = 2 9 and 27 us, k = 3 33 to 43 and 34 us)
    if (nmax <= 64 && nmax > 2) {
        const size_t smem = (size_t)3 * sq * 8 + (size_t)mh * (8 + 8) + (size_t)2 * sq * 4 + (size_t)mh * (4 + 4 + 4 + 4);
        // the largest shared memory of n <= 64, set once per device
        constexpr int kMax = (int)((size_t)3 * 64 * 65 * 8 + 33 * 16 + (size_t)2 * 64 * 65 * 4 + 33 * 16);
        if ((e = smem_attr_once<jacobi_kernel<true>>(kMax))) return e;
        // clusters of eight while all of them fit the chip at once, else one CTA a problem
        const int cs = (int64_t)n_layers * 2 * 8 <= 128 ? 8 : 1;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3((unsigned)(2 * cs), (unsigned)n_layers);
        cfg.blockDim = dim3(kKfThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if ((e = cudaLaunchKernelEx(&cfg, jacobi_kernel<true>, state, stride, ka, kg, cs))) return e;
        return cudaGetLastError();
    }
    const size_t smem = (size_t)(nmax <= 64 ? 2 : 1) * sq * 8 + (size_t)mh * (8 + 8 + 4 + 4);  // V in shared memory up to 64
    if ((e = cudaFuncSetAttribute(jacobi_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
        return e;
    jacobi_kernel<false><<<dim3(2, (unsigned)n_layers), kKfThreads, smem, s>>>(state, stride, ka, kg, 1);
    return cudaGetLastError();
}

// EK-FAC sums of n_layers layers whose features sit side by side in phi
// (layer l at column l*ka*kg); part holds n_layers * nblk * ka*kg floats.
cudaError_t launch_kfac_ekfac_accum(int n_layers, double* state, int64_t ka, int64_t kg, const float* phi, int64_t n,
                                    int64_t ld, float* part, int nblk, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const bool su = ka <= 64 && kg <= 64;
    const size_t smem = (size_t)(2 * ka * kg + (su ? ka * ka + kg * kg : 0)) * 4;
    const int64_t stride = (int64_t)kfac_state_bytes(ka, kg) / 8;
    const dim3 grid((unsigned)nblk, (unsigned)n_layers);
    const bool aligned = ((uintptr_t)phi & 15) == 0 && (ld & 3) == 0;
    if (ka == kg && aligned && (ka == 16 || ka == 32 || ka == 64)) {
        note_launches(2);
        if (ka == 16)
            ekfac_reg_kernel<16><<<grid, 256, 0, s>>>(phi, n, ld, state, stride, part);
        else if (ka == 32)
            ekfac_reg_kernel<32><<<grid, 256, 0, s>>>(phi, n, ld, state, stride, part);
        else
            ekfac_reg_kernel<64><<<grid, 256, 0, s>>>(phi, n, ld, state, stride, part);
        ekfac_reduce_kernel<<<dim3((unsigned)((ka * kg + 31) / 32), (unsigned)n_layers), 256, 0, s>>>(
            part, nblk, state, stride, ka, kg, (double)n);
        return cudaGetLastError();
    }
    cudaError_t e = su ? cudaFuncSetAttribute(ekfac_partial_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)smem)
                       : cudaFuncSetAttribute(ekfac_partial_kernel<false>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    note_launches(2);
    if (su)
        ekfac_partial_kernel<true><<<grid, kKfThreads, smem, s>>>(phi, n, ld, state, stride, ka, kg, part);
    else
        ekfac_partial_kernel<false><<<grid, kKfThreads, smem, s>>>(phi, n, ld, state, stride, ka, kg, part);
    ekfac_reduce_kernel<<<dim3((unsigned)((ka * kg + 31) / 32), (unsigned)n_layers), 256, 0, s>>>(
        part, nblk, state, stride, ka, kg, (double)n);
    return cudaGetLastError();
}

cudaError_t launch_kfac_apply(int kind, int n_layers, const double* state, int64_t ka, int64_t kg, double lambda_abs,
                              double lambda_rel, const float* q, int64_t n_q, int64_t ld_q, float* qhat,
                              int64_t ld_qhat, cudaStream_t s) {
    if (n_q == 0) return cudaSuccess;
    const bool su = ka <= 64 && kg <= 64;
    const size_t smem = (size_t)(2 * ka * kg + (su ? ka * (ka + 1) + kg * kg : 0)) * 4;
    const int64_t stride = (int64_t)kfac_state_bytes(ka, kg) / 8;
    cudaError_t e = su ? cudaFuncSetAttribute(kfac_apply_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)smem)
                       : cudaFuncSetAttribute(kfac_apply_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)smem);
    if (e != cudaSuccess) return e;
    note_launches(1);
    const dim3 grid((unsigned)n_q, (unsigned)n_layers);
    if (su)
        kfac_apply_kernel<true><<<grid, kKfThreads, smem, s>>>(kind, state, stride, (int)ka, (int)kg, lambda_abs, lambda_rel, q,
                                                               ld_q, qhat, ld_qhat);
    else
        kfac_apply_kernel<false><<<grid, kKfThreads, smem, s>>>(kind, state, stride, (int)ka, (int)kg, lambda_abs, lambda_rel,
                                                                q, ld_q, qhat, ld_qhat);
    return cudaGetLastError();
}

int64_t kfac_offset_sa(int64_t ka, int64_t kg) { return KfLayout(ka, kg).Sa; }
int64_t kfac_offset_sg(int64_t ka, int64_t kg) { return KfLayout(ka, kg).Sg; }

}  // namespace tda
