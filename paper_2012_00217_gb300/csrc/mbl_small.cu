// mbl_small.cu -- small dense kernels of the LOBPCG iteration (Sec. 3.2), each run by
// one block: symmetric eigendecomposition by parallel cyclic Jacobi, Cholesky with
// triangular inverse, the SVQB + Rayleigh-Ritz step on S = [X W P], and the selection
// of the Ritz pairs nearest sigma.
//
// Precision.  GB300 executes FP64 at about 1/64 of its FP32 rate, so in mixed mode
// the (3k x 3k) eigenproblems run in FP32 and only a k-dimensional refinement runs in
// FP64: the k Ritz directions picked in FP32 are re-orthonormalised (Cholesky, FP64)
// and a k x k Rayleigh-Ritz with the FP64 projection of A finishes the step.  The
// convergence test (H Rayleigh-Ritz and residuals) is always FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "mbl_dense.h"
#include "mbl_device.cuh"
#include "mbl_internal.h"

namespace mbl {

constexpr int kSmallThreads = 512;
constexpr int kMaxSweeps = 20;
constexpr int kMaxK = 64;        // block width limit of the solver
constexpr int kMaxW = 3 * kMaxK;  // width of S = [X W P]

template <typename T>
struct Eps;
template <>
struct Eps<float> {
    static __device__ __forceinline__ float v() { return 1.2e-7f; }
};
template <>
struct Eps<double> {
    static __device__ __forceinline__ double v() { return 2.3e-16; }
};

// Odd row stride for matrices in shared memory: walking down a column then touches a
// different bank in every lane.
__host__ __device__ inline int pad_ld(int n) { return n | 1; }

// The rotation (c, s) of one pair, or false where |a_pq| <= eps sqrt(|a_pp a_qq|):
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), tau = (a_qq - a_pp) / (2 a_pq), c = 1 / sqrt(1 +
// t^2), s = t c.
template <typename T>
__device__ __forceinline__ bool jacobi_rotation_exact(T apq, T app, T aqq, T &c, T &s)
{
    if (apq == (T)0 || !(fabs(apq) > Eps<T>::v() * sqrt(fabs(app * aqq)))) return false;
    const T tau = (aqq - app) / ((T)2 * apq);
    const T t = (tau >= (T)0 ? (T)1 : (T)-1) / (fabs(tau) + sqrt((T)1 + tau * tau));
    c = (T)1 / sqrt((T)1 + t * t);
    s = t * c;
    return true;
}

__device__ __forceinline__ bool jacobi_rotation(float apq, float app, float aqq, float &c, float &s)
{
    return jacobi_rotation_exact<float>(apq, app, aqq, c, s);
}

// FP64: the two divisions and three roots of the above are some hundred instructions of 64
// cycles each on GB300's FP64 pipe, more than the rest of a round.  A rotation only has to be
// orthogonal to FP64; that it leaves a_pq at 1e-7 of its value instead of zero costs nothing,
// the sweeps converge as before.  So t comes from FP32, from a_qq - a_pp and a_pq scaled by a
// common power of two, and c = 1 / sqrt(1 + t^2) from an FP32 start and two Newton steps in
// FP64 (relative error 1e-7 -> 1e-14 -> below rounding).  H Rayleigh-Ritz at k = 32, Grams
// and updates included: 2.01 -> 1.77 ms at L = 20, 1.36 -> 1.13 ms at L = 18.
// tau^2 has to stay within FP32: from |tau| = 2^64 on it overflows, t would be zero, and a pair
// counted as rotated but left as it was keeps the sweeps going to their limit.  So pairs whose
// a_qq - a_pp is 2^60 times a_pq and more (graded matrices) take the FP64 rotation.
constexpr int kTauExponents = 60 << 20;  // in the high word of a double

__device__ __forceinline__ bool jacobi_rotation(double apq, double app, double aqq, double &c, double &s)
{
    if (apq == 0.0) return false;
    if (!(apq * apq > (Eps<double>::v() * Eps<double>::v()) * fabs(app * aqq))) {
        // below the bound, or squares that underflow (or overflow, or a NaN): the plain test
        if (fabs(apq) > 1e-140) return false;
        return jacobi_rotation_exact<double>(apq, app, aqq, c, s);
    }
    const double d = aqq - app;
    const int hd = __double2hiint(d) & 0x7ff00000, ha = __double2hiint(apq) & 0x7ff00000;
    const int e = max(hd, ha);
    // a_pq's exponent not far below the difference's, both away from the ends of the range (a
    // difference far below a_pq is as good as zero: t is +-1 to FP64)
    if (ha < e - kTauExponents || e < (200 << 20) || e > (1900 << 20))
        return jacobi_rotation_exact<double>(apq, app, aqq, c, s);
    const int shift = (1023 << 20) - e;
    const float df = hd < e - kTauExponents ? 0.0f : (float)__hiloint2double(__double2hiint(d) + shift, __double2loint(d));
    const float af = (float)__hiloint2double(__double2hiint(apq) + shift, __double2loint(apq));
    const float tau = df / (2.0f * af);
    const float tf = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.0f)));
    const double t = (double)tf, u = fma(t, t, 1.0);
    double y = (double)rsqrtf((float)u);
    y = y * fma(-0.5 * u, y * y, 1.5);
    y = y * fma(-0.5 * u, y * y, 1.5);
    c = y;
    s = t * y;
    return true;
}

// Parallel cyclic Jacobi on the symmetric n x n matrix A (row stride ld): the
// round-robin (circle) ordering rotates n/2 disjoint pairs per round (jacobi_rotation); pairs
// with |a_pq| <= eps sqrt(|a_pp a_qq|) are skipped (the relative test keeps the small
// eigenvalues of graded matrices accurate); sweeps stop when one rotates nothing or after
// max_sweeps.  On exit diag(A) holds the eigenvalues and the columns of V (stride ld)
// the eigenvectors (WANT_V = false: eigenvalues only, V not touched).  Each warp rotates
// whole rows / columns of its pairs, lanes striding the other index.  cs, pairs: n + 2
// entries (shared or global memory of this block).
template <typename T, bool WANT_V = true>
__device__ void dev_jacobi(int n, int ld, T *A, T *V, T *cs, int *pairs, int *s_rot, int max_sweeps)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
    if (WANT_V)
        for (int i = warp; i < n; i += nwarps)
            for (int j = lane; j < n; j += 32) V[i * ld + j] = (i == j) ? (T)1 : (T)0;
    __syncthreads();
    if (n < 2) return;
    const int np = (n + 1) & ~1;
    const int half = np / 2;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        if (tid == 0) *s_rot = 0;
        __syncthreads();
        for (int round = 0; round < np - 1; ++round) {
            for (int i = tid; i < half; i += nt) {
                int p, q;
                if (i == 0) {
                    p = round;
                    q = np - 1;
                } else {
                    p = (round + i) % (np - 1);
                    q = (round - i + (np - 1)) % (np - 1);
                }
                if (p > q) {
                    const int t = p;
                    p = q;
                    q = t;
                }
                T c = (T)1, s = (T)0;
                if (q < n && jacobi_rotation(A[p * ld + q], A[p * ld + p], A[q * ld + q], c, s)) *s_rot = 1;
                pairs[2 * i] = p;
                pairs[2 * i + 1] = q;
                cs[2 * i] = c;
                cs[2 * i + 1] = s;
            }
            __syncthreads();
            for (int i = warp; i < half; i += nwarps) {  // rows p, q
                const T s = cs[2 * i + 1];
                if (s == (T)0) continue;
                const T c = cs[2 * i];
                T *Ap = A + pairs[2 * i] * ld, *Aq = A + pairs[2 * i + 1] * ld;
                for (int j = lane; j < n; j += 32) {
                    const T ap = Ap[j], aq = Aq[j];
                    Ap[j] = c * ap - s * aq;
                    Aq[j] = s * ap + c * aq;
                }
            }
            __syncthreads();
            for (int i = warp; i < half; i += nwarps) {  // columns p, q of A and V
                const T s = cs[2 * i + 1];
                if (s == (T)0) continue;
                const T c = cs[2 * i];
                const int p = pairs[2 * i], q = pairs[2 * i + 1];
                for (int j = lane; j < n; j += 32) {
                    T *Aj = A + j * ld;
                    const T ap = Aj[p], aq = Aj[q];
                    Aj[p] = c * ap - s * aq;
                    Aj[q] = s * ap + c * aq;
                    if (WANT_V) {
                        T *Vj = V + j * ld;
                        const T vp = Vj[p], vq = Vj[q];
                        Vj[p] = c * vp - s * vq;
                        Vj[q] = s * vp + c * vq;
                    }
                }
            }
            __syncthreads();
        }
        const int rot = *s_rot;
        __syncthreads();
        if (!rot) break;
    }
}

// Ascending sort of the eigenpairs left by dev_jacobi: w[rank] = A[j][j],
// Vs[:, rank] = V[:, j] (Vs row stride ldo).
template <typename T, typename TO>
__device__ void dev_sort_eig(int n, int ld, const T *A, const T *V, TO *w, TO *Vs, int ldo)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int j = tid; j < n; j += nt) {
        const T lj = A[j * ld + j];
        int rank = 0;
        for (int i = 0; i < n; ++i) {
            const T li = A[i * ld + i];
            if (li < lj || (li == lj && i < j)) ++rank;
        }
        w[rank] = (TO)lj;
        for (int i = 0; i < n; ++i) Vs[i * ldo + rank] = (TO)V[i * ld + j];
    }
    __syncthreads();
}

// Upper Cholesky G = R^T R of the symmetric part of G (n x n, ld ldg) and Rinv = R^-1.
// Returns 1 (in every thread) when a pivot is not positive and finite; Rinv is then I.
__device__ int dev_chol_inv(int n, const double *G, int ldg, double *R, double *Rinv, int *s_flag)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) *s_flag = 0;
    for (int e = tid; e < n * n; e += nt) {
        const int i = e / n, j = e % n;
        R[e] = (j >= i) ? 0.5 * (G[i * ldg + j] + G[j * ldg + i]) : 0.0;
    }
    __syncthreads();
    for (int kk = 0; kk < n; ++kk) {
        if (tid == 0) {
            const double d = R[kk * n + kk];
            double pv = 1.0;
            if (!(d > 0.0) || !isfinite(d)) *s_flag = 1;
            else pv = sqrt(d);
            R[kk * n + kk] = pv;
        }
        __syncthreads();
        const double piv = R[kk * n + kk];
        for (int j = kk + 1 + tid; j < n; j += nt) R[kk * n + j] /= piv;
        __syncthreads();
        const int m = n - kk - 1;
        for (int e = tid; e < m * m; e += nt) {
            const int i = kk + 1 + e / m, j = kk + 1 + e % m;
            if (j >= i) R[i * n + j] -= R[kk * n + i] * R[kk * n + j];
        }
        __syncthreads();
    }
    for (int j = tid; j < n; j += nt) {
        for (int i = n - 1; i >= 0; --i) {
            double s = (i == j) ? 1.0 : 0.0;
            for (int m = i + 1; m <= j; ++m) s -= R[i * n + m] * Rinv[m * n + j];
            Rinv[i * n + j] = (i <= j) ? s / R[i * n + i] : 0.0;
        }
    }
    __syncthreads();
    const int bad = *s_flag;
    if (bad)
        for (int e = tid; e < n * n; e += nt) Rinv[e] = (e / n == e % n) ? 1.0 : 0.0;
    __syncthreads();
    return bad;
}

// In-place upper Cholesky R^T R = A of the symmetric n x n matrix A (row stride ld, both
// triangles on entry; the upper one holds R on exit) when every pivot exceeds tol (A has a
// unit diagonal here, so tol bounds its conditioning); returns false (in every thread) as
// soon as one does not.
template <typename T>
__device__ bool dev_chol_upper(int n, T *A, int ld, T tol, int *s_flag)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) *s_flag = 0;
    __syncthreads();
    for (int kk = 0; kk < n; ++kk) {
        if (tid == 0) {
            const T d = A[kk * ld + kk];
            if (!(d > tol) || !isfinite(d)) *s_flag = 1;
            else A[kk * ld + kk] = sqrt(d);
        }
        __syncthreads();
        if (*s_flag) return false;
        const T piv = A[kk * ld + kk];
        for (int j = kk + 1 + tid; j < n; j += nt) A[kk * ld + j] /= piv;
        __syncthreads();
        const int m = n - kk - 1;
        for (int e = tid; e < m * m; e += nt) {
            const int i = kk + 1 + e / m, j = kk + 1 + e % m;
            if (j >= i) A[i * ld + j] -= A[kk * ld + i] * A[kk * ld + j];
        }
        __syncthreads();
    }
    return true;
}

// Ri = R^-1 for the upper-triangular R (row strides ldr, ldi), one column per thread.
template <typename T>
__device__ void dev_tri_inv_upper(int n, const T *R, int ldr, T *Ri, int ldi)
{
    for (int j = threadIdx.x; j < n; j += blockDim.x)
        for (int i = n - 1; i >= 0; --i) {
            T s = (i == j) ? (T)1 : (T)0;
            if (i < j)
                for (int m = i + 1; m <= j; ++m) s -= R[i * ldr + m] * Ri[m * ldi + j];
            Ri[i * ldi + j] = (i <= j) ? s / R[i * ldr + i] : (T)0;
        }
    __syncthreads();
}

// C (rows x cols, stride ldc) = op(A) op(B) in precision TA, one output per thread step.
// transA: A stored (inner x rows), else (rows x inner); B stored (inner x cols).
template <typename TC, typename TA, typename TB>
__device__ void dev_matmul(int rows, int cols, int inner, const TA *A, int lda, bool transA, const TB *B, int ldb,
                           TC *C, int ldc)
{
    for (int e = threadIdx.x; e < rows * cols; e += blockDim.x) {
        const int i = e / cols, j = e - (e / cols) * cols;
        TC acc = (TC)0;
        if (transA)
            for (int m = 0; m < inner; ++m) acc += (TC)A[m * lda + i] * (TC)B[m * ldb + j];
        else
            for (int m = 0; m < inner; ++m) acc += (TC)A[i * lda + m] * (TC)B[m * ldb + j];
        C[i * ldc + j] = acc;
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------------
// Symmetric eigendecomposition (FP64 Jacobi) of G (n x n, ld ldg): w ascending, Z
// (n x n, stride n) eigenvectors in columns.  A and V live in shared memory for n <= 64.
__global__ void __launch_bounds__(kSmallThreads) k_small_eig(int n, const double *G, int64_t ldg, double *w,
                                                             double *Z, double *work, int in_smem)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_rot;
    __shared__ double cs[kMaxW + 2];
    __shared__ int pairs[kMaxW + 2];
    const int ld = pad_ld(n);
    double *A = in_smem ? reinterpret_cast<double *>(smem_raw) : work;
    double *V = A + n * ld;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int i = e / n, j = e % n;
        A[i * ld + j] = 0.5 * (G[i * ldg + j] + G[j * ldg + i]);
    }
    __syncthreads();
    dev_jacobi<double>(n, ld, A, V, cs, pairs, &s_rot, kMaxSweeps);
    dev_sort_eig<double, double>(n, ld, A, V, w, Z, n);
}

static size_t eig_smem_bytes(int n) { return (size_t)2 * n * pad_ld(n) * sizeof(double); }

size_t small_eig_work_doubles(int n) { return (size_t)2 * n * pad_ld(n) + 8; }

int small_eig(int n, const double *G, int64_t ldg, double *w, double *Z, double *work, cudaStream_t st)
{
    static const bool attr_once = [&]() {
        cudaFuncSetAttribute(k_small_eig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eig_smem_bytes(64));
        return true;
    }();
    (void)attr_once;
    const int in_smem = n <= 64;
    note_launch();
    k_small_eig<<<1, kSmallThreads, in_smem ? eig_smem_bytes(n) : 0, st>>>(n, G, ldg, w, Z, work, in_smem);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

__global__ void __launch_bounds__(kSmallThreads) k_small_chol_inv(int n, const double *G, int64_t ldg, double *Rinv,
                                                                  double *work, int *flag)
{
    __shared__ int s_flag;
    const int bad = dev_chol_inv(n, G, (int)ldg, work, Rinv, &s_flag);
    if (threadIdx.x == 0) *flag = bad;
}

int small_chol_inv(int n, const double *G, int64_t ldg, double *Rinv, double *work, int *flag, cudaStream_t st)
{
    note_launch();
    k_small_chol_inv<<<1, kSmallThreads, 0, st>>>(n, G, ldg, Rinv, work, flag);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

// ---------------------------------------------------------------------------------
// Rayleigh-Ritz on span(S), S = [X W P] with w columns, in an S-orthonormal basis C_S:
//   D = diag(G_S)^-1/2; Cholesky D G_S D = R^T R when every pivot is well above zero,
//   C_S = D R^-1; else SVQB (Stathopoulos & Wu): eig(D G_S D) = U L U^T, keep
//   L_i > tau max L, C_S = D U_keep L_keep^-1/2.  Then eig(C_S^T G_A C_S) = Z theta,
//   coef = C_S Z[:, first k]  (the k smallest; the k largest, descending, if 'largest').
// T is the precision of the two w x w eigensolves.  With T = float a k-dimensional FP64
// refinement follows: Y = C_S Z_k R^-1 (R^T R = Z_k^T Z_k), M = Y^T G_A Y, eig(M) = Q mu
// (FP64), coef = Y Q.  info[0] = kept directions, info[1] = 1 on NaN/Inf or a failed
// refinement.

size_t small_rr_work_doubles(int w) { return (size_t)16 * w * w + 16 * w + 256; }

template <typename T>
__device__ void rr_body(int w, int k, int largest, const double *GS, const double *GA, double tau, double *coef,
                        double *theta, double *work, int *info, T *As, T *Vs, int use_smem)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    __shared__ int s_rot, s_keep, s_first, s_flag;
    __shared__ T csb[kMaxW + 2];
    __shared__ int pairs[kMaxW + 2];
    __shared__ double cs64[kMaxK + 2];
    __shared__ int pairs64[kMaxK + 2];
    const int ld = pad_ld(w);
    // FP64 workspace
    double *dsc = work;                       // w
    double *GAs = dsc + w;                    // w x w, symmetrised G_A
    double *Cs = GAs + w * w;                 // w x w (keep columns used)
    double *Zk = Cs + w * w;                  // w x k
    double *ZR = Zk + w * k;                  // w x k
    double *Y = ZR + w * k;                   // w x k
    double *Bm = Y + w * k;                   // w x k
    double *M = Bm + w * k;                   // k x k
    double *R = M + k * k;                    // k x k
    double *Ri = R + k * k;                   // k x k
    double *Q = Ri + k * k;                   // k x k
    double *mu = Q + k * k;                   // k
    T *lam = reinterpret_cast<T *>(mu + k);   // w
    T *GAt = lam + w + 2;                     // w x w
    T *Cst = GAt + w * w;                     // w x w
    T *U = Cst + w * w;                       // w x w
    T *T2 = U + w * w;                        // w x w
    T *Z = T2 + w * w;                        // w x w
    T *Ag = reinterpret_cast<T *>(((uintptr_t)(Z + w * w) + 15) & ~(uintptr_t)15);
    T *A = use_smem ? As : Ag;
    T *V = use_smem ? Vs : Ag + w * ld;

    for (int i = tid; i < w; i += nt) {
        const double d = GS[i * w + i];
        dsc[i] = (d > 0.0 && isfinite(d)) ? 1.0 / sqrt(d) : 0.0;
    }
    __syncthreads();
    for (int e = tid; e < w * w; e += nt) {
        const int i = e / w, j = e - (e / w) * w;
        const double g = 0.5 * (GA[i * w + j] + GA[j * w + i]);
        GAs[e] = g;
        GAt[e] = (T)g;
        A[i * ld + j] = (T)(dsc[i] * 0.5 * (GS[i * w + j] + GS[j * w + i]) * dsc[j]);
    }
    __syncthreads();
    // An S-orthonormal basis: from the Cholesky factor of D G_S D when that is well
    // conditioned (every pivot of the unit-diagonal matrix above chol_tol), C_S = D R^-1,
    // all w directions kept; otherwise SVQB, which drops the nearly dependent directions.
    const T chol_tol = sizeof(T) == sizeof(float) ? (T)1e-3 : (T)1e-8;
    // the factor and its inverse in shared memory when the w x w tiles are there (V is free
    // until the SVQB fallback sets it, A until the projection overwrites it): the column
    // loops of both are latency chains
    T *Rm = use_smem ? V : T2, *Ui = use_smem ? A : U;
    const int ldr = use_smem ? ld : w;
    for (int e = tid; e < w * w; e += nt) Rm[(e / w) * ldr + (e % w)] = A[(e / w) * ld + (e % w)];
    const bool chol = dev_chol_upper<T>(w, Rm, ldr, chol_tol, &s_flag);
    if (chol) {
        dev_tri_inv_upper<T>(w, Rm, ldr, Ui, ldr);
        for (int e = tid; e < w * w; e += nt) {
            const int i = e / w, j = e - i * w;
            const double c = dsc[i] * (double)Ui[i * ldr + j];
            Cs[e] = c;
            Cst[e] = (T)c;
        }
        if (tid == 0) {
            s_first = 0;
            s_keep = w;
        }
        __syncthreads();
    } else {
        dev_jacobi<T>(w, ld, A, V, csb, pairs, &s_rot, kMaxSweeps);
        dev_sort_eig<T, T>(w, ld, A, V, lam, U, w);
        if (tid == 0) {
            const double lmax = (double)lam[w - 1];
            int first = w;
            for (int i = 0; i < w; ++i)
                if ((double)lam[i] > tau * lmax) {
                    first = i;
                    break;
                }
            s_first = first;
            s_keep = w - first;
        }
        __syncthreads();
        const int first = s_first, keep = s_keep;
        for (int e = tid; e < w * keep; e += nt) {
            const int i = e / keep, j = e - (e / keep) * keep;
            const double c = dsc[i] * (double)U[i * w + first + j] / sqrt((double)lam[first + j]);
            Cs[i * w + j] = c;
            Cst[i * w + j] = (T)c;
        }
        __syncthreads();
    }
    const int keep = s_keep;
    // projected G_A in precision T: T2 = G_A Cs, A = Cs^T T2 (keep x keep, stride ldk)
    const int ldk = pad_ld(keep);
    dev_matmul<T, T, T>(w, keep, w, GAt, w, false, Cst, w, T2, w);
    dev_matmul<T, T, T>(keep, keep, w, Cst, w, true, T2, w, A, ldk);
    for (int e = tid; e < keep * keep; e += nt) {
        const int i = e / keep, j = e - (e / keep) * keep;
        if (i < j) {
            const T a = (T)0.5 * (A[i * ldk + j] + A[j * ldk + i]);
            A[i * ldk + j] = a;
            A[j * ldk + i] = a;
        }
    }
    __syncthreads();
    dev_jacobi<T>(keep, ldk, A, V, csb, pairs, &s_rot, kMaxSweeps);
    dev_sort_eig<T, T>(keep, ldk, A, V, lam, Z, keep);
    const int kk = k < keep ? k : keep;
    if (sizeof(T) == sizeof(double)) {
        for (int e = tid; e < w * k; e += nt) {
            const int i = e / k, j = e - (e / k) * k;
            double s = 0.0;
            if (j < kk) {
                const int col = largest ? keep - 1 - j : j;
                for (int m = 0; m < keep; ++m) s += Cs[i * w + m] * (double)Z[m * keep + col];
            }
            coef[e] = s;
        }
        for (int j = tid; j < k; j += nt) theta[j] = j < kk ? (double)lam[largest ? keep - 1 - j : j] : 0.0;
        if (tid == 0) {
            info[0] = keep;
            int bad = 0;
            for (int j = 0; j < kk; ++j)
                if (!isfinite((double)lam[j])) bad = 1;
            info[1] = bad;
        }
        return;
    }
    // FP64 refinement of the k-dimensional Ritz subspace
    for (int e = tid; e < keep * kk; e += nt) {
        const int i = e / kk, j = e - (e / kk) * kk;
        Zk[e] = (double)Z[i * keep + (largest ? keep - 1 - j : j)];
    }
    __syncthreads();
    dev_matmul<double, double, double>(kk, kk, keep, Zk, kk, true, Zk, kk, M, kk);
    const int bad_chol = dev_chol_inv(kk, M, kk, R, Ri, &s_flag);
    dev_matmul<double, double, double>(keep, kk, kk, Zk, kk, false, Ri, kk, ZR, kk);
    dev_matmul<double, double, double>(w, kk, keep, Cs, w, false, ZR, kk, Y, kk);
    dev_matmul<double, double, double>(w, kk, w, GAs, w, false, Y, kk, Bm, kk);
    // the k x k projection reuses the shared region (the w x w solves are done)
    const int ldkk = pad_ld(kk);
    const bool ref_smem = use_smem && (size_t)2 * kk * ldkk * sizeof(double) <= (size_t)2 * w * ld * sizeof(T);
    double *A64 = ref_smem ? reinterpret_cast<double *>(As) : reinterpret_cast<double *>(Ag);
    double *V64 = A64 + kk * ldkk;
    dev_matmul<double, double, double>(kk, kk, w, Y, kk, true, Bm, kk, A64, ldkk);
    for (int e = tid; e < kk * kk; e += nt) {
        const int i = e / kk, j = e - (e / kk) * kk;
        if (i < j) {
            const double a = 0.5 * (A64[i * ldkk + j] + A64[j * ldkk + i]);
            A64[i * ldkk + j] = a;
            A64[j * ldkk + i] = a;
        }
    }
    __syncthreads();
    dev_jacobi<double>(kk, ldkk, A64, V64, cs64, pairs64, &s_rot, kMaxSweeps);
    dev_sort_eig<double, double>(kk, ldkk, A64, V64, mu, Q, kk);
    for (int e = tid; e < w * k; e += nt) {  // coef = Y Q (descending for 'largest')
        const int i = e / k, j = e - (e / k) * k;
        double s = 0.0;
        if (j < kk) {
            const int col = largest ? kk - 1 - j : j;
            for (int m = 0; m < kk; ++m) s += Y[i * kk + m] * Q[m * kk + col];
        }
        coef[e] = s;
    }
    for (int j = tid; j < k; j += nt) theta[j] = j < kk ? mu[largest ? kk - 1 - j : j] : 0.0;
    if (tid == 0) {
        info[0] = keep;
        int bad = bad_chol;
        for (int j = 0; j < kk; ++j)
            if (!isfinite(mu[j])) bad = 1;
        info[1] = bad;
    }
}

template <typename T>
__global__ void __launch_bounds__(kSmallThreads) k_small_rr(int w, int k, int largest, const double *GS,
                                                            const double *GA, double tau, double *coef,
                                                            double *theta, double *work, int *info, int use_smem)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *As = reinterpret_cast<T *>(smem_raw);
    T *Vs = As + w * pad_ld(w);
    rr_body<T>(w, k, largest, GS, GA, tau, coef, theta, work, info, As, Vs, use_smem);
}

int small_svqb_rr(int w, int k, int largest, int mixed, const double *GS, const double *GA, double tau,
                  double *coef, double *theta, double *work, int *info, cudaStream_t st)
{
    const int cap = 160 * 1024;
    static const bool attr_once = [&]() {
        cudaFuncSetAttribute(k_small_rr<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
        cudaFuncSetAttribute(k_small_rr<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap);
        return true;
    }();
    (void)attr_once;
    const size_t es = mixed ? sizeof(float) : sizeof(double);
    const size_t sm = 2 * (size_t)w * pad_ld(w) * es;
    const int use_smem = sm <= (size_t)cap;
    note_launch();
    if (mixed)
        k_small_rr<float><<<1, kSmallThreads, use_smem ? sm : 0, st>>>(w, k, largest, GS, GA, tau, coef, theta,
                                                                       work, info, use_smem);
    else
        k_small_rr<double><<<1, kSmallThreads, use_smem ? sm : 0, st>>>(w, k, largest, GS, GA, tau, coef, theta,
                                                                        work, info, use_smem);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

// ---------------------------------------------------------------------------------
// Rayleigh-Ritz with H on span(X) for the convergence test and the final extraction.
// In: mu, V = eig(M), M = X^T (H - sigma) X; EtE = E^T E, E = (H - sigma)X - X M.
// Residual of pair j: sqrt(v_j^T EtE v_j).  Selects the nev values of mu nearest 0
// (ties: lower first), writes sel (ascending mu), res_sel, st[0] = converged,
// st[1] = NaN/Inf seen, dst[0] = max relative residual of the selection.
// res_all[j] = sqrt(v_j^T sym(EtE) v_j), one block per column j: thread a forms
// (sym(EtE) v_j)_a, the block sums v_j[a] times it in a fixed shape (warp shuffles, then
// the warps in order).
__global__ void __launch_bounds__(64) k_hrr_resid(int k, const double *V, const double *EtE, double *res_all)
{
    __shared__ double s_w[2];
    const int j = blockIdx.x, a = threadIdx.x;
    double s = 0.0;
    if (a < k) {
        double t = 0.0;
        for (int b = 0; b < k; ++b) t += 0.5 * (EtE[a * k + b] + EtE[b * k + a]) * V[b * k + j];
        s = V[a * k + j] * t;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((a & 31) == 0) s_w[a >> 5] = s;
    __syncthreads();
    if (a == 0) res_all[j] = sqrt(fmax(s_w[0] + s_w[1], 0.0));
}

// The nev Ritz values nearest 0 (|mu| ascending, ties: lower mu, then lower index), in
// ascending index order: thread j ranks its own value against all k, and the chosen
// ones are compacted by ballot.
__global__ void __launch_bounds__(64) k_hrr_pick(int k, int nev, const double *mu, const double *res_all,
                                                 double tol_abs, double norm_h, int *sel, double *res_sel, int *st,
                                                 double *dst)
{
    __shared__ unsigned s_ball[2];
    __shared__ int s_conv[2], s_bad[2];
    __shared__ double s_mx[2];
    const int j = threadIdx.x, lane = j & 31, w = j >> 5;
    bool pick = false;
    if (j < k) {
        const double mj = mu[j], aj = fabs(mj);
        int rank = 0;
        for (int i = 0; i < k; ++i) {
            const double mi = mu[i], ai = fabs(mi);
            if (ai < aj || (ai == aj && (mi < mj || (mi == mj && i < j)))) ++rank;
        }
        pick = rank < nev;
    }
    const unsigned ball = __ballot_sync(0xffffffffu, pick);
    if (lane == 0) s_ball[w] = ball;
    __syncthreads();
    int conv = 1, bad = 0;
    double mx = 0.0;
    if (pick) {
        const int pos = __popc(ball & ((1u << lane) - 1u)) + (w ? __popc(s_ball[0]) : 0);
        const double r = res_all[j];
        sel[pos] = j;
        res_sel[pos] = r;
        if (!isfinite(r) || !isfinite(mu[j])) bad = 1;
        if (!(r <= tol_abs)) conv = 0;
        mx = r / norm_h;
    }
    conv = __all_sync(0xffffffffu, conv);
    bad = __any_sync(0xffffffffu, bad);
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (lane == 0) {
        s_conv[w] = conv;
        s_bad[w] = bad;
        s_mx[w] = mx;
    }
    __syncthreads();
    if (j == 0) {
        st[0] = s_conv[0] && s_conv[1];
        st[1] = s_bad[0] || s_bad[1];
        dst[0] = fmax(s_mx[0], s_mx[1]);
    }
}

int hrr_select(int k, int nev, const double *mu, const double *V, const double *EtE, double tol_abs, double norm_h,
               double *res_all, int *sel, double *res_sel, int *st, double *dst, cudaStream_t s)
{
    note_launch();
    k_hrr_resid<<<k, 64, 0, s>>>(k, V, EtE, res_all);
    note_launch();
    k_hrr_pick<<<1, 64, 0, s>>>(k, nev, mu, res_all, tol_abs, norm_h, sel, res_sel, st, dst);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

// Csel (k x nev) = V[:, sel]
__global__ void k_gather_cols(int k, int nev, const double *V, const int *sel, double *Csel)
{
    for (int e = threadIdx.x; e < k * nev; e += blockDim.x) {
        const int i = e / nev, j = e % nev;
        Csel[e] = V[i * k + sel[j]];
    }
}

int gather_cols(int k, int nev, const double *V, const int *sel, double *Csel, cudaStream_t st)
{
    note_launch();
    k_gather_cols<<<1, 256, 0, st>>>(k, nev, V, sel, Csel);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

// ---------------------------------------------------------------------------------
// Half-chain entanglement entropy (Sec. 2.2) of sector vectors.  Cut after the first la
// sites.  With p up spins on the left, a vector's entries form the R x T matrix
// M_p[i][c] = v[off_c + i]: i the colex rank of the left pattern among those with p ones,
// c the colex rank of the right pattern among those with n_up - p ones, off_c the row of
// the first state with that right pattern (the left p spins lowest).  The reduced density
// matrix of the left block is the direct sum of the M_p M_p^T.  For each (vector, p):
//   k_ent_gather   M_p, dense, with the index of the smaller Gram innermost;
//   k_ent_gram     the smaller Gram (M M^T or M^T M, the same nonzero eigenvalues), in
//                  tiles of 32 x 32 over all SMs;
//   k_ent_tridiag  Householder reduction to tridiagonal form by a cluster of four blocks;
//   k_ent_eig      its eigenvalues by bisection on Sturm counts, one lane each, and the
//                  sum of lambda ln lambda;
// and k_ent_combine forms S = ln N - (sum lambda ln lambda) / N with N = sum lambda, the
// trace of the Grams, so v need not be normalised.  Every sum has a fixed order.  Eigenvalues
// are absolute to 2^-60 of the trace (their share of S to 1e-14).  Cuts of small Grams take
// k_ent_block instead (ent_one_block).
//
// All of it is bound by the FP64 pipe (two FMA a cycle and SM on GB300).  At L = 20,
// l_a = 10, 16 vectors, the one-block FP64 Jacobi in L2 (k_ent_block) took 590 ms,
// about 20 sweeps of n^3 rotations; the reduction needs n^3 FMA once, spread over four SMs
// a matrix (6.7 ms the whole call).

constexpr int kEntCluster = 4;    // blocks per matrix in the reduction
constexpr int kEntThreads = 256;  // threads of the gather, Gram and reduction blocks
constexpr int kEntTile = 32;      // Gram tile edge
constexpr int kEntSmem = 224 * 1024;  // rows of the reduction kept in shared memory up to this

// The cut's values of p that occur, largest Gram first.
struct EntCut {
    int L, n_up, la, np, job0;  // job0: the first (vector, p) of this launch
    int p[kMaxL + 1];
    int64_t block_doubles, mmax, dmax;
};

// One (vector, p): its sizes and its part of the workspace.
struct EntJob {
    int vec, p, R, T, d, t, ld;  // d: Gram side, t: the other side
    bool left;                   // d = R: Gram over the left patterns
    // off2[d]: the exponent ex, diag and off2 being those of the matrix over 2^ex
    double *M, *A, *diag, *off2, *sums;
};

__device__ __forceinline__ EntJob ent_job(const EntCut &cut, int nvec, int job, double *work)
{
    EntJob j;
    const int q = job / nvec;
    j.vec = job % nvec;
    j.p = cut.p[q];
    j.R = (int)__ldg(&g_binom.v[cut.la * kBinomDim + j.p]);
    j.T = (int)__ldg(&g_binom.v[(cut.L - cut.la) * kBinomDim + cut.n_up - j.p]);
    j.left = j.R <= j.T;
    j.d = j.left ? j.R : j.T;
    j.t = j.left ? j.T : j.R;
    j.ld = pad_ld(j.d);
    j.M = work + (int64_t)job * cut.block_doubles;
    j.A = j.M + cut.mmax;
    j.diag = j.A + cut.dmax * (int64_t)pad_ld((int)cut.dmax);
    j.off2 = j.diag + cut.dmax + 2;
    j.sums = j.off2 + cut.dmax + 2;  // [0] the trace, [1 + g] lambda ln lambda of 32 eigenvalues
    return j;
}

EntanglementPlan entanglement_plan(int L, int n_up, int la)
{
    EntanglementPlan pl{};
    const int lb = L - la;
    for (int p = 0; p <= la; ++p) {
        const int q = n_up - p;
        if (q < 0 || q > lb) continue;
        const int64_t R = host_binom(la, p), T = host_binom(lb, q);
        const int64_t d = R < T ? R : T;
        if (d > pl.dmax) pl.dmax = d;
        if (T > pl.tmax) pl.tmax = T;
        if (R * T > pl.mmax) pl.mmax = R * T;
    }
    // M (mmax), A (dmax x pad_ld(dmax)), the tridiagonal (2 (dmax + 2)), the sums (1 + dmax / 32)
    pl.block_doubles = pl.mmax + pl.dmax * (int64_t)pad_ld((int)pl.dmax) + 2 * (pl.dmax + 2) + pl.tmax + 8;
    pl.blocks_per_vector = la + 1;
    return pl;
}

// M[s][g]: g the Gram index (innermost), s the summed index.
__global__ void __launch_bounds__(kEntThreads) k_ent_gather(EntCut cut, int nvec, const double *__restrict__ V,
                                                            int64_t ldv, double *work)
{
    __shared__ uint32_t sb[kBinomDim * kBinomDim];
    load_binom(sb);
    __syncthreads();
    const EntJob j = ent_job(cut, nvec, cut.job0 + (int)blockIdx.y, work);
    const int lb = cut.L - cut.la, q = cut.n_up - j.p;
    const double *v = V + j.vec;
    // a thread per right pattern c and a run of left patterns: the unranking is done once
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = gridDim.x * (kEntThreads / 32);
    for (int c = blockIdx.x * (kEntThreads / 32) + warp; c < j.T; c += nwarps) {
        const uint32_t b = cns_unrank(sb, lb, q, (uint32_t)c);
        const uint32_t off = cns_rank(sb, (b << cut.la) | ((1u << j.p) - 1u));
        for (int i = lane; i < j.R; i += 32)
            j.M[j.left ? (int64_t)c * j.R + i : (int64_t)i * j.T + c] = v[((int64_t)off + i) * ldv];
    }
}

// One 32 x 32 tile (and its mirror image) of a Gram per block, 2 x 2 outputs a thread.
__global__ void __launch_bounds__(kEntThreads) k_ent_gram(EntCut cut, int nvec, double *work)
{
    constexpr int TS = kEntTile, KS = 16;
    __shared__ double sa[KS][TS], sc[KS][TS];
    const EntJob j = ent_job(cut, nvec, cut.job0 + (int)blockIdx.y, work);
    const int d = j.d, nt = (d + TS - 1) / TS;
    if ((int)blockIdx.x >= nt * (nt + 1) / 2) return;
    int bi = 0, rem = blockIdx.x;  // tile (bi, bj), bj >= bi
    while (rem >= nt - bi) rem -= nt - bi++;
    const int i0 = bi * TS, j0 = (bi + rem) * TS;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[2][2] = {};
    for (int s0 = 0; s0 < j.t; s0 += KS) {
        for (int e = threadIdx.x; e < KS * TS; e += kEntThreads) {
            const int s = e / TS, g = e % TS;
            const double *row = j.M + (int64_t)(s0 + s) * d;
            sa[s][g] = (s0 + s < j.t && i0 + g < d) ? row[i0 + g] : 0.0;
            sc[s][g] = (s0 + s < j.t && j0 + g < d) ? row[j0 + g] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            const double a0 = sa[s][ty], a1 = sa[s][ty + 16], c0 = sc[s][tx], c1 = sc[s][tx + 16];
            acc[0][0] += a0 * c0;
            acc[0][1] += a0 * c1;
            acc[1][0] += a1 * c0;
            acc[1][1] += a1 * c1;
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int gi = i0 + ty + 16 * a, gj = j0 + tx + 16 * c;
            if (gi < d && gj < d && gj >= gi) {
                j.A[(int64_t)gi * j.ld + gj] = acc[a][c];
                j.A[(int64_t)gj * j.ld + gi] = acc[a][c];
            }
        }
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The shared-memory address that holds `p` in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

__device__ __forceinline__ double cluster_ld(uint32_t addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void cluster_st(uint32_t addr, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

__device__ __forceinline__ double warp_sum(double x)
{
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

// Householder reduction of A to tridiagonal form: step k takes x = row k beyond the diagonal,
// v = x - alpha e_1 with alpha = -sign(x_1) ||x||, y = A v, and A -= v w^T + w v^T with
// w = b y - (b^2 (v.y) / 2) v, b = 2 / v.v.  Row i lives in block i mod 4 of the cluster,
// column-major (thread = row, so a column's rows are read side by side), in shared memory
// while a block's rows fit there, else in the workspace.  Per step two cluster barriers: y
// is spread to all blocks, and the next row is read once every row is updated.  The matrix is
// scaled by the power of two above its trace; an x whose norm beyond x_1 is below 2^-100 of
// that is taken as zero (squares of a graded matrix' smallest parts would underflow).
__global__ void __cluster_dims__(kEntCluster, 1, 1) __launch_bounds__(kEntThreads)
    k_ent_tridiag(EntCut cut, int nvec, double *work, int in_smem)
{
    extern __shared__ __align__(16) double ent_raw[];
    __shared__ double s_b, s_c, s_part[kEntThreads];
    const int rank = blockIdx.x % kEntCluster;
    const EntJob j = ent_job(cut, nvec, cut.job0 + (int)(blockIdx.x / kEntCluster), work);
    const int d = j.d, nr = (d + kEntCluster - 1) / kEntCluster, dmax = (int)cut.dmax;
    double *v = ent_raw, *w = v + dmax, *y = w + dmax, *rows = y + dmax;
    // element (own row li, column c) at At[li * si + c * sc]
    double *At = in_smem ? rows : j.A + rank;
    const int64_t si = in_smem ? 1 : kEntCluster, sc = in_smem ? nr : j.ld;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp == 0) {
        double tr = 0.0;
        for (int i = lane; i < d; i += 32) tr += j.A[(int64_t)i * j.ld + i];
        tr = warp_sum(tr);
        if (lane == 0) s_b = (tr > 0.0 && isfinite(tr)) ? (double)(ilogb(tr) + 1) : 0.0;
    }
    __syncthreads();
    const int ex = (int)s_b;
    if (rank == 0 && tid == 0) j.off2[d] = s_b;
    cluster_barrier();  // every block has read the diagonal
    for (int e = tid; e < nr * d; e += kEntThreads) {
        const int c = e / nr, li = e - c * nr, i = rank + kEntCluster * li;
        if (i < d) At[li * si + c * sc] = scalbn(j.A[(int64_t)c * j.ld + i], -ex);
    }
    cluster_barrier();
    // thread = (row group of 32, column segment): rows tid % 32 + 32 * g, segment warp
    constexpr int SEG = kEntThreads / 32;
    for (int k = 0; k < d; ++k) {
        const int owner = k % kEntCluster, lk = k / kEntCluster;
        // row k of the reduced matrix, from its owner
        for (int c = k + tid; c < d; c += kEntThreads) {
            const double x = in_smem ? cluster_ld(cluster_addr(rows + (int64_t)c * nr + lk, owner))
                                     : __ldcg(j.A + (int64_t)c * j.ld + k);
            v[c] = x;
        }
        __syncthreads();
        if (rank == 0 && tid == 0) j.diag[k] = v[k];
        const int m = d - 1 - k;  // order of the trailing matrix
        if (m == 0) break;
        if (m == 1) {
            if (rank == 0 && tid == 0) j.off2[k] = v[k + 1] * v[k + 1];
        } else {
            if (warp == 0) {
                double s = 0.0;
                for (int c = k + 2 + lane; c < d; c += 32) s += v[c] * v[c];
                s = warp_sum(s);
                if (lane == 0) {
                    const double x1 = v[k + 1];
                    double b = 0.0, n2 = x1 * x1;
                    if (s > 0x1p-200) {
                        n2 += s;
                        const double v1 = x1 + copysign(sqrt(n2), x1);
                        b = 2.0 / (s + v1 * v1);
                        v[k + 1] = v1;
                    }
                    s_b = b;
                    if (rank == 0) j.off2[k] = n2;
                }
            }
            __syncthreads();
            const double b = s_b;
            if (b != 0.0) {  // the same in all blocks
                // y = A v over own rows, SEG column segments
                const int first = k + 1;
                for (int g = 0; g < nr; g += 32) {
                    const int li = g + lane;
                    if (rank + kEntCluster * (g + 31) <= k) continue;  // a group of finished rows
                    double acc = 0.0;
                    if (li < nr)
                        for (int c = first + warp; c < d; c += SEG) acc += At[li * si + c * sc] * v[c];
                    s_part[tid] = acc;
                    __syncthreads();
                    if (warp == 0 && li < nr && rank + kEntCluster * li < d) {
                        double t = 0.0;
#pragma unroll
                        for (int q = 0; q < SEG; ++q) t += s_part[32 * q + lane];
                        const int i = rank + kEntCluster * li;
                        for (int r = 0; r < kEntCluster; ++r) cluster_st(cluster_addr(y + i, r), t);
                    }
                    __syncthreads();
                }
                cluster_barrier();
                if (warp == 0) {
                    double s = 0.0;
                    for (int c = first + lane; c < d; c += 32) s += v[c] * y[c];
                    s = warp_sum(s);
                    if (lane == 0) s_c = 0.5 * b * s;
                }
                __syncthreads();
                const double h = s_c;
                for (int c = first + tid; c < d; c += kEntThreads) w[c] = b * (y[c] - h * v[c]);
                __syncthreads();
                for (int g = 0; g < nr; g += 32) {
                    const int li = g + lane, i = rank + kEntCluster * li;
                    if (i > k && i < d) {
                        const double vi = v[i], wi = w[i];
                        for (int c = first + warp; c < d; c += SEG) {
                            double *a = At + li * si + c * sc;
                            *a = fma(-wi, v[c], fma(-vi, w[c], *a));
                        }
                    }
                }
            }
        }
        cluster_barrier();
    }
    cluster_barrier();  // no block leaves while another may read its rows
}

// Number of eigenvalues of T below x: sign changes of p_i = (a_i - x) p_{i-1} - b_{i-1}^2
// p_{i-2}.  Three FP64 operations a step and no division; the exponents are brought back by
// integer operations after each step, and an exact zero stands for -2^-60 p_{i-1} (a_i moved
// by 2^-60 of the matrix' scale).  ab[i] = (a_i, b_{i-1}^2).
__device__ __forceinline__ int sturm_count(const double2 *ab, int d, double x)
{
    double p0 = 0.0, p1 = 1.0;
    int cnt = 0;
    for (int i = 0; i < d; ++i) {
        const double2 q = ab[i];
        const double pn = fma(q.x - x, p1, -(q.y * p0));
        int h = __double2hiint(pn), lo = __double2loint(pn);
        const int h1 = __double2hiint(p1);
        if ((((unsigned)h & 0x7ff00000u) == 0u)) {  // zero (or subnormal): see above
            h = (int)(((unsigned)h1 ^ 0x80000000u) - (60u << 20));
            lo = 0;
        }
        cnt += (int)(((unsigned)(h ^ h1)) >> 31);
        const int e = (int)(((unsigned)h >> 20) & 0x7ffu) - 1023;  // p_{i-1} has exponent 0
        p0 = __hiloint2double(h1 - (int)((unsigned)e << 20), __double2loint(p1));
        p1 = __hiloint2double(h - (int)((unsigned)e << 20), lo);
    }
    return cnt;
}

// Eigenvalues 32 g .. 32 g + 31 of one matrix by one warp: bisection to 2^-60 of its scale.
// A warp alone on its quarter of an SM has the whole of that quarter's FP64 pipe.
__global__ void __launch_bounds__(32) k_ent_eig(EntCut cut, int nvec, double *work)
{
    extern __shared__ __align__(16) double2 ent_ab[];
    const EntJob j = ent_job(cut, nvec, cut.job0 + (int)blockIdx.y, work);
    const int d = j.d, lane = threadIdx.x, idx = blockIdx.x * 32 + lane;
    if ((int)blockIdx.x * 32 >= d) return;
    const int ex = (int)j.off2[d];
    double tr = 0.0;
    for (int i = lane; i < d; i += 32) tr += j.diag[i];
    tr = warp_sum(tr);
    double sum = 0.0;
    if (!(tr > 0.0) || !isfinite(tr)) {
        sum = tr == 0.0 ? 0.0 : NAN;
        if (tr < 0.0) tr = NAN;
    } else {
        // scaled by the power of two above the trace: all eigenvalues in [0, 1], up to rounding
        for (int i = lane; i < d; i += 32) ent_ab[i] = make_double2(j.diag[i], i > 0 ? j.off2[i - 1] : 0.0);
        __syncwarp();
        double lo = -0x1p-40, hi = 1.0 + 0x1p-40;
        for (int it = 0; it < 64; ++it) {
            const double mid = 0.5 * (lo + hi);
            const bool open = hi - lo > 0x1p-60 && mid > lo && mid < hi;
            if (!__any_sync(0xffffffffu, open)) break;
            const int c = sturm_count(ent_ab, d, mid);
            if (open) {
                if (c > idx) hi = mid;
                else lo = mid;
            }
        }
        const double lam = scalbn(0.5 * (lo + hi), ex);
        if (idx < d && lam > 0.0) sum = lam * log(lam);
    }
    sum = warp_sum(sum);
    if (lane == 0) {
        j.sums[1 + blockIdx.x] = sum;
        if (blockIdx.x == 0) j.sums[0] = scalbn(tr, ex);
    }
}

__global__ void k_ent_combine(EntCut cut, int nvec, double *work, double *S)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nvec) return;
    double n2 = 0.0, a1 = 0.0;
    for (int q = 0; q < cut.np; ++q) {
        const EntJob j = ent_job(cut, nvec, q * nvec + e, work);
        n2 += j.sums[0];
        for (int g = 0; 32 * g < j.d; ++g) a1 += j.sums[1 + g];
    }
    S[e] = n2 > 0.0 ? log(n2) - a1 / n2 : NAN;
}

// The whole of one (vector, p) in one block, and the sums over p: for cuts whose Grams are small
// or long sums.
__global__ void __launch_bounds__(kSmallThreads)
    k_ent_block(int L, int n_up, int la, const double *__restrict__ V, int64_t ldv, double *work,
                int64_t block_doubles, int64_t mmax, int64_t dmax, double *parts)
{
    __shared__ uint32_t sb[kBinomDim * kBinomDim];
    __shared__ int s_rot;
    __shared__ double s_r0[kSmallThreads / 32], s_r1[kSmallThreads / 32];
    load_binom(sb);
    __syncthreads();
    const int e = blockIdx.x / (la + 1), p = blockIdx.x % (la + 1);
    const int lb = L - la, q = n_up - p;
    double *out = parts + 2 * (int64_t)blockIdx.x;
    if (q < 0 || q > lb) {  // no state has p up spins on the left
        if (threadIdx.x == 0) {
            out[0] = 0.0;
            out[1] = 0.0;
        }
        return;
    }
    const int R = (int)binom(sb, la, p), T = (int)binom(sb, lb, q);
    const bool left = R <= T;  // Gram over the left patterns (d = R), else over the right ones
    const int d = left ? R : T, ld = pad_ld(d);
    double *M = work + (int64_t)blockIdx.x * block_doubles;  // R x T, row-major
    double *A = M + mmax;
    double *cs = A + dmax * (int64_t)pad_ld((int)dmax);
    int *pairs = reinterpret_cast<int *>(cs + dmax + 2);
    uint32_t *off = reinterpret_cast<uint32_t *>(cs + 2 * (dmax + 2));
    for (int c = threadIdx.x; c < T; c += blockDim.x) {
        const uint32_t b = cns_unrank(sb, lb, q, (uint32_t)c);
        off[c] = cns_rank(sb, (b << la) | ((1u << p) - 1u));
    }
    __syncthreads();
    const double *v = V + e;
    for (int64_t x = threadIdx.x; x < (int64_t)R * T; x += blockDim.x) {
        const int i = (int)(x % R), c = (int)(x / R);  // consecutive threads: consecutive rows of a tile
        M[(int64_t)i * T + c] = v[((int64_t)off[c] + i) * ldv];
    }
    __syncthreads();
    for (int64_t x = threadIdx.x; x < (int64_t)d * d; x += blockDim.x) {
        const int i = (int)(x / d), j = (int)(x % d);
        if (j < i) continue;
        double acc = 0.0;
        if (left) {
            const double *mi = M + (int64_t)i * T, *mj = M + (int64_t)j * T;
            for (int c = 0; c < T; ++c) acc += mi[c] * mj[c];
        } else {
            for (int r = 0; r < R; ++r) acc += M[(int64_t)r * T + i] * M[(int64_t)r * T + j];
        }
        A[(int64_t)i * ld + j] = acc;
        A[(int64_t)j * ld + i] = acc;
    }
    __syncthreads();
    dev_jacobi<double, false>(d, ld, A, nullptr, cs, pairs, &s_rot, kMaxSweeps);
    double s0 = 0.0, s1 = 0.0;
    for (int i = threadIdx.x; i < d; i += blockDim.x) {
        const double lam = A[(int64_t)i * ld + i];
        if (!(lam <= 0.0)) {  // NaN too: an entry that is not finite makes S NaN
            s0 += lam;
            s1 += lam * log(lam);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        s_r0[threadIdx.x >> 5] = s0;
        s_r1[threadIdx.x >> 5] = s1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a0 = 0.0, a1 = 0.0;
        for (int w = 0; w < kSmallThreads / 32; ++w) {
            a0 += s_r0[w];
            a1 += s_r1[w];
        }
        out[0] = a0;
        out[1] = a1;
    }
}

__global__ void k_ent_block_combine(int nvec, int per, const double *parts, double *S)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nvec) return;
    double n2 = 0.0, a1 = 0.0;
    for (int p = 0; p < per; ++p) {
        n2 += parts[2 * ((int64_t)e * per + p)];
        a1 += parts[2 * ((int64_t)e * per + p) + 1];
    }
    S[e] = n2 > 0.0 ? log(n2) - a1 / n2 : NAN;
}

// Whether a cut takes k_ent_block: Grams of side 4 and less, or 6 for few vectors, whose four
// kernels are all launches, and those with sums over more than d^3 / 4 entries, which k_ent_gram
// forms for the whole of a 32 x 32 tile.  us, k_ent_block / the kernels above: d = 4, t = 15, 16
// vectors 62 / 95;  d = 6, t = 20, 1 vector 95 / 116, 200 vectors 225 / 200;  16 vectors, d = 6,
// t = 210 128 / 177;  d = 10, t = 126 241 / 197, t = 462 250 / 297, t = 6435 485 / 2106;  d = 20,
// t = 924 723 / 565, t = 3432 728 / 1318;  d = 35, t = 1716 2608 / 1352.
static bool ent_one_block(int L, int n_up, int la, int nvec, int64_t d)
{
    int64_t t = 0;
    for (int p = std::max(0, n_up - (L - la)); p <= std::min(la, n_up); ++p)
        t = std::max<int64_t>(t, std::max(host_binom(la, p), host_binom(L - la, n_up - p)));
    return d <= 4 || (d <= 6 && nvec <= 8) || 4 * t > d * d * d;
}

int entanglement_launch(int L, int n_up, int la, int nvec, const double *V, int64_t ldv, double *S, void *work,
                        size_t work_bytes, cudaStream_t st)
{
    const EntanglementPlan pl = entanglement_plan(L, n_up, la);
    const size_t need = entanglement_work_bytes(pl, nvec);
    if (work_bytes < need) return MBL_ERR_WORKSPACE;
    double *w = (double *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
    if (ent_one_block(L, n_up, la, nvec, pl.dmax)) {
        const int64_t nblk = (int64_t)nvec * pl.blocks_per_vector;
        double *parts = w + nblk * pl.block_doubles;
        note_launch();
        k_ent_block<<<(unsigned)nblk, kSmallThreads, 0, st>>>(L, n_up, la, V, ldv, w, pl.block_doubles, pl.mmax, pl.dmax,
                                                              parts);
        if (cudaGetLastError() != cudaSuccess) return MBL_ERR_CUDA;
        note_launch();
        k_ent_block_combine<<<(nvec + 127) / 128, 128, 0, st>>>(nvec, pl.blocks_per_vector, parts, S);
        return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
    }
    EntCut cut{};
    cut.L = L;
    cut.n_up = n_up;
    cut.la = la;
    cut.block_doubles = pl.block_doubles;
    cut.mmax = pl.mmax;
    cut.dmax = pl.dmax;
    auto side = [&](int p) { return std::min(host_binom(la, p), host_binom(L - la, n_up - p)); };
    for (int p = std::max(0, n_up - (L - la)); p <= std::min(la, n_up); ++p) {
        int i = cut.np++;
        for (; i > 0 && side(cut.p[i - 1]) < side(p); --i) cut.p[i] = cut.p[i - 1];
        cut.p[i] = p;
    }
    const unsigned njob = (unsigned)(cut.np * nvec);
    const int d = (int)pl.dmax, nt = (d + kEntTile - 1) / kEntTile, nr = (d + kEntCluster - 1) / kEntCluster;
    static const cudaError_t attr = cudaFuncSetAttribute(k_ent_tridiag, cudaFuncAttributeMaxDynamicSharedMemorySize, kEntSmem);
    if (attr != cudaSuccess) return MBL_ERR_CUDA;
    const size_t vec_bytes = (size_t)3 * d * sizeof(double), row_bytes = (size_t)nr * d * sizeof(double);
    const int in_smem = vec_bytes + row_bytes <= (size_t)kEntSmem;
    for (unsigned done = 0; done < njob; done += 32768u) {  // a grid's second dimension ends at 65,535
        const unsigned now = std::min(njob - done, 32768u);
        cut.job0 = (int)done;
        note_launch(4);
        k_ent_gather<<<dim3(8, now), kEntThreads, 0, st>>>(cut, nvec, V, ldv, w);
        k_ent_gram<<<dim3((unsigned)(nt * (nt + 1) / 2), now), kEntThreads, 0, st>>>(cut, nvec, w);
        k_ent_tridiag<<<now * kEntCluster, kEntThreads, vec_bytes + (in_smem ? row_bytes : 0), st>>>(cut, nvec, w,
                                                                                                     in_smem);
        k_ent_eig<<<dim3((unsigned)((d + 31) / 32), now), 32, (size_t)d * sizeof(double2), st>>>(cut, nvec, w);
        if (cudaGetLastError() != cudaSuccess) return MBL_ERR_CUDA;
    }
    note_launch();
    k_ent_combine<<<(nvec + 127) / 128, 128, 0, st>>>(cut, nvec, w, S);
    return cudaGetLastError() == cudaSuccess ? MBL_OK : MBL_ERR_CUDA;
}

size_t entanglement_work_bytes(const EntanglementPlan &pl, int nvec)
{
    const int64_t nblk = (int64_t)nvec * pl.blocks_per_vector;
    return (size_t)(nblk * pl.block_doubles + 2 * nblk + 64) * sizeof(double) + 256;
}


}  // namespace mbl
