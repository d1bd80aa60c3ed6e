// Dense FP64 linear algebra on the device: a tiled DGEMM, blocked Cholesky
// S = L L^T, the triangular inverse L^-1, closed-form overlap/kinetic
// integrals, reductions and the Lanczos spectral bounds.
//
// The paper applies S^-1 to columns by PCG with an incomplete-Cholesky
// preconditioner (footnote 2); here S is factored once per geometry in FP64
// and L^-1 is kept, which gives the same operator to roundoff.
#include "dft_internal.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

namespace dft {
namespace {

constexpr int GB = 64;   // tile edge
constexpr int GK = 16;   // k-slab

// C = A^T B (row-major, A Kd x M, B Kd x N), 256 threads, 4x4 outputs each
__global__ void __launch_bounds__(256) k_dgemm_tn(int M, int N, int Kd, const double* __restrict__ A, int lda,
                                                  const double* __restrict__ B, int ldb, double* __restrict__ C,
                                                  int ldc) {
    __shared__ double As[GK][GB + 1];
    __shared__ double Bs[GK][GB + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int m0 = blockIdx.y * GB, n0 = blockIdx.x * GB;
    double acc[4][4] = {};
    for (int k0 = 0; k0 < Kd; k0 += GK) {
        for (int e = threadIdx.x; e < GB * GK; e += 256) {
            const int mm = e % GB, kk = e / GB, gk = k0 + kk;
            As[kk][mm] = m0 + mm < M && gk < Kd ? A[(long long)gk * lda + m0 + mm] : 0.0;
            Bs[kk][mm] = n0 + mm < N && gk < Kd ? B[(long long)gk * ldb + n0 + mm] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        int gm = m0 + ty + 16 * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int gn = n0 + tx + 16 * j;
            if (gn < N) C[(long long)gm * ldc + gn] = acc[i][j];
        }
    }
}

// Square K x K products with a triangular factor: the k range of each GB x GB
// (64, or 32 where 64 would leave SMs idle: K < ~800)
// output tile is cut to where the triangular operand is nonzero, and with
// UPPER only tiles on or above the diagonal are computed (symmetric results,
// mirrored afterwards).  KR: 0 full, 1 k < end of row tile, 2 k < end of
// column tile, 3 k >= start of row tile, 4 k >= start of column tile.
template <int GB, bool TA, bool TB, int KR, bool UPPER>
__global__ void __launch_bounds__(256) k_dgemm_tri(int K, const double* __restrict__ A, const double* __restrict__ B,
                                                   double* __restrict__ C) {
    if (UPPER && blockIdx.x < blockIdx.y) return;
    __shared__ double As[GK][GB + 1];
    __shared__ double Bs[GK][GB + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int m0 = blockIdx.y * GB, n0 = blockIdx.x * GB;
    int klo = 0, khi = K;
    if (KR == 1) khi = min(K, m0 + GB);
    if (KR == 2) khi = min(K, n0 + GB);
    if (KR == 3) klo = m0;
    if (KR == 4) klo = n0;
    constexpr int TM = GB / 16;
    double acc[TM][TM] = {};
    for (int k0 = klo; k0 < khi; k0 += GK) {
        for (int e = threadIdx.x; e < GB * GK; e += 256) {
            int mm, kk;
            if (!TA) { kk = e % GK; mm = e / GK; } else { mm = e % GB; kk = e / GB; }
            int gm = m0 + mm, gk = k0 + kk;
            double v = 0.0;
            if (gm < K && gk < khi) v = TA ? A[(long long)gk * K + gm] : A[(long long)gm * K + gk];
            As[kk][mm] = v;
        }
        for (int e = threadIdx.x; e < GB * GK; e += 256) {
            int nn, kk;
            if (!TB) { nn = e % GB; kk = e / GB; } else { kk = e % GK; nn = e / GK; }
            int gn = n0 + nn, gk = k0 + kk;
            double v = 0.0;
            if (gn < K && gk < khi) v = TB ? B[(long long)gn * K + gk] : B[(long long)gk * K + gn];
            Bs[kk][nn] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            double a[TM], b[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TM; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        int gm = m0 + ty + 16 * i;
        if (gm >= K) continue;
#pragma unroll
        for (int j = 0; j < TM; ++j) {
            int gn = n0 + tx + 16 * j;
            if (gn < K) C[(long long)gm * K + gn] = acc[i][j];
        }
    }
}

// lower triangle from the upper one (for results of k_dgemm_tri<..., true>)
__global__ void k_mirror_upper(int K, double* C) {
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)K * K) return;
    int i = (int)(e / K), j = (int)(e % K);
    if (i > j) C[e] = C[(long long)j * K + i];
}

// in-place Cholesky of the nb x nb diagonal block at (kb, kb); lower factor
__global__ void __launch_bounds__(256) k_potrf_diag(double* A, int K, int kb, int nb, int* flag) {
    __shared__ double s[GB][GB + 1];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        int i = e / nb, j = e % nb;
        s[i][j] = A[(long long)(kb + i) * K + kb + j];
    }
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        __shared__ double d;
        if (threadIdx.x == 0) {
            double v = s[j][j];
            if (!(v > 0.0)) { atomicExch(flag, 1); v = 1.0; }
            d = sqrt(v);
            s[j][j] = d;
        }
        __syncthreads();
        for (int i = j + 1 + threadIdx.x; i < nb; i += blockDim.x) s[i][j] /= d;
        __syncthreads();
        int rem = nb - j - 1;
        for (int e = threadIdx.x; e < rem * rem; e += blockDim.x) {
            int i = j + 1 + e / rem, k = j + 1 + e % rem;
            if (k <= i) s[i][k] -= s[i][j] * s[k][j];
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        int i = e / nb, j = e % nb;
        if (j <= i) A[(long long)(kb + i) * K + kb + j] = s[i][j];
    }
}

// C -= P P^T on the 64 x 64 tiles on and below the diagonal (P: n x nb, nb <= GB)
__global__ void __launch_bounds__(256) k_syrk_lower(int n, int nb, const double* __restrict__ P, double* __restrict__ C,
                                                    int ld) {
    __shared__ double As[GK][GB + 1];
    __shared__ double Bs[GK][GB + 1];
    int ti = 0, tj = blockIdx.x;   // row tile ti, column tile tj <= ti
    while (tj > ti) {
        tj -= ti + 1;
        ++ti;
    }
    const int m0 = ti * GB, n0 = tj * GB, tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[4][4] = {};
    for (int k0 = 0; k0 < nb; k0 += GK) {
        for (int e = threadIdx.x; e < GB * GK; e += 256) {
            const int kk = e % GK, mm = e / GK;
            As[kk][mm] = (m0 + mm < n && k0 + kk < nb) ? P[(long long)(m0 + mm) * ld + k0 + kk] : 0.0;
            Bs[kk][mm] = (n0 + mm < n && k0 + kk < nb) ? P[(long long)(n0 + mm) * ld + k0 + kk] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + ty + 16 * i;
        if (gm >= n) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tx + 16 * j;
            if (gn < n) C[(long long)gm * ld + gn] -= acc[i][j];
        }
    }
}

// rows below the diagonal block: a <- a L_kk^-T (solve x L^T = a), TRSM_R rows
// per warp, two columns per lane: x_j is passed to all lanes, which take it out
// of the columns behind j.  (One thread per row, with its 64 unknowns in local
// memory, took 160 us per panel.)
constexpr int TRSM_R = 4, TRSM_W = 4;   // rows per warp, warps per block
__global__ void __launch_bounds__(32 * TRSM_W) k_trsm_panel(double* A, int K, int kb, int nb) {
    __shared__ double Lt[GB][GB + 1];   // Lt[j][c] = L[c][j]
    __shared__ double inv[GB];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const int i = e / nb, j = e % nb;
        Lt[j][i] = A[(long long)(kb + i) * K + kb + j];
    }
    __syncthreads();
    for (int j = threadIdx.x; j < nb; j += blockDim.x) inv[j] = 1.0 / Lt[j][j];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int r0 = kb + nb + (blockIdx.x * TRSM_W + (threadIdx.x >> 5)) * TRSM_R;
    double a[TRSM_R][2];
#pragma unroll
    for (int q = 0; q < TRSM_R; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            a[q][h] = (r0 + q < K && c < nb) ? A[(long long)(r0 + q) * K + kb + c] : 0.0;
        }
    auto steps = [&](int h, int j0, int j1) {   // h is a constant in each call
        for (int j = j0; j < j1; ++j) {
            const double l0 = lane < nb ? Lt[j][lane] : 0.0, l1 = lane + 32 < nb ? Lt[j][lane + 32] : 0.0;
            const double d = Lt[j][j], id = inv[j];
#pragma unroll
            for (int q = 0; q < TRSM_R; ++q) {
                const double v = __shfl_sync(0xffffffffu, h ? a[q][1] : a[q][0], j & 31);
                double x = v * id;
                x = fma(fma(-x, d, v), id, x);   // v / d to rounding
                if (h == 0) {
                    if (lane > j) a[q][0] = fma(-x, l0, a[q][0]);
                    else if (lane == j) a[q][0] = x;
                    a[q][1] = fma(-x, l1, a[q][1]);
                } else {
                    if (lane + 32 > j) a[q][1] = fma(-x, l1, a[q][1]);
                    else if (lane + 32 == j) a[q][1] = x;
                }
            }
        }
    };
    steps(0, 0, min(nb, 32));
    steps(1, 32, nb);
#pragma unroll
    for (int q = 0; q < TRSM_R; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = lane + 32 * h;
            if (r0 + q < K && c < nb) A[(long long)(r0 + q) * K + kb + c] = a[q][h];
        }
}

__global__ void k_zero_upper(double* A, int K) {
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)K * K) return;
    int i = (int)(e / K), j = (int)(e % K);
    if (j > i) A[e] = 0.0;
}

constexpr int TIB = 32;  // leaf size of the recursive triangular inverse

// inverse of an n x n (n <= TIB) lower-triangular block in shared memory, one
// column per thread (forward substitution), written with leading dimension ld
// (block b: rows and columns b TIB ... of the K x K factor)
__global__ void __launch_bounds__(TIB) k_tri_inv_block(const double* __restrict__ L, double* __restrict__ X, int K) {
    const int ld = K, n = min(TIB, K - (int)blockIdx.x * TIB);
    L += (long long)blockIdx.x * TIB * (K + 1);
    X += (long long)blockIdx.x * TIB * (K + 1);
    __shared__ double Ls[TIB][TIB + 1];
    __shared__ double Xs[TIB][TIB + 1];
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        int i = e / n, j = e % n;
        Ls[i][j] = L[(long long)i * ld + j];
    }
    __syncthreads();
    const int c = threadIdx.x;
    if (c < n) {
        for (int r = 0; r < n; ++r) {
            double v = 0.0;
            if (r >= c) {
                double acc = (r == c) ? 1.0 : 0.0;
                for (int m = c; m < r; ++m) acc -= Ls[r][m] * Xs[m][c];
                v = acc / Ls[r][r];
            }
            Xs[r][c] = v;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        int i = e / n, j = e % n;
        X[(long long)i * ld + j] = Xs[i][j];
    }
}

// One level of the triangular inverse: neighbouring diagonal blocks of b rows
// are inverted, X_21 = -C^-1 (B A^-1) joins them, for all pairs blockIdx.z at
// once.  Phase 1: tmp = B A^-1 (A^-1 lower triangular: k from the column tile on);
// phase 2: X_21 = -C^-1 tmp (k up to the row tile's end).  Tiles of 64 x 64, or
// 32 x 32 for the small blocks; tmp in a K x K scratch at X_21's place.
template <int GB>
__global__ void __launch_bounds__(256) k_tri_level(int K, int b, int phase, const double* __restrict__ L,
                                                   double* __restrict__ X, double* __restrict__ tmp) {
    constexpr int TM = GB / 16;
    __shared__ double As[GK][GB + 1];
    __shared__ double Bs[GK][GB + 1];
    const int c0 = blockIdx.z * 2 * b, r0 = c0 + b;   // the pair's first column, and first row of its lower block
    const int n2 = min(b, K - r0);
    const int m0 = blockIdx.y * GB, n0 = blockIdx.x * GB;
    if (n2 <= 0 || m0 >= n2) return;
    const double* P = phase == 1 ? L + (long long)r0 * K + c0 : X + (long long)r0 * K + r0;     // n2 x (b or n2)
    const double* Q = phase == 1 ? X + (long long)c0 * K + c0 : tmp + (long long)r0 * K + c0;   // (b or n2) x b
    double* out = (phase == 1 ? tmp : X) + (long long)r0 * K + c0;
    const int klo = phase == 1 ? n0 : 0, khi = phase == 1 ? b : min(n2, m0 + GB);
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[TM][TM] = {};
    for (int k0 = klo; k0 < khi; k0 += GK) {
        for (int e = threadIdx.x; e < GB * GK; e += 256) {
            const int kk = e % GK, mm = e / GK;
            As[kk][mm] = (m0 + mm < n2 && k0 + kk < khi) ? P[(long long)(m0 + mm) * K + k0 + kk] : 0.0;
            const int nn = e % GB, kb = e / GB;
            Bs[kb][nn] = (n0 + nn < b && k0 + kb < khi) ? Q[(long long)(k0 + kb) * K + n0 + nn] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            double av[TM], bv[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) av[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TM; ++j) bv[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TM; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    const double sign = phase == 1 ? 1.0 : -1.0;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int gm = m0 + ty + 16 * i;
        if (gm >= n2) continue;
#pragma unroll
        for (int j = 0; j < TM; ++j) {
            const int gn = n0 + tx + 16 * j;
            if (gn < b) out[(long long)gm * K + gn] = sign * acc[i][j];
        }
    }
}

// --- closed-form overlap and kinetic integrals of Cartesian primitives ---
// 1D integrals int (x-A)^i (x-B)^j exp(-a (x-A)^2 - b (x-B)^2) dx for i, j <= 3
// (powers up to 2, one more for the kinetic integrals), from the Gaussian
// product e^{-mu (A-B)^2} e^{-p (x-P)^2} and the moments
// int u^n e^{-p u^2} du = sqrt(pi/p) (n-1)!! / (2p)^(n/2) for even n.
constexpr int OS_N = 4;
__device__ void overlap_1d(double a, double b, double A, double B, double s[OS_N][OS_N]) {
    double p = a + b, mu = a * b / p, P = (a * A + b * B) / p;
    double E = sqrt(M_PI / p) * exp(-mu * (A - B) * (A - B));
    double xa = P - A, xb = P - B;
    const double q = 0.5 / p;
    const double g[7] = {1.0, 0.0, q, 0.0, 3.0 * q * q, 0.0, 15.0 * q * q * q};
    const double binom[OS_N][OS_N] = {{1, 0, 0, 0}, {1, 1, 0, 0}, {1, 2, 1, 0}, {1, 3, 3, 1}};
    // powers by multiplication (a general pow costs hundreds of FP64
    // operations on this part's narrow FP64 pipe)
    const double pa[OS_N] = {1.0, xa, xa * xa, xa * xa * xa};
    const double pb[OS_N] = {1.0, xb, xb * xb, xb * xb * xb};
#pragma unroll
    for (int i = 0; i < OS_N; ++i)
#pragma unroll
        for (int j = 0; j < OS_N; ++j) {
            double acc = 0.0;
#pragma unroll
            for (int r = 0; r <= i; ++r)
#pragma unroll
                for (int t = 0; t <= j; ++t)
                    if (((r + t) & 1) == 0) acc += binom[i][r] * binom[j][t] * pa[i - r] * pb[j - t] * g[r + t];
            s[i][j] = E * acc;
        }
}

__global__ void k_overlap_kinetic(const Fn* __restrict__ fn, int K, double* __restrict__ S, double* __restrict__ T) {
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)K * K) return;
    int i = (int)(e / K), j = (int)(e % K);
    if (j < i) return;   // mirrored below
    const Fn fa = fn[i], fb = fn[j];
    const double Ac[3] = {fa.cx, fa.cy, fa.cz}, Bc[3] = {fb.cx, fb.cy, fb.cz};
    const int pa[3] = {fa.px, fa.py, fa.pz}, pb[3] = {fb.px, fb.py, fb.pz};
    double Sd[3], Td[3];
    for (int d = 0; d < 3; ++d) {
        double s[OS_N][OS_N];
        overlap_1d(fa.zeta, fb.zeta, Ac[d], Bc[d], s);
        int u = pa[d], v = pb[d];
        Sd[d] = s[u][v];
        // 1/2 int (d/dx phi_u)(d/dx phi_v): d/dx[(x-A)^u e^{-a(x-A)^2}] = u (x-A)^{u-1} - 2a (x-A)^{u+1}
        double t = 4.0 * fa.zeta * fb.zeta * s[u + 1][v + 1];
        if (u > 0) t -= 2.0 * fb.zeta * u * s[u - 1][v + 1];
        if (v > 0) t -= 2.0 * fa.zeta * v * s[u + 1][v - 1];
        if (u > 0 && v > 0) t += u * v * s[u - 1][v - 1];
        Td[d] = 0.5 * t;
    }
    double nn = fa.norm * fb.norm;
    const long long m = (long long)j * K + i;
    if (S) S[e] = S[m] = nn * Sd[0] * Sd[1] * Sd[2];
    if (T) T[e] = T[m] = nn * (Td[0] * Sd[1] * Sd[2] + Sd[0] * Td[1] * Sd[2] + Sd[0] * Sd[1] * Td[2]);
}

__global__ void k_axpby(long long n, double a, const double* X, double b, const double* Y, double* Z) {
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) Z[e] = a * X[e] + b * Y[e];
}

__global__ void k_normalise_h(int K, const double* __restrict__ Ft, const double* __restrict__ scal,
                              double* __restrict__ H) {
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)K * K) return;
    double emin = scal[SCAL_EMIN], emax = scal[SCAL_EMAX];
    double eb = 0.5 * (emax + emin), de = 0.5 * (emax - emin);
    int i = (int)(e / K), j = (int)(e % K);
    // symmetrise while normalising: H_N = ((F~ + F~^T)/2 - Ebar I) / dE
    double v = 0.5 * (Ft[e] + Ft[(long long)j * K + i]);
    if (i == j) v -= eb;
    H[e] = v / de;
}

template <int BS>
__device__ double block_sum(double v) {
    __shared__ double red[BS / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = threadIdx.x < BS / 32 ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;  // valid in thread 0
}

__global__ void __launch_bounds__(256) k_dot_part(long long n, const double* __restrict__ X,
                                                  const double* __restrict__ Y, double* part) {
    double s = 0.0;
    for (long long e = (long long)blockIdx.x * 256 + threadIdx.x; e < n; e += (long long)gridDim.x * 256)
        s = fma(X[e], Y[e], s);
    s = block_sum<256>(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void __launch_bounds__(256) k_sum_parts(int np, const double* part, double* out) {
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += 256) s += part[i];
    s = block_sum<256>(s);
    if (threadIdx.x == 0) *out = s;
}

// --- Lanczos ---
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// single CTA: v0 = random, normalised; beta_0 = 0
__global__ void __launch_bounds__(1024) k_lanczos_start(int K, unsigned long long seed, double* v, double* scal) {
    double s = 0.0;
    for (int i = threadIdx.x; i < K; i += 1024) {
        double r = (double)(splitmix64(seed * 0x100000001B3ull + (unsigned long long)i) >> 11) * 0x1.0p-53 - 0.5;
        v[i] = r;
        s += r * r;
    }
    s = block_sum<1024>(s);
    __shared__ double nrm;
    if (threadIdx.x == 0) { nrm = sqrt(s); scal[SCAL_BETA] = 0.0; }
    __syncthreads();
    for (int i = threadIdx.x; i < K; i += 1024) v[i] /= nrm;
}

// y = A x, one warp per row
__global__ void __launch_bounds__(256) k_gemv(int K, const double* __restrict__ A, const double* __restrict__ x,
                                              double* __restrict__ y) {
    int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= K) return;
    const double* a = A + (long long)row * K;
    double s = 0.0;
    for (int c = threadIdx.x & 31; c < K; c += 32) s = fma(a[c], x[c], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) y[row] = s;
}

// single CTA: alpha_j = w.v_j; w -= alpha v_j + beta_j v_{j-1}; (twice, for
// local orthogonality); beta_{j+1} = |w|; v_{j+1} = w / beta_{j+1}
// (NT threads: each FP64 warp instruction takes 16 clocks of the SM, so the
// reductions cost in proportion to the warps; a small K takes few)
template <int NT>
__global__ void __launch_bounds__(NT) k_lanczos_update(int K, int j, double* w, const double* vj,
                                                         const double* vjm1, double* vnext, double* scal) {
    __shared__ double sh;
    double s = 0.0;
    for (int i = threadIdx.x; i < K; i += NT) s = fma(w[i], vj[i], s);
    s = block_sum<NT>(s);
    if (threadIdx.x == 0) sh = s;
    __syncthreads();
    double alpha = sh;
    double beta = scal[SCAL_BETA + j];
    for (int i = threadIdx.x; i < K; i += NT) w[i] = w[i] - alpha * vj[i] - (j > 0 ? beta * vjm1[i] : 0.0);
    __syncthreads();
    // second pass against v_j (cheap reorthogonalisation)
    s = 0.0;
    for (int i = threadIdx.x; i < K; i += NT) s = fma(w[i], vj[i], s);
    s = block_sum<NT>(s);
    if (threadIdx.x == 0) sh = s;
    __syncthreads();
    double c = sh;
    alpha += c;
    s = 0.0;
    for (int i = threadIdx.x; i < K; i += NT) {
        double v = w[i] - c * vj[i];
        w[i] = v;
        s = fma(v, v, s);
    }
    s = block_sum<NT>(s);
    if (threadIdx.x == 0) sh = sqrt(s);
    __syncthreads();
    double bn = sh;
    double inv = bn > 0.0 ? 1.0 / bn : 0.0;
    for (int i = threadIdx.x; i < K; i += NT) vnext[i] = w[i] * inv;
    if (threadIdx.x == 0) {
        scal[SCAL_ALPHA + j] = alpha;
        scal[SCAL_BETA + j + 1] = bn;
    }
}

// The whole Lanczos run of a small matrix as one launch of a cluster of CL
// CTAs: each holds all of v_j and v_{j-1} and owns every CL-th run of rows; per step three
// cluster barriers, after the partial sums of alpha, of the correction c and of
// |w|^2 (published with the CTA's part of w) have been written to all CTAs.
// 64 steps as 128 launches took 0.65 ms at K = 370 (and, with a batch's host
// threads launching together, several ms of the driver's lock).
constexpr int LC_CL = 8, LC_THREADS = 128, LC_MAX_K = 448;   // K: a CTA's rows of A stay in its shared memory
__global__ void __cluster_dims__(LC_CL, 1, 1) __launch_bounds__(LC_THREADS)
    k_lanczos_cluster(int K, int m, unsigned long long seed, const double* __restrict__ A, double* scal) {
    namespace cgx = cooperative_groups;
    cgx::cluster_group cl = cgx::this_cluster();
    __shared__ double vj[LC_MAX_K], vp[LC_MAX_K], w[LC_MAX_K], part[3][LC_CL];
    __shared__ double sh;
    const int rank = (int)cl.block_rank(), t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (K + LC_CL - 1) / LC_CL, r0 = min(K, rank * per), r1 = min(K, r0 + per);
    extern __shared__ double rows[];
    for (int e = t; e < (r1 - r0) * K; e += LC_THREADS) rows[e] = A[(long long)r0 * K + e];
    // start vector, formed by every CTA for itself
    double s = 0.0;
    for (int i = t; i < K; i += LC_THREADS) {
        const double r = (double)(splitmix64(seed * 0x100000001B3ull + (unsigned long long)i) >> 11) * 0x1.0p-53 - 0.5;
        vj[i] = r;
        vp[i] = 0.0;
        s += r * r;
    }
    s = block_sum<LC_THREADS>(s);
    if (t == 0) sh = sqrt(s);
    __syncthreads();
    for (int i = t; i < K; i += LC_THREADS) vj[i] /= sh;
    double beta = 0.0;
    if (rank == 0 && t == 0) scal[SCAL_BETA] = 0.0;
    // this CTA's partial sum to slot `which` of every CTA
    auto publish = [&](double x, int which) {
        x = block_sum<LC_THREADS>(x);
        if (t == 0) sh = x;
        __syncthreads();
        if (t < LC_CL) cl.map_shared_rank(&part[which][rank], t)[0] = sh;
    };
    auto total = [&](int which) {
        double x = 0.0;
        for (int q = 0; q < LC_CL; ++q) x += part[which][q];
        return x;
    };
    cl.sync();
    for (int j = 0; j < m; ++j) {
        s = 0.0;
        // one row per 8 lanes: three shuffle additions per row instead of five
        for (int r = r0 + 4 * warp + (lane >> 3); r - (lane >> 3) < r1; r += 4 * LC_THREADS / 32) {
            const double* a = rows + (r - r0) * K;
            double x = 0.0, y = 0.0;
            if (r < r1)
                for (int c = lane & 7; c < K; c += 16) {
                    x = fma(a[c], vj[c], x);
                    if (c + 8 < K) y = fma(a[c + 8], vj[c + 8], y);
                }
            x += y;
            for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if ((lane & 7) == 0 && r < r1) {
                w[r] = x;
                s = fma(x, vj[r], s);
            }
        }
        publish(s, 0);
        cl.sync();
        double alpha = total(0);
        s = 0.0;
        for (int r = r0 + t; r < r1; r += LC_THREADS) {
            const double x = w[r] - alpha * vj[r] - beta * vp[r];
            w[r] = x;
            s = fma(x, vj[r], s);
        }
        publish(s, 1);
        cl.sync();
        const double c = total(1);   // second pass against v_j (local orthogonality)
        alpha += c;
        s = 0.0;
        for (int r = r0 + t; r < r1; r += LC_THREADS) {
            const double x = w[r] - c * vj[r];
            s = fma(x, x, s);
            w[r] = x;
            for (int q = 0; q < LC_CL; ++q)
                if (q != rank) cl.map_shared_rank(&w[r], q)[0] = x;
        }
        publish(s, 2);
        cl.sync();
        const double bn = sqrt(total(2)), inv = bn > 0.0 ? 1.0 / bn : 0.0;
        for (int i = t; i < K; i += LC_THREADS) {
            vp[i] = vj[i];
            vj[i] = w[i] * inv;
        }
        beta = bn;
        if (rank == 0 && t == 0) {
            scal[SCAL_ALPHA + j] = alpha;
            scal[SCAL_BETA + j + 1] = bn;
        }
        __syncthreads();
        // w of the next step is written by its own CTA only, and read here above by
        // threads of this CTA; others write into it after the next two barriers
    }
    cl.sync();   // no CTA leaves while its shared memory may still be written
}

// number of eigenvalues of the m x m tridiagonal below x (Sturm sequence)
__device__ int sturm_count(const double* al, const double* be, int m, double x) {
    int cnt = 0;
    double q = al[0] - x;
    if (q < 0) ++cnt;
    for (int i = 1; i < m; ++i) {
        double qq = (q == 0.0) ? 1e-300 : q;
        q = (al[i] - x) - be[i] * be[i] / qq;
        if (q < 0) ++cnt;
    }
    return cnt;
}

// extreme eigenvalues of the Lanczos tridiagonal by multisection on the Sturm
// count, one launch per round: TRI_BLOCKS blocks of 32 points for the smallest
// (blocks 0 ..) and as many for the largest eigenvalue, so the bracket shrinks
// by 32 TRI_BLOCKS + 1 per round; every warp first reduces the counts of the
// round before to its bracket.  One warp per block and SM: the divisions of
// the Sturm sequence keep the SM's FP64 pipe busy by themselves (both ends on
// one SM with 32 points each took 417 us).  The last round pads the bounds
// by 2% of the width on each side (the paper does not say how E_min and E_max
// are found).  state: two rounds' {a, b} and counts per end.
constexpr int TRI_BLOCKS = 32, TRI_PTS = 32 * TRI_BLOCKS, TRI_ROUNDS = 6;
constexpr int TRI_STATE = 2 + TRI_PTS;   // doubles per end and round
__global__ void __launch_bounds__(32) k_tridiag_round(int round, int m, double* scal, double* state) {
    const double* al = scal + SCAL_ALPHA;
    const double* be = scal + SCAL_BETA;
    const int lane = threadIdx.x;
    auto bracket = [&](int end, double& a, double& b) {
        const int target = end == 0 ? 1 : m;
        if (round == 0) {
            double lo = 1e300, hi = -1e300;
            for (int i = lane; i < m; i += 32) {
                const double r = (i > 0 ? fabs(be[i]) : 0.0) + (i + 1 < m ? fabs(be[i + 1]) : 0.0);
                lo = fmin(lo, al[i] - r);
                hi = fmax(hi, al[i] + r);
            }
            for (int o = 16; o > 0; o >>= 1) {
                lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            }
            a = lo;   // count(a) < target <= count(b)
            b = hi;
            return;
        }
        const double* st = state + (((round + 1) & 1) * 2 + end) * TRI_STATE;
        int j = TRI_PTS;   // first point with count >= target
        for (int i = lane; i < TRI_PTS; i += 32)
            if (st[2 + i] >= (double)target) {
                j = i;
                break;
            }
        for (int o = 16; o > 0; o >>= 1) j = min(j, __shfl_xor_sync(0xffffffffu, j, o));
        const double w = (st[1] - st[0]) / (TRI_PTS + 1);
        a = j == 0 ? st[0] : st[0] + w * j;
        b = j == TRI_PTS ? st[1] : st[0] + w * (j + 1);
    };
    if (round == TRI_ROUNDS) {
        double a, b, e[2];
        for (int end = 0; end < 2; ++end) {
            bracket(end, a, b);
            e[end] = 0.5 * (a + b);
        }
        if (lane == 0) {
            const double pad = 0.02 * (e[1] - e[0]) + 1e-3;
            scal[SCAL_EMIN] = e[0] - pad;
            scal[SCAL_EMAX] = e[1] + pad;
        }
        return;
    }
    const int end = blockIdx.x / TRI_BLOCKS, p = (blockIdx.x % TRI_BLOCKS) * 32 + lane;
    double a, b;
    bracket(end, a, b);
    double* st = state + ((round & 1) * 2 + end) * TRI_STATE;
    st[2 + p] = (double)sturm_count(al, be, m, a + (b - a) / (TRI_PTS + 1) * (p + 1));
    if (p == 0) {
        st[0] = a;
        st[1] = b;
    }
}

inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

void dgemm_tn(int M, int N, int Kd, const double* A, int lda, const double* B, int ldb, double* C, int ldc,
              cudaStream_t s) {
    if (M <= 0 || N <= 0) return;
    dim3 grid((N + GB - 1) / GB, (M + GB - 1) / GB);
    k_dgemm_tn<<<grid, 256, 0, s>>>(M, N, Kd, A, lda, B, ldb, C, ldc);
    check_launch("dgemm_tn");
}

int cholesky_inplace(double* A, int K, int* d_flag, cudaStream_t s) {
    for (int kb = 0; kb < K; kb += GB) {
        int nb = std::min(GB, K - kb);
        k_potrf_diag<<<1, 256, 0, s>>>(A, K, kb, nb, d_flag);
        check_launch("potrf_diag");
        int rows = K - kb - nb;
        if (rows > 0) {
            k_trsm_panel<<<blocks_for(rows, TRSM_R * TRSM_W), 32 * TRSM_W, 0, s>>>(A, K, kb, nb);
            check_launch("trsm_panel");
            double* P = A + (long long)(kb + nb) * K + kb;
            const int tb = (rows + GB - 1) / GB;
            k_syrk_lower<<<tb * (tb + 1) / 2, 256, 0, s>>>(rows, nb, P, A + (long long)(kb + nb) * K + kb + nb, K);
            check_launch("syrk_lower");
        }
    }
    k_zero_upper<<<blocks_for((long long)K * K, 256), 256, 0, s>>>(A, K);
    check_launch("cholesky");
    return 0;
}

void congruence_lower(int K, const double* Linv, const double* F, double* tmp, double* out, cudaStream_t s) {
    // out = Linv F Linv^T, Linv lower triangular, F and out symmetric
    auto go = [&](auto tile) {
        constexpr int TB = decltype(tile)::value;
        const int nb = (K + TB - 1) / TB;
        const dim3 grid(nb, nb);
        k_dgemm_tri<TB, false, false, 1, false><<<grid, 256, 0, s>>>(K, Linv, F, tmp);
        k_dgemm_tri<TB, false, true, 2, true><<<grid, 256, 0, s>>>(K, tmp, Linv, out);
    };
    if ((K + 63) / 64 * ((K + 63) / 64) < 152) go(std::integral_constant<int, 32>{});
    else go(std::integral_constant<int, 64>{});
    k_mirror_upper<<<blocks_for((long long)K * K, 256), 256, 0, s>>>(K, out);
    check_launch("congruence_lower", 3);
}

void congruence_lower_t(int K, const double* Linv, const double* R, double* tmp, double* out, cudaStream_t s) {
    // out = Linv^T R Linv, Linv lower triangular, R and out symmetric
    auto go = [&](auto tile) {
        constexpr int TB = decltype(tile)::value;
        const int nb = (K + TB - 1) / TB;
        const dim3 grid(nb, nb);
        k_dgemm_tri<TB, true, false, 3, false><<<grid, 256, 0, s>>>(K, Linv, R, tmp);
        k_dgemm_tri<TB, false, false, 4, true><<<grid, 256, 0, s>>>(K, tmp, Linv, out);
    };
    if ((K + 63) / 64 * ((K + 63) / 64) < 152) go(std::integral_constant<int, 32>{});
    else go(std::integral_constant<int, 64>{});
    k_mirror_upper<<<blocks_for((long long)K * K, 256), 256, 0, s>>>(K, out);
    check_launch("congruence_lower_t", 3);
}

// L^-1 by block pairs, [A 0; B C]^-1 = [A^-1 0; -C^-1 B A^-1  C^-1], from leaves
// of TIB rows upwards: two launches per level (a recursion over single blocks
// took 178 launches and multiplied the zeros too: 17.7 of 34.6 ms at K = 1910)
void tri_inverse_lower(const double* L, double* Linv, int K, double* tmp, cudaStream_t s) {
    // the strictly upper part of L^-1 is zero
    DFT_CUDA_CHECK(cudaMemsetAsync(Linv, 0, sizeof(double) * (size_t)K * K, s));
    k_tri_inv_block<<<(K + TIB - 1) / TIB, TIB, 0, s>>>(L, Linv, K);
    check_launch("tri_inv_block");
    for (int b = TIB; b < K; b *= 2) {
        const int pairs = (K + 2 * b - 1) / (2 * b);
        for (int phase = 1; phase <= 2; ++phase) {
            const int t64 = (b + 63) / 64, t32 = (b + 31) / 32;
            if ((long long)t64 * t64 * pairs >= 2 * 152)
                k_tri_level<64><<<dim3(t64, t64, pairs), 256, 0, s>>>(K, b, phase, L, Linv, tmp);
            else
                k_tri_level<32><<<dim3(t32, t32, pairs), 256, 0, s>>>(K, b, phase, L, Linv, tmp);
        }
        check_launch("tri_level", 2);
    }
}

// (M_c)_ab = N_a N_b sum_{s in a, t in b} Mt_st
__global__ void k_contract(int K, int Kt, const int* __restrict__ tp, const double* __restrict__ nrm,
                           const double* __restrict__ Mt, double* __restrict__ out) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)K * K) return;
    const int a = (int)(e / K), b = (int)(e % K);
    double acc = 0.0;
    for (int si = tp[a]; si < tp[a + 1]; ++si)
        for (int ti = tp[b]; ti < tp[b + 1]; ++ti) acc += Mt[(long long)si * Kt + ti];
    out[e] = nrm[a] * nrm[b] * acc;
}

// N_a = (sum_{s, t in a} St_st)^(-1/2): unit norm of every contracted function
__global__ void k_contract_norms(int K, int Kt, const int* __restrict__ tp, const double* __restrict__ St,
                                 double* __restrict__ nrm) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= K) return;
    double acc = 0.0;
    for (int si = tp[a]; si < tp[a + 1]; ++si)
        for (int ti = tp[a]; ti < tp[a + 1]; ++ti) acc += St[(long long)si * Kt + ti];
    nrm[a] = 1.0 / sqrt(acc);
}

// P_t,st = N_a(s) N_a(t) P_a(s)a(t)
__global__ void k_expand(int K, int Kt, const int* __restrict__ par, const double* __restrict__ nrm,
                         const double* __restrict__ P, double* __restrict__ Pt) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)Kt * Kt) return;
    const int a = par[e / Kt], b = par[e % Kt];
    Pt[e] = nrm[a] * nrm[b] * P[(long long)a * K + b];
}

void launch_contract(const Ctx& c, const double* Mt, double* out, cudaStream_t s) {
    k_contract<<<blocks_for((long long)c.K * c.K, 256), 256, 0, s>>>(c.K, c.Kt, c.d_term_ptr, c.d_cnorm, Mt, out);
    check_launch("contract");
}

void launch_contract_norms(const Ctx& c, const double* St, cudaStream_t s) {
    k_contract_norms<<<(c.K + 255) / 256, 256, 0, s>>>(c.K, c.Kt, c.d_term_ptr, St, c.d_cnorm);
    check_launch("contract_norms");
}

void launch_expand(const Ctx& c, const double* P, double* Pt, cudaStream_t s) {
    k_expand<<<blocks_for((long long)c.Kt * c.Kt, 256), 256, 0, s>>>(c.K, c.Kt, c.d_term_par, c.d_cnorm, P, Pt);
    check_launch("expand");
}

void launch_overlap_kinetic_terms(const Ctx& c, double* St, cudaStream_t s) {
    k_overlap_kinetic<<<blocks_for((long long)c.Kt * c.Kt, 256), 256, 0, s>>>(c.d_fn, c.Kt, St, nullptr);
    check_launch("overlap_kinetic");
}

void launch_overlap_kinetic(const Ctx& c, double* S, double* T, cudaStream_t s) {
    if (!c.contracted) {
        k_overlap_kinetic<<<blocks_for((long long)c.K * c.K, 256), 256, 0, s>>>(c.d_fn, c.K, S, T);
        check_launch("overlap_kinetic");
        return;
    }
    // contracted functions: the terms' closed forms, then contraction (the
    // norms N_a were formed at set-up)
    const unsigned nb = blocks_for((long long)c.Kt * c.Kt, 256);
    k_overlap_kinetic<<<nb, 256, 0, s>>>(c.d_fn, c.Kt, c.d_Mt, nullptr);
    check_launch("overlap_kinetic");
    launch_contract(c, c.d_Mt, S, s);
    k_overlap_kinetic<<<nb, 256, 0, s>>>(c.d_fn, c.Kt, nullptr, c.d_Mt);
    check_launch("overlap_kinetic");
    launch_contract(c, c.d_Mt, T, s);
}

void launch_axpby_mat(int K, double a, const double* X, double b, const double* Y, double* Z, cudaStream_t s) {
    long long n = (long long)K * K;
    k_axpby<<<blocks_for(n, 256), 256, 0, s>>>(n, a, X, b, Y, Z);
    check_launch("axpby");
}

void launch_normalise_h(int K, const double* Ft, const double* scal, double* H, cudaStream_t s) {
    k_normalise_h<<<blocks_for((long long)K * K, 256), 256, 0, s>>>(K, Ft, scal, H);
    check_launch("normalise_h");
}

void launch_frob_dot(long long n, const double* X, const double* Y, double* part, double* out, cudaStream_t s) {
    int np = (int)std::min<long long>(1024, (n + 255) / 256);
    k_dot_part<<<np, 256, 0, s>>>(n, X, Y, part);
    k_sum_parts<<<1, 256, 0, s>>>(np, part, out);
    check_launch("frob_dot", 2);
}

// Lanczos bounds with caller-given buffers: vec holds 4 K doubles, scal
// SCAL_COUNT doubles, state TRI_STATE_DOUBLES; the padded bounds land in
// scal[SCAL_EMIN], scal[SCAL_EMAX]
void lanczos_bounds_at(int K, const double* A, int steps, unsigned long long seed, double* vec, double* scal,
                       double* state, cudaStream_t s) {
    static_assert(4 * TRI_STATE <= TRI_STATE_DOUBLES, "scratch of the tridiagonal bounds");
    int m = std::max(2, std::min(steps, std::min(K, 120)));
    double* v[3] = {vec, vec + K, vec + 2 * K};
    double* w = vec + 3 * K;
    if (K <= LC_MAX_K) {
        constexpr int most = (LC_MAX_K + LC_CL - 1) / LC_CL * LC_MAX_K * (int)sizeof(double);
        static_assert(most <= 204800, "rows of a CTA in shared memory");
        DFT_CUDA_CHECK(cudaFuncSetAttribute(k_lanczos_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        k_lanczos_cluster<<<LC_CL, LC_THREADS, (size_t)((K + LC_CL - 1) / LC_CL) * K * sizeof(double), s>>>(K, m, seed, A, scal);
        check_launch("lanczos_cluster");
    } else {
        k_lanczos_start<<<1, 1024, 0, s>>>(K, seed, v[0], scal);
        check_launch("lanczos_start");
    }
    for (int j = 0; j < m && K > LC_MAX_K; ++j) {
        double* vj = v[j % 3];
        double* vjm1 = v[(j + 2) % 3];
        double* vn = v[(j + 1) % 3];
        k_gemv<<<blocks_for(K, 8), 256, 0, s>>>(K, A, vj, w);
        // 128 threads up to K = 1024
        if (K <= 1024) k_lanczos_update<128><<<1, 128, 0, s>>>(K, j, w, vj, vjm1, vn, scal);
        else k_lanczos_update<256><<<1, 256, 0, s>>>(K, j, w, vj, vjm1, vn, scal);
        check_launch("lanczos_step", 2);
    }
    for (int r = 0; r <= TRI_ROUNDS; ++r) k_tridiag_round<<<r < TRI_ROUNDS ? 2 * TRI_BLOCKS : 1, 32, 0, s>>>(r, m, scal, state);
    check_launch("lanczos", TRI_ROUNDS + 1);
}

void lanczos_bounds(const Ctx& c, const double* A, int steps, cudaStream_t s) {
    lanczos_bounds_at(c.K, A, steps, c.p.seed, c.d_vec, c.d_scal, c.d_gram, s);
}

}  // namespace dft
