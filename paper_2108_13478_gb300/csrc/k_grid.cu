// Grid <-> basis kernels: separable tables (Supp. A.1), collocation of the
// density (Eq. 2.7, Supp. A.1.2) and quadrature of a grid potential into a
// matrix (Eq. 2.5 / A.6), plus Gaussian sums on the grid (v_loc, Eq. 2.6).
//
// Work is organised by grid tiles of 8x8x8 points.  Every tile carries the
// list of basis functions whose cubic window W_a (Supp. A.1.1) meets it;
// the per-tile slices of the 1D tables are staged in shared memory so that
// phi_a(r_g) costs two multiplications (Supp. A.1).
#include "dft_internal.cuh"

#include <algorithm>

namespace dft {
namespace {

__global__ void k_build_tables(const Fn* __restrict__ fn, int K, int W, double ox, double oy,
                               double oz, double h, double* __restrict__ tab) {
    long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long total = (long long)K * 3 * W;
    if (idx >= total) return;
    int t = (int)(idx % W);
    int d = (int)((idx / W) % 3);
    int f = (int)(idx / (3LL * W));
    const Fn F = fn[f];
    int i = F.lo[d] + t;
    double val = 0.0;
    if (i <= F.hi[d]) {
        double o = d == 0 ? ox : (d == 1 ? oy : oz);
        double c = d == 0 ? F.cx : (d == 1 ? F.cy : F.cz);
        int pw = d == 0 ? F.px : (d == 1 ? F.py : F.pz);
        double x = (o + h * i) - c;
        val = exp(-F.zeta * x * x);
        if (pw >= 1) val *= x;
        if (pw == 2) val *= x;
        if (d == 0) val *= F.norm;
    }
    tab[idx] = val;
}

// Collocation and quadrature of one 8^3 tile run as small matrix products over
// pairs (ca <= cb) of chunks of CH functions of the tile's list, plane by plane
// (z fixed, 64 points): FP32 with CH = 64 and 8 x 8 sums per thread, so that 4
// shared-memory reads of 16 bytes feed 64 multiply-adds (the FMA pipe is the
// limit, not shared memory); FP64 with CH = 32 and 4 x 4.  A block has two
// groups of 64 threads, one per half of the z planes; both groups share the
// chunk's x, y, z slices.  Only ca <= cb is computed: half of the products
// of the full double sum.  Tiles are launched by falling list length, so that
// the last blocks to run are short ones.
template <typename R>
struct GridCfg {
    static constexpr int TI = sizeof(R) == 4 ? 8 : 4;   // sums per thread and side
    static constexpr int CH = 8 * TI;                   // functions per chunk
    static constexpr int V = TI / 2;                    // elements per 16-byte access
    struct __align__(16) Vec { R v[V]; };
};

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 64;" ::"r"(1 + g) : "memory"); }

// the 8-point slices of CH functions' tables for the tile at t0 (zero outside
// the windows and beyond the list), [axis][function][point]
template <typename R, int CH>
__device__ __forceinline__ void stage_slices(const Fn* __restrict__ fn, const double* __restrict__ tab, int W,
                                             const int* __restrict__ list, int n_t, int c0, const int t0[3],
                                             R (*s)[CH][TILE]) {
    for (int e = threadIdx.x; e < CH * 3 * TILE; e += blockDim.x) {
        const int q = e % TILE, fl = (e / TILE) % CH, d = e / (TILE * CH);
        double val = 0.0;
        if (c0 + fl < n_t) {
            const int f = list[c0 + fl];
            const int i = t0[d] + q;
            const int lo = fn[f].lo[d], hi = fn[f].hi[d];
            if (i >= lo && i <= hi) val = tab[((long long)f * 3 + d) * W + (i - lo)];
        }
        s[d][fl][q] = (R)val;
    }
}

// TI x TI sums of a thread.  FP32 sums are kept in pairs along j and updated by
// the packed fma.rn.f32x2 (same rounding as two scalar ones): the loop is
// bound by instruction issue, and this halves its multiply-adds (1470 functions:
// collocation 2.62 -> 2.21 ms, quadrature 2.36 -> 1.81 ms, the same bits)
template <typename R>
struct Sums;
template <>
struct Sums<double> {
    static constexpr int TI = GridCfg<double>::TI;
    double v[TI][TI];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TI; ++j) v[i][j] = 0.0;
    }
    __device__ __forceinline__ void step(const double (&a)[TI], const double (&b)[TI]) {
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TI; ++j) v[i][j] = fma(a[i], b[j], v[i][j]);
    }
    // row i += z * row i of g
    __device__ __forceinline__ void add_row(int i, double z, const Sums& g) {
#pragma unroll
        for (int j = 0; j < TI; ++j) v[i][j] = fma(z, g.v[i][j], v[i][j]);
    }
    __device__ __forceinline__ void row(int i, double (&o)[TI]) const {
#pragma unroll
        for (int j = 0; j < TI; ++j) o[j] = v[i][j];
    }
};
template <>
struct Sums<float> {
    static constexpr int TI = GridCfg<float>::TI;
    unsigned long long v[TI][TI / 2];
    static __device__ __forceinline__ unsigned long long pack(float x, float y) {
        unsigned long long r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
        return r;
    }
    static __device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TI / 2; ++j) v[i][j] = 0ull;
    }
    __device__ __forceinline__ void step(const float (&a)[TI], const float (&b)[TI]) {
        unsigned long long b2[TI / 2];
#pragma unroll
        for (int j = 0; j < TI / 2; ++j) b2[j] = pack(b[2 * j], b[2 * j + 1]);
#pragma unroll
        for (int i = 0; i < TI; ++i) {
            const unsigned long long a2 = pack(a[i], a[i]);
#pragma unroll
            for (int j = 0; j < TI / 2; ++j) fma2(v[i][j], a2, b2[j]);
        }
    }
    __device__ __forceinline__ void add_row(int i, float z, const Sums& g) {
        const unsigned long long z2 = pack(z, z);
#pragma unroll
        for (int j = 0; j < TI / 2; ++j) fma2(v[i][j], z2, g.v[i][j]);
    }
    __device__ __forceinline__ void row(int i, float (&o)[TI]) const {
#pragma unroll
        for (int j = 0; j < TI / 2; ++j) asm("mov.b64 {%0, %1}, %2;" : "=f"(o[2 * j]), "=f"(o[2 * j + 1]) : "l"(v[i][j]));
    }
};

// sums over NK terms: acc_ij += A[k][i of ty] B[k][j of tx], rows of
// pitch pa, pb; thread indexes i: V ty + (0..V-1) and CH / 2 + V ty + (0..V-1)
template <typename R, int NK>
__device__ __forceinline__ void tile_product(const R* A, int pa, const R* B, int pb, int ty, int tx, Sums<R>& acc) {
    using C = GridCfg<R>;
    using Vec = typename C::Vec;
#pragma unroll 4
    for (int k = 0; k < NK; ++k) {
        R a[C::TI], b[C::TI];
        *(Vec*)&a[0] = *(const Vec*)(A + k * pa + C::V * ty);
        *(Vec*)&a[C::V] = *(const Vec*)(A + k * pa + C::CH / 2 + C::V * ty);
        *(Vec*)&b[0] = *(const Vec*)(B + k * pb + C::V * tx);
        *(Vec*)&b[C::V] = *(const Vec*)(B + k * pb + C::CH / 2 + C::V * tx);
        acc.step(a, b);
    }
}
// function (point) of sum i of thread row (column) t
template <typename R>
__device__ __forceinline__ int sum_at(int t, int i) {
    using C = GridCfg<R>;
    return (i / C::V) * (C::CH / 2) + C::V * t + i % C::V;
}

// n(r_g) = 2 sum_ab P_ab phi_a phi_b for the points of one tile (Eq. A.5): per
// chunk pair and plane Y[q][a] = sum_b phi_b(q) Q_ba, n(q) += sum_a phi_a(q) Y[q][a],
// Q = P_ba + P_ab off the chunk diagonal (P need not be symmetric), P on it.
// FP32 sums are at most CH long and meet in FP64.  Double: the 64 points of a
// plane go through 4 x 4 sums in two halves.
template <typename R>
struct CollSmem {
    using C = GridCfg<R>;
    static constexpr int NB = 32;   // functions of chunk b staged at a time
    R w[2][NB][64];           // phi_b of the group's plane
    R P[C::CH][C::CH + 16 / sizeof(R)];
    R xy[64][C::CH];          // x y of chunk a
    R sa[3][C::CH][TILE], sb[3][C::CH][TILE];
    double n[TILE_PTS];
    int la[C::CH], lb[C::CH];
};
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 3 : 2) k_collocate(
    const Fn* __restrict__ fn, const double* __restrict__ tab, int W, const int* __restrict__ tile_ptr,
    const int* __restrict__ tile_fn, const int* __restrict__ tile_order, int ntx, int nty, int nx, int ny, int nz, int K,
    const double* __restrict__ P, double* __restrict__ n_out) {
    using C = GridCfg<R>;
    constexpr int TI = C::TI, CH = C::CH, NB = CollSmem<R>::NB;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    CollSmem<R>& s = *(CollSmem<R>*)smem_raw;
    const int t = tile_order[blockIdx.x];
    const int tx_ = t % ntx, ty_ = (t / ntx) % nty, tz_ = t / (ntx * nty);
    const int t0[3] = {tx_ * TILE, ty_ * TILE, tz_ * TILE};
    const int* list = tile_fn + tile_ptr[t];
    const int n_t = tile_ptr[t + 1] - tile_ptr[t];
    const int g = threadIdx.x >> 6, u = threadIdx.x & 63, tx = u & 7, ty = u >> 3;
    // planes of this block (gridDim.y blocks share a tile), and of this group
    const int nz_block = TILE / gridDim.y, nz_group = nz_block / 2, z0 = blockIdx.y * nz_block + g * nz_group;
    for (int p = threadIdx.x; p < TILE_PTS; p += 128) s.n[p] = 0.0;
    for (int ca = 0; ca < n_t; ca += CH) {
        __syncthreads();
        stage_slices<R, CH>(fn, tab, W, list, n_t, ca, t0, s.sa);
        for (int e = threadIdx.x; e < CH; e += 128) s.la[e] = ca + e < n_t ? list[ca + e] : -1;
        __syncthreads();
        for (int e = threadIdx.x; e < 64 * CH; e += 128) {
            const int f = e % CH, q = e / CH;
            s.xy[q][f] = s.sa[0][f][q & 7] * s.sa[1][f][q >> 3];
        }
        for (int cb = ca; cb < n_t; cb += CH) {
            __syncthreads();
            stage_slices<R, CH>(fn, tab, W, list, n_t, cb, t0, s.sb);
            for (int e = threadIdx.x; e < CH; e += 128) s.lb[e] = cb + e < n_t ? list[cb + e] : -1;
            __syncthreads();
            // 8 loads in flight per thread (they are scattered runs of a few functions)
            for (int e0 = threadIdx.x; e0 < CH * CH; e0 += 128 * 8) {
                double x[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int e = e0 + 128 * k, fa = s.la[e % CH], fb = s.lb[e / CH];
                    x[k] = fa >= 0 && fb >= 0 ? P[(long long)fb * K + fa] : 0.0;
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) s.P[(e0 + 128 * k) / CH][(e0 + 128 * k) % CH] = (R)x[k];
            }
            if (ca != cb) {
                __syncthreads();
                for (int e0 = threadIdx.x; e0 < CH * CH; e0 += 128 * 8) {
                    double x[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int e = e0 + 128 * k, fa = s.la[e / CH], fb = s.lb[e % CH];
                        x[k] = fa >= 0 && fb >= 0 ? P[(long long)fa * K + fb] : 0.0;
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) s.P[(e0 + 128 * k) % CH][(e0 + 128 * k) / CH] += (R)x[k];
                }
            }
            __syncthreads();
            for (int z = z0; z < z0 + nz_group; ++z) {
#pragma unroll 1
                for (int q0 = 0; q0 < 64; q0 += CH) {   // CH points at a time
                    Sums<R> Y;
                    Y.zero();
#pragma unroll 1
                    for (int b0 = 0; b0 < CH; b0 += NB) {
                        if (q0 == 0 || CH > NB) {
                            group_sync(g);
                            // this thread's point of the plane
                            const int x = u & 7, y = u >> 3;
#pragma unroll 8
                            for (int b = 0; b < NB; ++b)
                                s.w[g][b][u] = s.sb[0][b0 + b][x] * s.sb[1][b0 + b][y] * s.sb[2][b0 + b][z];
                            group_sync(g);
                        }
                        tile_product<R, NB>(&s.w[g][0][q0], 64, &s.P[b0][0], CH + 16 / sizeof(R), ty, tx, Y);
                    }
                    R za[TI];
#pragma unroll
                    for (int j = 0; j < TI; ++j) za[j] = s.sa[2][sum_at<R>(tx, j)][z];
#pragma unroll
                    for (int i = 0; i < TI; ++i) {
                        const int q = q0 + sum_at<R>(ty, i);
                        R c = (R)0, xa[TI], y[TI];
                        Y.row(i, y);
                        *(typename C::Vec*)&xa[0] = *(const typename C::Vec*)&s.xy[q][C::V * tx];
                        *(typename C::Vec*)&xa[C::V] = *(const typename C::Vec*)&s.xy[q][CH / 2 + C::V * tx];
#pragma unroll
                        for (int j = 0; j < TI; ++j) c = fma(xa[j] * za[j], y[j], c);
                        for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                        if (tx == 0) s.n[64 * z + q] += (double)c;
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int p = blockIdx.y * nz_block * 64 + threadIdx.x; p < (int)(blockIdx.y + 1) * nz_block * 64; p += 128) {
        const int gx = t0[0] + (p & 7), gy = t0[1] + ((p >> 3) & 7), gz = t0[2] + (p >> 6);
        if (gx < nx && gy < ny && gz < nz) n_out[((long long)gz * ny + gy) * nx + gx] = 2.0 * s.n[p];
    }
}

// The same for short lists: 256 threads of two points each, SCH functions a at a
// time in registers, phi_b formed by each thread, P taken whole.  k_collocate
// pads the list to chunks of 64 (32) in both indexes and pays for staging a whole
// chunk and its 64 x y products, which a short list does not repay.  Sums as long as
// there: at most 64 functions b, then 8 functions a, then FP64.
constexpr int SCH = 32;
template <typename R>
__global__ void __launch_bounds__(256) k_collocate_short(
    const Fn* __restrict__ fn, const double* __restrict__ tab, int W, const int* __restrict__ tile_ptr,
    const int* __restrict__ tile_fn, const int* __restrict__ tile_order, int ntx, int nty, int nx, int ny, int nz, int K,
    const double* __restrict__ P, double* __restrict__ n_out) {
    __shared__ R sa[3][SCH][TILE], sb[3][SCH][TILE];
    __shared__ __align__(16) R sP[SCH][SCH];
    const int t = tile_order[blockIdx.x];
    const int tx = t % ntx, ty = (t / ntx) % nty, tz = t / (ntx * nty);
    const int t0[3] = {tx * TILE, ty * TILE, tz * TILE};
    const int* list = tile_fn + tile_ptr[t];
    const int n_t = tile_ptr[t + 1] - tile_ptr[t];
    const int px = threadIdx.x & 7, py = (threadIdx.x >> 3) & 7, pz0 = threadIdx.x >> 6, pz1 = pz0 + 4;
    double acc0 = 0.0, acc1 = 0.0;
    for (int ca = 0; ca < n_t; ca += SCH) {
        for (int cb = 0; cb < n_t;) {
            R y0[SCH], y1[SCH];
#pragma unroll
            for (int j = 0; j < SCH; ++j) y0[j] = y1[j] = (R)0;
            for (const int end = min(n_t, cb + 2 * SCH); cb < end; cb += SCH) {
                __syncthreads();
                if (cb == 0) stage_slices<R, SCH>(fn, tab, W, list, n_t, ca, t0, sa);
                stage_slices<R, SCH>(fn, tab, W, list, n_t, cb, t0, sb);
                for (int e = threadIdx.x; e < SCH * SCH; e += 256) {
                    const int i = e / SCH, j = e % SCH;
                    sP[i][j] = (R)(cb + i < n_t && ca + j < n_t ? P[(long long)list[cb + i] * K + list[ca + j]] : 0.0);
                }
                __syncthreads();
                const int nb = min(SCH, n_t - cb);
#pragma unroll 2
                for (int i = 0; i < nb; ++i) {
                    const R pxy = sb[0][i][px] * sb[1][i][py], pb0 = pxy * sb[2][i][pz0], pb1 = pxy * sb[2][i][pz1];
#pragma unroll
                    for (int j = 0; j < SCH; ++j) {
                        y0[j] = fma(pb0, sP[i][j], y0[j]);
                        y1[j] = fma(pb1, sP[i][j], y1[j]);
                    }
                }
            }
            R c0[4] = {}, c1[4] = {};
#pragma unroll
            for (int j = 0; j < SCH; ++j) {
                const R pxy = sa[0][j][px] * sa[1][j][py];
                c0[j % 4] = fma(pxy * sa[2][j][pz0], y0[j], c0[j % 4]);
                c1[j % 4] = fma(pxy * sa[2][j][pz1], y1[j], c1[j % 4]);
            }
            acc0 += (double)((c0[0] + c0[1]) + (c0[2] + c0[3]));
            acc1 += (double)((c1[0] + c1[1]) + (c1[2] + c1[3]));
        }
    }
    const int gx = t0[0] + px, gy = t0[1] + py, gz0 = t0[2] + pz0, gz1 = t0[2] + pz1;
    if (gx < nx && gy < ny) {
        if (gz0 < nz) n_out[((long long)gz0 * ny + gy) * nx + gx] = 2.0 * acc0;
        if (gz1 < nz) n_out[((long long)gz1 * ny + gy) * nx + gx] = 2.0 * acc1;
    }
}

// V_ab += h^3 sum_{g in tile} phi_a v phi_b for all pairs of the tile's list
// (Eq. A.6): per chunk pair and plane G_ab = sum_q (x y)_a(q) w_b(q) with w =
// v phi_b, V_ab += z_a G_ab.  Contributions of different tiles meet as
// integers: each is rounded to a multiple of 2^-48 and added with a 64-bit
// integer atomic into the upper triangle of V's own storage (the lists ascend,
// so la <= lb is fa <= fb), so the sum is exact and independent of the order
// in which tiles finish (the result is the same bit for bit on every run and
// in every batch); k_fixed_to_double then turns the integers into doubles and
// mirrors them.  Rounding each tile's contribution costs
// at most 2^-49 (1.8e-15; ~1e-12 over the ~10^3 tiles two diffuse functions
// share); partial sums must stay within +-2^15 (|V| is O(10) for potentials
// of tens of hartree).
constexpr double QFIX = 281474976710656.0;   // 2^48
template <typename R>
struct QuadSmem {
    using C = GridCfg<R>;
    R w[2][64][C::CH];        // v phi_b of the group's plane; the group's sums at the end
    R xy[64][C::CH];          // x y of chunk a
    R sa[3][C::CH][TILE], sb[3][C::CH][TILE];
    R v[TILE_PTS];
    int la[C::CH], lb[C::CH];
};
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 3 : 2) k_quadrature(
    const Fn* __restrict__ fn, const double* __restrict__ tab, int W, const int* __restrict__ tile_ptr,
    const int* __restrict__ tile_fn, const int* __restrict__ tile_order, int ntx, int nty, int nx, int ny, int nz, int K, double h3,
    const double* __restrict__ v, double* __restrict__ V) {
    using C = GridCfg<R>;
    constexpr int TI = C::TI, CH = C::CH;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    QuadSmem<R>& s = *(QuadSmem<R>*)smem_raw;
    const int t = tile_order[blockIdx.x];
    const int tx_ = t % ntx, ty_ = (t / ntx) % nty, tz_ = t / (ntx * nty);
    const int t0[3] = {tx_ * TILE, ty_ * TILE, tz_ * TILE};
    const int* list = tile_fn + tile_ptr[t];
    const int n_t = tile_ptr[t + 1] - tile_ptr[t];
    if (n_t == 0) return;
    for (int p = threadIdx.x; p < TILE_PTS; p += 128) {
        const int gx = t0[0] + (p & 7), gy = t0[1] + ((p >> 3) & 7), gz = t0[2] + (p >> 6);
        s.v[p] = (R)((gx < nx && gy < ny && gz < nz) ? v[((long long)gz * ny + gy) * nx + gx] : 0.0);
    }
    const int g = threadIdx.x >> 6, u = threadIdx.x & 63, tx = u & 7, ty = u >> 3;
    const int nch = (n_t + CH - 1) / CH, npair = nch * (nch + 1) / 2;
    // this block's run of chunk pairs (gridDim.y blocks share a tile), in row order
    const int p_end = (int)((long long)npair * (blockIdx.y + 1) / gridDim.y);
    int pair = (int)((long long)npair * blockIdx.y / gridDim.y);
    if (pair >= p_end) return;
    int ia = 0, ib = pair;
    while (ib >= nch - ia) {
        ib -= nch - ia;
        ++ia;
    }
    ib += ia;
    for (; pair < p_end; ++ia, ib = ia) {
        const int ca = ia * CH;
        __syncthreads();
        stage_slices<R, CH>(fn, tab, W, list, n_t, ca, t0, s.sa);
        for (int e = threadIdx.x; e < CH; e += 128) s.la[e] = ca + e < n_t ? list[ca + e] : -1;
        __syncthreads();
        for (int e = threadIdx.x; e < 64 * CH; e += 128) {
            const int f = e % CH, q = e / CH;
            s.xy[q][f] = s.sa[0][f][q & 7] * s.sa[1][f][q >> 3];
        }
        for (; ib < nch && pair < p_end; ++ib, ++pair) {
            const int cb = ib * CH;
            __syncthreads();
            stage_slices<R, CH>(fn, tab, W, list, n_t, cb, t0, s.sb);
            for (int e = threadIdx.x; e < CH; e += 128) s.lb[e] = cb + e < n_t ? list[cb + e] : -1;
            __syncthreads();
            Sums<R> acc;
            acc.zero();
            for (int z = 4 * g; z < 4 * g + 4; ++z) {
                group_sync(g);
                {
                    // one function of chunk b per thread (two threads each in FP64), its points of the plane
                    const int f = u % CH, y0 = (u / CH) * (TILE * CH / 64);
                    const R zb = s.sb[2][f][z];
                    R x[TILE];
#pragma unroll
                    for (int k = 0; k < TILE; ++k) x[k] = s.sb[0][f][k] * zb;
#pragma unroll 2
                    for (int y = y0; y < y0 + TILE * CH / 64; ++y) {
                        const R yb = s.sb[1][f][y];
#pragma unroll
                        for (int k = 0; k < TILE; ++k) s.w[g][8 * y + k][f] = x[k] * (yb * s.v[64 * z + 8 * y + k]);
                    }
                }
                group_sync(g);
                Sums<R> G;
                G.zero();
                tile_product<R, 64>(&s.xy[0][0], CH, &s.w[g][0][0], CH, ty, tx, G);
#pragma unroll
                for (int i = 0; i < TI; ++i) acc.add_row(i, s.sa[2][sum_at<R>(ty, i)][z], G);
            }
            group_sync(g);
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                R o[TI];
                acc.row(i, o);
#pragma unroll
                for (int j = 0; j < TI; ++j) s.w[g][sum_at<R>(ty, i)][sum_at<R>(tx, j)] = o[j];
            }
            __syncthreads();
            for (int e = threadIdx.x; e < CH * CH; e += 128) {
                const int a = e / CH, b = e % CH, fa = s.la[a], fb = s.lb[b];
                if (fa < 0 || fb < 0 || fa > fb) continue;
                const R sum = s.w[0][a][b] + s.w[1][a][b];
                const unsigned long long q = (unsigned long long)llrint(h3 * (double)sum * QFIX);
                atomicAdd((unsigned long long*)&V[(long long)fa * K + fb], q);
            }
        }
    }
}

// V's 64-bit integer sums (units of 2^-48, upper triangle) -> doubles, both triangles
__global__ void __launch_bounds__(256) k_fixed_to_double(int K, double* V) {
    __shared__ double sh[32][33];
    const int nb = (K + 31) / 32;
    int ti = 0, tj = blockIdx.x;
    while (tj >= nb - ti) {
        tj -= nb - ti;
        ++ti;
    }
    tj += ti;
    const int c = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < 32; r += 8) {
        const int i = ti * 32 + r, j = tj * 32 + c;
        double x = 0.0;
        if (i < K && j < K && j >= i) {
            const long long e = (long long)i * K + j;
            x = (double)reinterpret_cast<const long long*>(V)[e] * (1.0 / QFIX);
            V[e] = x;
        }
        sh[c][r] = x;
    }
    __syncthreads();
    for (int r = threadIdx.x >> 5; r < 32; r += 8) {
        const int i = tj * 32 + r, j = ti * 32 + c;
        if (i < K && j < K && i > j) V[(long long)i * K + j] = sh[r][c];
    }
}

// out(r_g) = sum_C amp exp(-|r_g - R_C|^2 / w^2), terms below 1e-30 |amp| dropped
__global__ void k_gaussian_sum(const double* __restrict__ xyz, int n_atoms, int nx, int ny, int nz,
                               double ox, double oy, double oz, double h, double amp, double inv_w2,
                               double rc, double* __restrict__ out) {
    long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long ng = (long long)nx * ny * nz;
    if (g >= ng) return;
    int ix = (int)(g % nx), iy = (int)((g / nx) % ny), iz = (int)(g / ((long long)nx * ny));
    double x = ox + h * ix, y = oy + h * iy, z = oz + h * iz;
    double s = 0.0;
    for (int a = 0; a < n_atoms; ++a) {
        double dx = x - xyz[3 * a], dy = y - xyz[3 * a + 1], dz = z - xyz[3 * a + 2];
        if (fabs(dx) > rc || fabs(dy) > rc || fabs(dz) > rc) continue;
        s += exp(-dx * dx * inv_w2) * exp(-dy * dy * inv_w2) * exp(-dz * dz * inv_w2);
    }
    out[g] = amp * s;
}

}  // namespace

// Longest list (of a context) that k_collocate_short takes.  Density on the grid
// in us by k_collocate / k_collocate_short, by longest list: FP32 8 terms (465
// atoms, grid 147^3) 286 / 56, 22 380 / 85, 77 82 / 60, 113 135 / 109, 149 221 /
// 176, 173 237 / 247, 242 397 / 461; FP64 8 2731 / 480, 29 312 / 161, 50 404 /
// 453, 64 543 / 570, 77 1082 / 1054.
constexpr int SHORT_F32 = 160, SHORT_F64 = 32;

// Blocks per grid tile: a tile's work grows with the square of its list, and a
// small cluster has few tiles, so tiles are split (collocation by planes,
// quadrature by chunk pairs) until the longest takes at most a third of what an SM
// gets on average (K = 240 in FP64: 343 tiles, the longest lists of 432 terms
// against 170 on average)
void grid_split(Ctx& c, const int* tile_ptr) {
    const int ch = c.p.precision == DFT_PREC_FP64 ? GridCfg<double>::CH : GridCfg<float>::CH;
    double total = 0.0, longest = 0.0;
    c.n_busy = 0;
    for (long long t = 0; t < c.n_tiles; ++t) {
        c.n_busy += tile_ptr[t + 1] > tile_ptr[t];
        const double n = (tile_ptr[t + 1] - tile_ptr[t] + ch - 1) / ch, w = n * (n + 1) / 2;
        total += w;
        longest = std::max(longest, w);
    }
    c.grid_split = c.plane_split = 1;
    while (c.grid_split < 8 && longest / c.grid_split > total / 152.0 / 3.0) c.grid_split *= 2;
    // every block of a plane split reads the tile's part of P again (1470
    // functions, FP32, scalar sums: 2.6 ms with one block per tile, 2.95 with four), so it
    // only keeps a tile from outlasting an SM's share; each thread group needs a plane
    while (c.plane_split < 4 && longest / c.plane_split > total / 152.0) c.plane_split *= 2;
}

void launch_build_tables_for(const Ctx& c, const Fn* fn, int count, int W, double* tab, cudaStream_t s) {
    long long total = (long long)count * 3 * W;
    if (total == 0) return;
    int bs = 256;
    k_build_tables<<<(unsigned)((total + bs - 1) / bs), bs, 0, s>>>(fn, count, W, c.origin[0], c.origin[1],
                                                                    c.origin[2], c.h, tab);
    check_launch("build_tables");
}

void launch_build_tables(const Ctx& c, cudaStream_t s) { launch_build_tables_for(c, c.d_fn, c.Kt, c.tab_w, c.d_tab, s); }

namespace {
template <class Kern>
void allow_smem(Kern k, size_t bytes) {
    DFT_CUDA_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}
}  // namespace

void launch_collocate(const Ctx& c, const double* P, double* n, cudaStream_t s) {
    // contracted functions: collocate their terms with P_t = C^T P C
    if (c.contracted) {
        launch_expand(c, P, c.d_Mt, s);
        P = c.d_Mt;
    }
    auto go = [&](auto kern, unsigned split, int threads, size_t bytes) {
        allow_smem(kern, bytes);
        const dim3 grid((unsigned)c.n_tiles, split);
        kern<<<grid, threads, bytes, s>>>(c.d_fn, c.d_tab, c.tab_w, c.d_tile_ptr, c.d_tile_fn, c.d_tile_order, c.ntile[0],
                                          c.ntile[1], c.n[0], c.n[1], c.n[2], c.Kt, P, n);
    };
    const bool f64 = c.p.precision == DFT_PREC_FP64;
    if (c.tile_max <= (f64 ? SHORT_F64 : SHORT_F32)) {
        if (f64) go(k_collocate_short<double>, 1, 256, 0);
        else go(k_collocate_short<float>, 1, 256, 0);
    } else {
        if (f64) go(k_collocate<double>, c.plane_split, 128, sizeof(CollSmem<double>));
        else go(k_collocate<float>, c.plane_split, 128, sizeof(CollSmem<float>));
    }
    check_launch("collocate");
}

void launch_quadrature(const Ctx& c, const double* v, double* V, cudaStream_t s) {
    // contracted functions: the terms' matrix, then V = C V_t C^T
    double* Vq = c.contracted ? c.d_Mt : V;
    const int K = c.Kt;
    DFT_CUDA_CHECK(cudaMemsetAsync(Vq, 0, sizeof(double) * (size_t)K * K, s));
    auto go = [&](auto kern, size_t bytes) {
        allow_smem(kern, bytes);
        if (c.n_busy == 0) return;
        kern<<<dim3((unsigned)c.n_busy, c.grid_split), 128, bytes, s>>>(c.d_fn, c.d_tab, c.tab_w, c.d_tile_ptr, c.d_tile_fn, c.d_tile_order, c.ntile[0],
                                                     c.ntile[1], c.n[0], c.n[1], c.n[2], K, c.h * c.h * c.h, v, Vq);
    };
    if (c.p.precision == DFT_PREC_FP64) go(k_quadrature<double>, sizeof(QuadSmem<double>));
    else go(k_quadrature<float>, sizeof(QuadSmem<float>));
    const long long nb = (K + 31) / 32;
    k_fixed_to_double<<<(unsigned)(nb * (nb + 1) / 2), 256, 0, s>>>(K, Vq);
    check_launch("quadrature", 2);
    if (c.contracted) launch_contract(c, c.d_Mt, V, s);
}

void launch_gaussian_sum(const Ctx& c, double amp, double width, double* out, cudaStream_t s) {
    // exp(-r^2/w^2) < 1e-30 beyond r = w sqrt(69.1)
    double rc = width * 8.32;
    int bs = 256;
    k_gaussian_sum<<<(unsigned)((c.ng + bs - 1) / bs), bs, 0, s>>>(c.d_xyz, c.n_atoms, c.n[0], c.n[1], c.n[2],
                                                                  c.origin[0], c.origin[1], c.origin[2], c.h,
                                                                  amp, 1.0 / (width * width), rc, out);
    check_launch("gaussian_sum");
}

}  // namespace dft
