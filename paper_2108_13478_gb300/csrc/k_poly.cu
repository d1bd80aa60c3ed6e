// Evaluation of the Chebyshev expansion (Supp. B) with about 2 sqrt(2 N_C)
// matrix products instead of 3/2 N_C: the grouping of matrix polynomials of
// Paterson and Stockmeyer (SIAM J. Comput. 2, 60 (1973)) in the Chebyshev
// form of Liang, Baer, Saravanan, Shao, Bell and Head-Gordon (J. Comput.
// Phys. 194, 575 (2004)).  With "babies" T_r, r < s, and "giants"
// G_q = T_{qs}, q <= Q = (N_C - 1) / s (T_l short for T_l(H_N)):
//
//   rho = sum_l a_l T_l = C_0 + sum_{q=1..Q} G_q C_q,  C_q = sum_{r<s} c_qr T_r,
//   c from T_{qs+r} = 2 T_{qs} T_r - T_{qs-r}, top down: c_q0 = a_{qs},
//   c_qr = 2 a_{qs+r} with a_{qs-r} -= a_{qs+r};
//   m_{qs+r} = Tr T_{qs+r} = 2 <G_q, T_r> - m_{qs-r}  (moments without a product).
//
// The babies come by the three-term recurrence, one product after the other:
// by doubling (T_{2m} = 2 T_m^2 - I) their rounding errors no longer act as a
// shift of the energies, and in a basis with a well-conditioned overlap P was
// off by 70 times as much.  The giants come by doubling, G_{m+j} = 2 G_m G_j -
// G_{m-j}, m products per launch, with no such loss ("direct" plan).  Where the
// workspace cannot hold the giants, they roll in two buffers and the sum is
// taken by Clenshaw's recurrence in T_s, b_q = C_q + 2 T_s b_{q+1} - b_{q+2},
// rho = C_0 + T_s b_1 - b_2 ("Clenshaw" plan: same number of products, one
// per launch).
//
// The FP64 products run on the FP64 pipe (2 FMA per SM per clock on GB300,
// the limit of every kernel here).  All operands are symmetric polynomials
// of H_N, so products are formed on upper tiles and mirrored.  Whole density
// matrix at tail 1e-10 (N_C ~ 2900), the three-term recurrence with full
// products before and this now: K = 80 133 -> 4.7 ms, K = 370 560 -> 14.2 ms,
// error against an exact eigensolve 6e-14 relative on both sides.
#include "dft_internal.cuh"
#include "ps_plan.cuh"

#include <algorithm>
#include <cmath>

namespace dft {
namespace {

// upper tile t of an nb x nb tile grid, row by row -> (i, j), j >= i
__device__ __forceinline__ void upper_tile(int t, int nb, int& i, int& j) {
    i = 0;
    while (t >= nb - i) {
        t -= nb - i;
        ++i;
    }
    j = i + t;
}

// out_y = alpha sum_{f_y <= p < f_{y+1}} A_p B_p - prev_y on the upper TB x TB
// tiles, mirrored; prev: none, a matrix (may be out itself) or the identity.
// One tile per block of 128 threads (2 x 4 sums each; 1 x 2 at TB = 16):
// the FP64 pipe needs one warp per scheduler with a few independent FMAs, so
// small tiles cost nothing and spread a small K over the SMs.  32 x 32 tiles
// read 16 bytes per 32 FMA from L2.
template <int TB>
__global__ void __launch_bounds__(128) k_ps_prod(int K, Ps64Items it, double alpha,
                                                                          double limit, int* __restrict__ flags) {
    constexpr int KS = 32;
    constexpr int NT = 128;                          // four warps: one for each quarter of the SM's FP64 pipe
    constexpr int MR = TB == 32 ? 2 : 1, MC = TB == 32 ? 4 : 2;   // sums per thread
    constexpr int TX = TB / MC;                      // threads along a row
    __shared__ double As[KS][TB + 1];
    __shared__ double Bs[KS][TB + 1];
    const int nb = (K + TB - 1) / TB;
    int ti, tj;
    upper_tile(blockIdx.x, nb, ti, tj);
    const int m0 = ti * TB, n0 = tj * TB;
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    double acc[MR][MC] = {};
    const int y = blockIdx.y;
    for (int p = it.first[y]; p < it.first[y + 1]; ++p) {
        const double* __restrict__ A = it.A[p];
        const double* __restrict__ B = it.B[p];
        for (int k0 = 0; k0 < K; k0 += KS) {
            for (int e = threadIdx.x; e < TB * KS; e += NT) {
                const int kk = e % KS, mm = e / KS;
                As[kk][mm] = (m0 + mm < K && k0 + kk < K) ? A[(long long)(m0 + mm) * K + k0 + kk] : 0.0;
                const int nn = e % TB, kb = e / TB;
                Bs[kb][nn] = (n0 + nn < K && k0 + kb < K) ? B[(long long)(k0 + kb) * K + n0 + nn] : 0.0;
            }
            __syncthreads();
#pragma unroll 8
            for (int kk = 0; kk < KS; ++kk) {
                double a[MR], b[MC];
#pragma unroll
                for (int i = 0; i < MR; ++i) a[i] = As[kk][ty + (TB / MR) * i];
#pragma unroll
                for (int j = 0; j < MC; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
                for (int i = 0; i < MR; ++i)
#pragma unroll
                    for (int j = 0; j < MC; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
            __syncthreads();
        }
    }
    static_assert(KS >= TB, "the mirror is staged in As");
    const double* prev = it.prev[y];
    double* out = it.out[y];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < MR; ++i) {
        const int lm = ty + (TB / MR) * i, gm = m0 + lm;
#pragma unroll
        for (int j = 0; j < MC; ++j) {
            const int ln = tx + TX * j, gn = n0 + ln;
            double x = alpha * acc[i][j];
            if (gm < K && gn < K) {
                const long long e = (long long)gm * K + gn;
                if (prev) x -= prev[e];
                else if (it.ident[y] && gm == gn) x -= 1.0;
                out[e] = x;
                bad |= !(fabs(x) <= limit);
            }
            As[ln][lm] = x;
        }
    }
    if (bad && limit > 0.0) atomicExch(&flags[FLAG_SPECTRUM], 1);
    if (ti == tj) return;
    __syncthreads();
    for (int e = threadIdx.x; e < TB * TB; e += NT) {
        const int r = e / TB, c = e % TB;
        if (n0 + r < K && m0 + c < K) out[(long long)(n0 + r) * K + m0 + c] = As[r][c];
    }
}

// out_q = sp prev_q + sc sum_{r<s} c_qr T_r (T_0 = I) for NQ values of q at
// once, upper 32 x 32 tiles mirrored; T_1 .. T_{s-1} in T[1..]
constexpr int PS_NQ = 8;
__global__ void __launch_bounds__(256) k_ps_combine(int K, int s, PsList T, Ps64Out out, int q0, int nq,
                                                    const double* __restrict__ c, double sp, double sc) {
    __shared__ double sh[32][33];
    const int nb = (K + 31) / 32;
    int ti, tj;
    upper_tile(blockIdx.x, nb, ti, tj);
    const int qb = blockIdx.y * PS_NQ, n = min(PS_NQ, nq - qb);
    const int lc = threadIdx.x & 31, lr0 = threadIdx.x >> 5;   // rows lr0 + 8 u
    const int gc = tj * 32 + lc;
    double acc[4][PS_NQ];
    bool in[4];
    long long e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int gr = ti * 32 + lr0 + 8 * u;
        in[u] = gr < K && gc < K;
        e[u] = in[u] ? (long long)gr * K + gc : 0;
#pragma unroll
        for (int q = 0; q < PS_NQ; ++q) acc[u][q] = (gr == gc && q < n) ? c[(long long)(q0 + qb + q) * s] : 0.0;
    }
    for (int r = 1; r < s; ++r) {
        const double* __restrict__ t = T.p[r];
        double x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = in[u] ? t[e[u]] : 0.0;
#pragma unroll
        for (int q = 0; q < PS_NQ; ++q) {
            if (q >= n) break;
            const double cq = c[(long long)(q0 + qb + q) * s + r];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u][q] = fma(cq, x[u], acc[u][q]);
        }
    }
#pragma unroll
    for (int q = 0; q < PS_NQ; ++q) {
        if (q >= n) break;
        double* o = out.p[qb + q];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            double x = sc * acc[u][q];
            if (in[u]) {
                if (sp != 0.0) x = fma(sp, o[e[u]], x);
                o[e[u]] = x;
            }
            sh[lc][lr0 + 8 * u] = x;
        }
        if (ti == tj) continue;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int gr = tj * 32 + lr0 + 8 * u, gcc = ti * 32 + lc;
            if (gr < K && gcc < K) o[(long long)gr * K + gcc] = sh[lr0 + 8 * u][lc];
        }
    }
}

// rho = base + sum of the np partial products (upper tiles), mirrored
__global__ void __launch_bounds__(256) k_ps_add(int K, int np, Ps64Out part, const double* base, double* rho) {
    __shared__ double sh[32][33];
    const int nb = (K + 31) / 32;
    int ti, tj;
    upper_tile(blockIdx.x, nb, ti, tj);
    const int lc = threadIdx.x & 31, lr0 = threadIdx.x >> 5;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int gr = ti * 32 + lr0 + 8 * u, gc = tj * 32 + lc;
        double x = 0.0;
        if (gr < K && gc < K) {
            const long long e = (long long)gr * K + gc;
            for (int p = 0; p < np; ++p) x += part.p[p][e];
            x += base[e];
            rho[e] = x;
        }
        sh[lc][lr0 + 8 * u] = x;
    }
    if (ti == tj) return;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int gr = tj * 32 + lr0 + 8 * u, gc = ti * 32 + lc;
        if (gr < K && gc < K) rho[(long long)gr * K + gc] = sh[lr0 + 8 * u][lc];
    }
}

// partial Gram sums <G_q, T_r> over the upper 32 x 32 tiles blockIdx.x,
// + gridDim.x, ... (off-diagonal elements twice); 64 x 32 pairs per block of
// 256 threads, 4 x 2 each
__global__ void __launch_bounds__(256) k_ps_gram(int K, PsList G, int nq, PsList T, int s, double* __restrict__ part) {
    __shared__ double g[32][65], t[32][33];
    const int nb = (K + 31) / 32, nt = nb * (nb + 1) / 2;
    const int qb = blockIdx.y * 64, rb = blockIdx.z * 32;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[4][2] = {};
    int ni = 0;   // live sums per thread along q
#pragma unroll
    for (int i = 0; i < 4; ++i) ni += qb + ty + 16 * i < nq;
    for (int tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        int ti, tj;
        upper_tile(tile, nb, ti, tj);
        for (int row = ti * 32; row < min(K, ti * 32 + 32); ++row) {
            __syncthreads();
            for (int e = threadIdx.x; e < 32 * 64; e += 256) {
                const int c = e & 31, m = e >> 5, gc = tj * 32 + c;
                const double w = gc >= K || gc < row ? 0.0 : (gc == row ? 1.0 : 2.0);
                g[c][m] = (w != 0.0 && qb + m < nq) ? w * G.p[qb + m][(long long)row * K + gc] : 0.0;
                if (m < 32) t[c][m] = (gc < K && rb + m < s && rb + m > 0) ? T.p[rb + m][(long long)row * K + gc] : 0.0;
            }
            __syncthreads();
            if (ni == 0) continue;
#pragma unroll 4
            for (int c = 0; c < 32; ++c) {
                double a[4], b[2];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = g[c][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < 2; ++j) b[j] = t[c][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= ni) break;
#pragma unroll
                    for (int j = 0; j < 2; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int q = qb + ty + 16 * i;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = rb + tx + 16 * j;
            if (q < nq && r < s) part[((long long)blockIdx.x * nq + q) * s + r] = acc[i][j];
        }
    }
}

// D[q][r] = sum of the partials in a fixed order
__global__ void k_ps_gram_sum(int nsplit, int n, const double* __restrict__ part, double* __restrict__ D) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double x = 0.0;
    for (int p = 0; p < nsplit; ++p) x += part[(long long)p * n + e];
    D[e] = x;
}

// traces of a list of matrices, one block each
__global__ void __launch_bounds__(128) k_ps_trace(int K, PsList L, double* __restrict__ out, int stride) {
    __shared__ double red[4];
    const double* X = L.p[blockIdx.x];
    double x = 0.0;
    for (int i = threadIdx.x; i < K; i += 128) x += X[(long long)i * K + i];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) out[(long long)blockIdx.x * stride] = red[0] + red[1] + red[2] + red[3];
}

// m_l, l < n_c, from D: row 0 the traces of the babies (m_0 = K), row q the
// Gram sums of G_q with its trace in column 0
__global__ void __launch_bounds__(256) k_ps_moments(int K, int n_c, int s, int Q, const double* __restrict__ D,
                                                    double* mom) {
    for (int r = threadIdx.x; r < s && r < n_c; r += 256) mom[r] = r == 0 ? (double)K : D[r];
    for (int q = 1; q <= Q; ++q) {
        __syncthreads();
        for (int r = threadIdx.x; r < s && q * s + r < n_c; r += 256) {
            const double d = D[(long long)q * s + r];
            mom[q * s + r] = r == 0 ? d : 2.0 * d - mom[q * s - r];
        }
    }
}

// c_qr from a_l (the header's top-down elimination), times down for q >= 1;
// work holds (Q + 1) s doubles
__global__ void __launch_bounds__(256) k_ps_coefs(int n_c, int s, int Q, double down, const double* __restrict__ a,
                                                  double* c, double* work) {
    const int n = (Q + 1) * s;
    for (int l = threadIdx.x; l < n; l += 256) work[l] = l < n_c ? a[l] : 0.0;
    for (int q = Q; q >= 0; --q) {
        __syncthreads();
        for (int r = threadIdx.x; r < s; r += 256) {
            const double x = work[q * s + r];
            c[q * s + r] = q == 0 ? x : down * (r == 0 ? x : 2.0 * x);
            if (r > 0 && q > 0) work[q * s - r] -= x;
        }
    }
}

inline int upper_tiles(int K, int tb) {
    const int nb = (K + tb - 1) / tb;
    return nb * (nb + 1) / 2;
}

}  // namespace

// Baby count and plan for n_c terms on nslot buffers: s + 2 Q products, Q =
// (n_c - 1) / s.  Direct: s - 1 babies (T_1 = H_N is not counted), the
// giants G_2 .. G_Q and PS_CQ buffers for the C_q and the partial sums of the
// weighted products.  Clenshaw: the babies T_2 .. T_s and nroll buffers.
// seq: time of a product that has a launch to itself, par: its share of a
// launch of many; babies and all products of a Clenshaw plan are of the first
// kind, so a small matrix takes fewer babies and more giants.  Below PS_MIN_S
// babies the giants' rounding errors would outgrow the recurrence's.
PsPlan ps_plan(int n_c, int nslot, double seq, double par, int nroll) {
    PsPlan p;
    p.n_c = n_c;
    double best = 1e300;
    const int smax = std::min(n_c, PS_MAX_S);
    for (int pass = 0; pass < 2 && best > 1e299; ++pass)   // second pass: fewer babies than PS_MIN_S
        for (int s = pass == 0 ? std::min(PS_MIN_S, smax) : 1; s <= smax; ++s) {
            const int Q = (n_c - 1) / s;
            const int need_d = (s - 1) + std::max(0, Q - 1) + (Q > 0 ? PS_CQ + 1 : 0);
            const int need_c = (s - 1) + nroll;
            if (need_d <= nslot && Q <= PS_MAX_Q && s * seq + 2 * Q * par < best) {
                best = s * seq + 2 * Q * par;
                p.s = s;
                p.Q = Q;
                p.direct = true;
            }
            if (need_c <= nslot && (s + 2 * Q) * seq < best) {
                best = (s + 2 * Q) * seq;
                p.s = s;
                p.Q = Q;
                p.direct = false;
            }
        }
    return p;
}

void launch_ps_moments(int K, const PsPlan& p, const double* D, double* mom, cudaStream_t s) {
    k_ps_moments<<<1, 256, 0, s>>>(K, p.n_c, p.s, p.Q, D, mom);
    check_launch("ps_moments");
}

void launch_ps_coefs(const PsPlan& p, const double* a, double* c, double* work, cudaStream_t s) {
    k_ps_coefs<<<1, 256, 0, s>>>(p.n_c, p.s, p.Q, (double)p.down, a, c, work);
    check_launch("ps_coefs");
}

// ---- FP64 ----
namespace {

struct Ps64 {
    const Ctx& c;
    const PsPlan& p;
    cudaStream_t st;
    const double* baby(int r) const { return r == 1 ? c.d_H : c.ps_slot[r - 2]; }   // r >= 1
    // direct: babies T_2 .. T_s, giants G_2 .. G_Q, then the C buffers
    const double* giant(int q) const { return q == 1 ? baby(p.s) : c.ps_slot[p.s - 1 + q - 2]; }
    double* cbuf(int i) const { return c.ps_slot[p.s - 1 + std::max(0, p.Q - 1) + i]; }

    void products(const Ps64Items& it, int n, double alpha, double limit) const {
        const int big = upper_tiles(c.K, 32);
        // 32 x 32 tiles unless they would leave SMs idle: 16 x 16 tiles give
        // four times the blocks (K = 80: 15 against 6 per product)
        if ((long long)big * n >= 2 * 152) {
            k_ps_prod<32><<<dim3(big, n), 128, 0, st>>>(c.K, it, alpha, limit, c.d_flags);
        } else {
            k_ps_prod<16><<<dim3(upper_tiles(c.K, 16), n), 128, 0, st>>>(c.K, it, alpha, limit, c.d_flags);
        }
        check_launch("ps_prod");
    }
    // X_{m+1} .. X_{min(2m, top)} from X_1 .. X_m by doubling, for X given by get
    template <class Get>
    void doubling(int top, Get&& get, double last_limit) const {
        for (int m = 1; m < top; m *= 2) {
            for (int j0 = 1; j0 <= std::min(m, top - m); j0 += PS_MAX_ITEMS) {
                const int n = std::min(PS_MAX_ITEMS, std::min(m, top - m) - j0 + 1);
                Ps64Items it{};
                double lim = 4.0;
                for (int y = 0; y < n; ++y) {
                    const int j = j0 + y;
                    it.A[y] = get(m);
                    it.B[y] = get(j);
                    it.prev[y] = m - j > 0 ? get(m - j) : nullptr;
                    it.ident[y] = m == j;
                    it.out[y] = const_cast<double*>(get(m + j));
                    it.first[y] = y;
                    if (m + j == top) lim = last_limit;
                }
                it.first[n] = n;
                products(it, n, 2.0, lim);
            }
        }
    }
    // the spectrum check beyond the last giant (ps_check), in slots s0 and s0 + 1
    void check(int s0) const {
        const PsCheck k = ps_check(p, true);
        const double* cur = baby(std::max(1, k.baby));
        for (int i = 0, l = k.baby; i < k.doublings; ++i) {
            // T_{2l} = 2 T_l^2 - I or T_{2l+1} = 2 T_l T_{l+1} - T_1
            Ps64Items it{};
            it.A[0] = cur;
            it.B[0] = k.odd ? baby(l + 1) : cur;
            it.prev[0] = k.odd ? baby(1) : nullptr;
            it.ident[0] = k.odd ? 0 : 1;
            it.out[0] = c.ps_slot[s0 + (i & 1)];
            it.first[1] = 1;
            l *= 2;
            products(it, 1, 2.0, i + 1 == k.doublings ? growth_limit(l + k.odd, p.n_c) : 4.0);
            cur = it.out[0];
        }
    }
    void gram(int q0, int nq, const PsList& G, double* D) const {
        const int s = p.s;
        PsList T{};
        for (int r = 1; r < s; ++r) T.p[r] = baby(r);
        const int nt = upper_tiles(c.K, 32);
        const int nsplit = (int)std::max<long long>(1, std::min<long long>({(long long)nt, 2 * 152LL, c.gram_cap / ((long long)nq * s)}));
        if ((long long)nq * s > c.gram_cap) throw Error(DFT_EINTERNAL, "Gram partials exceed their buffer");
        k_ps_gram<<<dim3(nsplit, (nq + 63) / 64, (s + 31) / 32), 256, 0, st>>>(c.K, G, nq, T, s, c.d_gram);
        k_ps_gram_sum<<<(nq * s + 255) / 256, 256, 0, st>>>(nsplit, nq * s, c.d_gram, D + (long long)q0 * s);
        k_ps_trace<<<nq, 128, 0, st>>>(c.K, G, D + (long long)q0 * s, s);
        check_launch("ps_gram", 3);
    }
};

}  // namespace

// babies, giants and m_l; the plan is kept in c.ps
void ps64_pass1(Ctx& c, cudaStream_t st) {
    const double waves = upper_tiles(c.K, 16) / 152.0;
    c.ps = ps_plan(c.n_c_cur, (int)c.ps_slot.size(), std::ceil(waves), waves, 2);
    const PsPlan& p = c.ps;
    Ps64 e{c, p, st};
    const int s = p.s, Q = p.Q;
    // T_s is needed as soon as there is a giant
    const int top = Q > 0 ? s : s - 1;
    for (int r = 1; r < top; ++r) {
        Ps64Items it{};
        it.A[0] = c.d_H;
        it.B[0] = e.baby(r);
        it.prev[0] = r > 1 ? e.baby(r - 1) : nullptr;
        it.ident[0] = r == 1;
        it.out[0] = const_cast<double*>(e.baby(r + 1));
        it.first[1] = 1;
        e.products(it, 1, 2.0, r + 1 == s && Q == 1 ? growth_limit(s, p.n_c) : 4.0);
    }
    double* D = c.d_wk;   // (Q + 1) s doubles, consumed before the moment weights are written there
    if (s > 1) {
        PsList L{};
        for (int r = 1; r < s; ++r) L.p[r - 1] = e.baby(r);
        k_ps_trace<<<s - 1, 128, 0, st>>>(c.K, L, D + 1, 1);
        check_launch("ps_trace");
    }
    if (p.direct) {
        e.doubling(Q, [&](int q) { return e.giant(q); }, growth_limit(Q * s, p.n_c));
        if (Q > 0)
            for (int q0 = 1; q0 <= Q; q0 += PS_MAX_S) {
                const int nq = std::min(PS_MAX_S, Q - q0 + 1);
                PsList G{};
                for (int q = 0; q < nq; ++q) G.p[q] = e.giant(q0 + q);
                e.gram(q0, nq, G, D);
            }
    } else {
        double* roll[2] = {c.ps_slot[s - 1], c.ps_slot[s]};
        const double* Ts = e.baby(s);
        const double *prev = nullptr, *cur = Ts;
        for (int q = 1; q <= Q; ++q) {
            PsList G{};
            G.p[0] = cur;
            e.gram(q, 1, G, D);
            if (q == Q) break;
            Ps64Items it{};
            it.A[0] = Ts;
            it.B[0] = cur;
            it.prev[0] = q > 1 ? prev : nullptr;
            it.ident[0] = q == 1;
            // G_{q+1} over G_{q-1} (T_s itself stays)
            it.out[0] = q > 2 ? const_cast<double*>(prev) : roll[q - 1];
            it.first[1] = 1;
            e.products(it, 1, 2.0, q + 1 == Q ? growth_limit(Q * s, p.n_c) : 4.0);
            prev = cur;
            cur = it.out[0];
        }
    }
    e.check(p.direct ? s - 1 + std::max(0, Q - 1) : s - 1);   // the buffers behind the giants, or those they rolled in
    launch_ps_moments(c.K, p, D, c.d_mom, st);
}

// rho = sum_l a_l T_l with the coefficients in c.d_coef
void ps64_pass2(Ctx& c, cudaStream_t st) {
    const PsPlan& p = c.ps;
    Ps64 e{c, p, st};
    const int s = p.s, Q = p.Q, K = c.K;
    double* cf = c.d_coef + c.n_c_cur;   // behind a_l: (Q + 1) s <= 2 n_c doubles, then as many of scratch
    launch_ps_coefs(p, c.d_coef, cf, cf + (long long)(Q + 1) * s, st);
    PsList T{};
    for (int r = 1; r < s; ++r) T.p[r] = e.baby(r);
    const int nt = upper_tiles(K, 32);
    auto combine = [&](int q0, int nq, const Ps64Out& o, double sp, double sc) {
        k_ps_combine<<<dim3(nt, (nq + PS_NQ - 1) / PS_NQ), 256, 0, st>>>(K, s, T, o, q0, nq, cf, sp, sc);
        check_launch("ps_combine");
    };
    Ps64Out o{};
    if (p.direct || Q == 0) {
        o.p[0] = c.d_rho;
        combine(0, 1, o, 0.0, 1.0);
        const int spare = (int)c.ps_slot.size() - (s - 1) - std::max(0, Q - 1);   // C buffers and partial sums
        for (int q0 = 1; q0 <= Q;) {
            // as many partial sums as fill the SMs, the rest of the buffers for C_q
            const int np_want = std::max(1, std::min(4 * 152 / nt + 1, Q - q0 + 1));
            const int np = std::max(1, std::min({np_want, spare / 4, PS_MAX_ITEMS}));
            const int nq = std::min({Q - q0 + 1, spare - np, PS_MAX_ITEMS});
            Ps64Out cq{};
            for (int q = 0; q < nq; ++q) cq.p[q] = e.cbuf(q);
            combine(q0, nq, cq, 0.0, 1.0);
            Ps64Items it{};
            Ps64Out part{};
            const int npu = std::min(np, nq);
            for (int q = 0; q < nq; ++q) {
                it.A[q] = e.giant(q0 + q);
                it.B[q] = cq.p[q];
            }
            for (int y = 0; y < npu; ++y) {
                it.first[y] = (int)((long long)nq * y / npu);
                it.out[y] = part.p[y] = e.cbuf(nq + y);
            }
            it.first[npu] = nq;
            e.products(it, npu, 1.0, 0.0);
            k_ps_add<<<nt, 256, 0, st>>>(K, npu, part, c.d_rho, c.d_rho);
            check_launch("ps_add");
            q0 += nq;
        }
        return;
    }
    // Clenshaw in T_s: two buffers, b_{q+1} and b_{q+2} (turned into b_{q+2} - C_q, then b_q)
    double* b1 = c.ps_slot[s - 1];
    double* b2 = c.ps_slot[s];
    const double* Ts = e.baby(s);
    o.p[0] = b1;
    combine(Q, 1, o, 0.0, 1.0);
    bool have2 = false;
    for (int q = Q - 1; q >= 0; --q) {
        o.p[0] = b2;
        combine(q, 1, o, have2 ? 1.0 : 0.0, -1.0);
        have2 = true;
        Ps64Items it{};
        it.A[0] = Ts;
        it.B[0] = b1;
        it.prev[0] = b2;
        it.out[0] = q > 0 ? b2 : c.d_rho;
        it.first[1] = 1;
        e.products(it, 1, q > 0 ? 2.0 : 1.0, 0.0);
        std::swap(b1, b2);
    }
}

}  // namespace dft
