// Chebyshev engine (Supp. B): expansion coefficients of the Fermi-Dirac
// function, Chebyshev moments, the chemical potential by bisection on the
// electron count (Eq. 2.8).
#include "dft_internal.cuh"

#include <algorithm>

namespace dft {
namespace {

__device__ __forceinline__ double fermi(double e, double mu, double beta) {
    const double t = 0.5 * beta * (e - mu);
    // beyond |t| = 40, 1 - |tanh t| < 1e-34: f is 0 or 1 in FP64, and the
    // tanh (dozens of operations on GB300's narrow FP64 pipe) is skipped for
    // the many nodes far from mu
    if (t > 40.0) return 0.0;
    if (t < -40.0) return 1.0;
    return 0.5 * (1.0 - tanh(t));
}

// cos_tab[j] = cos(pi j / (2M)), j < 4M: cos(l th_k) with th_k = pi (k + 1/2) / M
// is cos_tab[(l (2k+1)) mod 4M]
__global__ void k_cos_table(int M, double* c) {
    long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < 4LL * M) c[j] = cospi((double)j / (2.0 * M));
}

// f at the M Chebyshev-Gauss nodes mapped to [E_min, E_max]
__global__ void k_fermi_nodes(int M, const double* __restrict__ c, const double* __restrict__ scal, double beta,
                              double mu_o, int use_o, double* __restrict__ fk) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    double emin = scal[SCAL_EMIN], emax = scal[SCAL_EMAX];
    double eb = 0.5 * (emax + emin), de = 0.5 * (emax - emin);
    double mu = use_o ? mu_o : scal[SCAL_MU];
    fk[k] = fermi(eb + de * c[2 * k + 1], mu, beta);
}

// cos(pi j / (2M)), 0 <= j < 4M, from the first quarter wave c[0 .. M]
__device__ __forceinline__ double quarter_cos(const double* c, int j, int M) {
    if (j > 2 * M) j = 4 * M - j;
    return j <= M ? c[j] : -c[2 * M - j];
}

// The nodes' energies fall with k: f_k = 0 below k0 and 1 from k1 on (in FP64,
// |t| > 40, see fermi); between them lies the window in which f varies, about
// 80 kT of the spectrum
__device__ __forceinline__ int first_below(const double* c, int M, double eb, double de, double e) {
    int a = 0, b = M;   // first k with energy <= e
    while (a < b) {
        const int m = (a + b) >> 1;
        if (eb + de * c[2 * m + 1] <= e) b = m;
        else a = m + 1;
    }
    return a;
}
__device__ __forceinline__ void fermi_window(const double* c, int M, double eb, double de, double mu, double beta,
                                             int& k0, int& k1) {
    k0 = first_below(c, M, eb, de, mu + 81.0 / beta);
    k1 = first_below(c, M, eb, de, mu - 81.0 / beta);
}

// a_l = (2 - delta_l0)/M sum_k f_k cos(l th_k)  (DCT-II of the node values),
// one warp per coefficient, lanes over the nodes of the window; cos(l th_k) is
// cos_tab[(l (2k+1)) mod 4M], read from a quarter wave of the table in shared
// memory (SH; M <= DCT_SH_M) or from the whole table in L2.  The nodes with f = 1
// sum in closed form, sum_{k >= k1} cos(l (k + 1/2) h) = -sin(l k1 h) /
// (2 sin(l h / 2)), h = pi / M (all nodes: 0.29 ms at n_c = 2850, M = 11400).
constexpr int DCT_SH_M = 28000;
template <bool SH>
__global__ void __launch_bounds__(1024) k_dct_coeffs(int n_c, int M, const double* __restrict__ c,
                                                     const double* __restrict__ fk, const double* __restrict__ scal,
                                                     double beta, double mu_o, int use_o, double* __restrict__ a) {
    extern __shared__ double qc[];
    __shared__ int win[2];
    if (SH)
        for (int j = threadIdx.x; j <= M; j += 1024) qc[j] = c[j];
    if (threadIdx.x == 0) {
        const double emin = scal[SCAL_EMIN], emax = scal[SCAL_EMAX];
        fermi_window(c, M, 0.5 * (emax + emin), 0.5 * (emax - emin), use_o ? mu_o : scal[SCAL_MU], beta, win[0], win[1]);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, k0 = win[0], k1 = win[1], m4 = 4 * M;
    for (int l = blockIdx.x * 32 + (threadIdx.x >> 5); l < n_c; l += gridDim.x * 32) {
        int idx = (int)(((long long)l * (2 * (k0 + lane) + 1)) % m4);
        const int step = (int)((64LL * l) % m4);
        double s = 0.0;
        for (int k = k0 + lane; k < k1; k += 32) {
            s = fma(fk[k], SH ? quarter_cos(qc, idx, M) : c[idx], s);
            idx += step;
            if (idx >= m4) idx -= m4;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) {
            if (l == 0) {
                s += (double)(M - k1);
            } else {
                // sin(l k1 h) = -cos(l k1 h + pi / 2): entry 2 l k1 + M of the table
                const int q = (int)((2LL * l * k1 + M) % m4);
                s += (SH ? quarter_cos(qc, q, M) : c[q]) / (2.0 * sinpi((double)l / (2.0 * M)));
            }
            a[l] = (l == 0 ? 1.0 : 2.0) / M * s;
        }
    }
}

// w_k = (1/M) sum_l (2 - delta_l0) m_l cos(l th_k): N(mu) = 2 sum_k f(x_k; mu) w_k;
// one warp per node, lanes over the moments, the table as above
template <bool SH>
__global__ void __launch_bounds__(1024) k_moment_weights(int n_c, int M, const double* __restrict__ c,
                                                         const double* __restrict__ mom, double* __restrict__ wk) {
    extern __shared__ double qc[];
    if (SH) {
        for (int j = threadIdx.x; j <= M; j += 1024) qc[j] = c[j];
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    for (int k = blockIdx.x * 32 + (threadIdx.x >> 5); k < M; k += gridDim.x * 32) {
        const int m4 = 4 * M;
        int idx = (int)((2LL * k + 1) * lane % m4);
        const int step = (int)((2LL * k + 1) * 32 % m4);
        double s = 0.0;
        for (int l = lane; l < n_c; l += 32) {
            s = fma((l == 0 ? 1.0 : 2.0) * mom[l], SH ? quarter_cos(qc, idx, M) : c[idx], s);
            idx += step;
            if (idx >= m4) idx -= m4;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) wk[k] = s / M;
    }
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
    return r;
}

// mu by multisection on N(mu) = N_e over [E_min - 40/beta, E_max + 40/beta]
// (the paper fixes mu through Eq. 2.8 without naming a method).  One launch
// per round: block b evaluates N at point b of MU_PTS + 2 equally spaced ones
// (both ends among them); every block first finds the bracket of its round
// from the counts of the round before, so rounds need no other
// synchronisation.  Nodes outside the window of a point come from the suffix
// sums of the weights (k_suffix).  65-fold narrowing: MU_ROUNDS rounds reach FP64 resolution
// (one block bisecting took 1.2 ms at M = 5624, 2.2 ms at 11400).
// suf[k] = sum_{j >= k} w_j, k <= M: one block, runs of M / 1024 nodes per thread
__global__ void __launch_bounds__(1024) k_suffix(int M, const double* __restrict__ wk, double* __restrict__ suf) {
    __shared__ double tot[1024];
    const int t = threadIdx.x, run = (M + 1023) / 1024, a = min(M, t * run), b = min(M, a + run);
    double s = 0.0;
    for (int k = a; k < b; ++k) s += wk[k];
    tot[t] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o *= 2) {   // inclusive suffix sums of the runs
        const double x = t + o < 1024 ? tot[t + o] : 0.0;
        __syncthreads();
        tot[t] += x;
        __syncthreads();
    }
    s = t + 1 < 1024 ? tot[t + 1] : 0.0;
    if (t == 1023) suf[M] = 0.0;
    for (int k = b - 1; k >= a; --k) {
        s += wk[k];
        suf[k] = s;
    }
}

constexpr int MU_PTS = 64, MU_ROUNDS = 11;
__device__ __forceinline__ double mu_point(double lo, double hi, int i) {
    return i == 0 ? lo : (i == MU_PTS + 1 ? hi : lo + (hi - lo) * ((double)i / (MU_PTS + 1)));
}
// state: two rounds' {lo, hi, counts[MU_PTS + 2]} in turn
constexpr int MU_STATE = MU_PTS + 4;
__device__ void mu_bracket(const double* st, double n_e, double& lo, double& hi) {
    // invariant: N(lo) < n_e <= N(hi) up to rounding; the first point at or above n_e
    int j = MU_PTS + 1;
    for (int i = MU_PTS; i >= 1; --i)
        if (st[2 + i] >= n_e) j = i;
    lo = mu_point(st[0], st[1], j - 1);
    hi = mu_point(st[0], st[1], j);
}
__global__ void __launch_bounds__(256) k_mu_round(int round, int M, const double* __restrict__ c,
                                                  const double* __restrict__ wk, const double* __restrict__ suf,
                                                  double beta, double n_e,
                                                  double* state, double* scal, int* flags) {
    const double emin = scal[SCAL_EMIN], emax = scal[SCAL_EMAX];
    const double eb = 0.5 * (emax + emin), de = 0.5 * (emax - emin);
    const double* prev = state + ((round + 1) & 1) * MU_STATE;
    double* cur = state + (round & 1) * MU_STATE;
    double lo, hi;
    if (round == 0) {
        lo = emin - 40.0 / beta;
        hi = emax + 40.0 / beta;
    } else {
        if (round == 1 && threadIdx.x == 0 && blockIdx.x == 0 && (prev[2] > n_e || prev[2 + MU_PTS + 1] < n_e)) flags[FLAG_MU] = 1;
        mu_bracket(prev, n_e, lo, hi);
    }
    if (round == MU_ROUNDS) {
        if (threadIdx.x == 0) scal[SCAL_MU] = flags[FLAG_MU] ? eb : 0.5 * (lo + hi);
        return;
    }
    const double mu = mu_point(lo, hi, blockIdx.x);
    __shared__ int win[2];
    if (threadIdx.x == 0) fermi_window(c, M, eb, de, mu, beta, win[0], win[1]);
    __syncthreads();
    double s = 0.0;
    for (int k = win[0] + threadIdx.x; k < win[1]; k += 256) s = fma(fermi(eb + de * c[2 * k + 1], mu, beta), wk[k], s);
    s = block_sum<256>(s);
    if (threadIdx.x == 0) {
        s += suf[win[1]];
        cur[2 + blockIdx.x] = 2.0 * s;
        if (blockIdx.x == 0) {
            cur[0] = lo;
            cur[1] = hi;
        }
    }
}

// m_{even} = 2 <Xn,Xn> - m0, m_{odd} = 2 <Xn,Xc> - m1 (T_{2l} = 2T_l^2 - 1,
// T_{2l+1} = 2 T_{l+1} T_l - T_1), partials summed in a fixed order
__global__ void __launch_bounds__(256) k_moment_reduce(int np, const double* __restrict__ part, double* mom,
                                                       int ie, int io, double m0, const double* m1) {
    double s0 = 0.0, s1 = 0.0;
    for (int i = threadIdx.x; i < np; i += 256) {
        s0 += part[2 * i];
        s1 += part[2 * i + 1];
    }
    s0 = block_sum<256>(s0);
    s1 = block_sum<256>(s1);
    if (threadIdx.x == 0) {
        if (ie >= 0) mom[ie] = 2.0 * s0 - m0;
        if (io >= 0) mom[io] = 2.0 * s1 - *m1;
    }
}

inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

void launch_cos_table(int M, double* cos_tab, cudaStream_t s) {
    k_cos_table<<<blocks_for(4LL * M, 256), 256, 0, s>>>(M, cos_tab);
    check_launch("cos_table");
}

// coefficients for l < n_c with M nodes; the node values f_k are staged in
// coef[n_c .. n_c + M), so coef must hold n_c + M doubles
void launch_cheb_coeffs(int n_c, int M, const double* cos_tab, const double* scal, double beta,
                        double mu_override, bool use_override, double* coef, cudaStream_t s) {
    double* fk = coef + n_c;
    k_fermi_nodes<<<blocks_for(M, 256), 256, 0, s>>>(M, cos_tab, scal, beta, mu_override, use_override ? 1 : 0, fk);
    const size_t sh = sizeof(double) * ((size_t)M + 1);
    if (M <= DCT_SH_M) {
        DFT_CUDA_CHECK(cudaFuncSetAttribute(k_dct_coeffs<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sizeof(double) * (DCT_SH_M + 1)));   // the same for all callers: threads set it together
        k_dct_coeffs<true><<<std::min(152, (n_c + 31) / 32), 1024, sh, s>>>(n_c, M, cos_tab, fk, scal, beta, mu_override,
                                                                            use_override ? 1 : 0, coef);
    } else {
        k_dct_coeffs<false><<<(n_c + 31) / 32, 1024, 0, s>>>(n_c, M, cos_tab, fk, scal, beta, mu_override,
                                                             use_override ? 1 : 0, coef);
    }
    check_launch("cheb_coeffs", 2);
}

void launch_moment_weights(int n_c, int M, const double* cos_tab, const double* mom, double* wk, cudaStream_t s) {
    const size_t sh = sizeof(double) * ((size_t)M + 1);
    if (M <= DCT_SH_M) {
        DFT_CUDA_CHECK(cudaFuncSetAttribute(k_moment_weights<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)sizeof(double) * (DCT_SH_M + 1)));   // the same for all callers: threads set it together
        k_moment_weights<true><<<std::min(152, (M + 31) / 32), 1024, sh, s>>>(n_c, M, cos_tab, mom, wk);
    } else {
        k_moment_weights<false><<<(M + 31) / 32, 1024, 0, s>>>(n_c, M, cos_tab, mom, wk);
    }
    check_launch("moment_weights");
}

// state: MU_STATE_DOUBLES of scratch
void launch_mu_bisect(int M, const double* cos_tab, double* wk, double beta, double n_e, double* state,
                      double* scal, int* flags, cudaStream_t s) {
    static_assert(2 * MU_STATE <= MU_STATE_DOUBLES, "scratch of the mu search");
    double* suf = wk + M;   // M + 1 doubles behind the weights
    k_suffix<<<1, 1024, 0, s>>>(M, wk, suf);
    for (int r = 0; r <= MU_ROUNDS; ++r)
        k_mu_round<<<r < MU_ROUNDS ? MU_PTS + 2 : 1, 256, 0, s>>>(r, M, cos_tab, wk, suf, beta, n_e, state, scal, flags);
    check_launch("mu_rounds", MU_ROUNDS + 2);
}

void launch_moment_reduce(int nparts, const double* part, double* mom, int idx_even, int idx_odd, double m0,
                          const double* m1, cudaStream_t s) {
    k_moment_reduce<<<1, 256, 0, s>>>(nparts, part, mom, idx_even, idx_odd, m0, m1);
    check_launch("moment_reduce");
}

}  // namespace dft
