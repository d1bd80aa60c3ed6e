// Kernel arguments and limits of the grouped Chebyshev evaluation (k_poly.cu,
// k_poly_tc.cu); the plan itself (PsPlan) is declared with the context.
#pragma once

#include "dft_internal.cuh"

#include <cmath>

namespace dft {

constexpr int PS_MAX_S = 128;      // babies per plan, matrices per Gram or combination launch
constexpr int PS_MIN_S = 24;
constexpr int PS_MAX_Q = 1024;     // giants of a direct plan
constexpr int PS_MAX_ITEMS = 32;   // products per launch
constexpr int PS_CQ = 8;           // buffers a direct plan keeps for C_q and partial sums

struct PsList {
    const double* p[PS_MAX_S];
};
struct Ps64Out {
    double* p[PS_MAX_ITEMS];
};
// out_y = alpha sum_{first[y] <= q < first[y + 1]} A_q B_q - prev_y
struct Ps64Items {
    const double* A[PS_MAX_ITEMS];
    const double* B[PS_MAX_ITEMS];
    const double* prev[PS_MAX_ITEMS];
    double* out[PS_MAX_ITEMS];
    int first[PS_MAX_ITEMS + 1];
    int ident[PS_MAX_ITEMS];
};

// Spectrum check.  The three-term recurrence refuses a spectrum outside the
// interval when an element of T_{n_c - 1} exceeds 4.  The iterates grow like
// cosh(l t) there: the bound at l that corresponds to 4 at the last term
inline double growth_limit(int l, int n_c) {
    if (l >= n_c - 1 || n_c < 3) return 4.0;
    return std::cosh(std::acosh(4.0) * (double)l / (n_c - 1));
}
// The last giant T_{Qs} stands for the last term where its order is at least
// 9/10 of the last's (any Q >= 9); otherwise, and where no giants are formed,
// a baby T_b, b = (n_c - 1) / 2^i <= s, is doubled i times.  A single product
// then gives T_{n_c - 1} itself (an outlier whose elements are a tenth of its
// cosh is still below 1 at T_24 when it reaches 4 at T_39), more products an
// order within 1 / b of it.  Each doubling multiplies rounding errors by up
// to 4; one of 1e-5 stays below the limit through 8 of them.
struct PsCheck {
    int baby = 0, doublings = 0;   // 0: nothing beyond the last giant
    int odd = 0;                   // the single product is T_b T_{b+1}
};
inline PsCheck ps_check(const PsPlan& p, bool giants) {
    PsCheck c;
    const int n = p.n_c - 1;
    if (p.Q == 0 || (giants && 10LL * p.Q * p.s >= 9LL * n)) return c;
    while ((n >> c.doublings) > p.s) ++c.doublings;
    c.baby = n >> c.doublings;
    c.odd = c.doublings == 1 && n % 2 == 1 && c.baby < p.s;
    if (c.doublings > 8) c.doublings = 8;
    return c;
}

// ---- split 16-bit path (k_poly_tc.cu) ----
struct PstList {
    const void* p[PS_MAX_S];
};
struct PstOut {
    void* p[PS_MAX_ITEMS];
};

}  // namespace dft
