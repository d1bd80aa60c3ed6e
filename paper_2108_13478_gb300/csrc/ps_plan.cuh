// Kernel arguments and limits of the grouped Chebyshev evaluation (k_poly.cu,
// k_poly_tc.cu); the plan itself (PsPlan) is declared with the context.
#pragma once

#include "dft_internal.cuh"

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


// ---- split 16-bit path (k_poly_tc.cu) ----
struct PstList {
    const void* p[PS_MAX_S];
};
struct PstOut {
    void* p[PS_MAX_ITEMS];
};

}  // namespace dft
