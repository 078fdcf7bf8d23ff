// Interface of the mixed-precision solvers to the field step (field.cu).
#pragma once

#include "field.cuh"

namespace fempic {

constexpr int kResMaxSlices = 96;   // slices of a block of the on-chip solver, at most

#ifdef __CUDACC__
struct ResidentArgs {
    Sell S;
    const double* val;      // FP64 operator, SELL order (outer residual)
    const float* val32;     // FP32 copy and its 16-bit column offsets col - row
    const uint16_t* d16u;   // (as bit patterns)
    const __nv_bfloat16* dl16;   // learned preconditioner's correction on the same slots (null: off)
    const float* dinv32;
    const int32_t* perm;    // row -> DOF (null: rows in DOF order)
    const int32_t* pp;      // [ns + 1] slot pairs before each slice
    int64_t n;
    int ns, spb, pairs_max;
    const double* b;        // right-hand side, DOF order
    double* x;              // start and solution, DOF order
    double* px;             // solution in row order (x itself without a permutation)
    double* ax;             // null, or A x for the final x in DOF order
    bool x_zero;            // the start is zero, whatever x holds
    const double* scale_vec;
    double* r64;            // FP64 residual, row order
    float *z, *d0, *d1;     // vectors that products gather, row order
    void* sync;
    int deg;
    float theta, delta;
    double tol, inner_tol;
    int max_iter, max_outer;
    double* out;
    int32_t* status;
    int* lflag;
};

fp_status resident_solve(fem_pic* ctx, const ResidentPlan& P, ResidentArgs a, cudaStream_t s);

// sell_row without the evict-first hint: the FP64 operator of an on-chip solve is read once
// per refinement and stays in L2 between them
__device__ __forceinline__ double sell_row_cached(const Sell& S, const double* __restrict__ val, const double* x,
                                                  int64_t i) {
    const int64_t sl = i >> 5;
    const int64_t k0 = __ldg(S.ptr + sl) + (i & 31);
    const int w = __ldg(S.w + sl);
    double s = 0.0;
    for (int j0 = 0; j0 < w; j0 += kSellChunk) {
        int c[kSellChunk];
        double v[kSellChunk], xv[kSellChunk];
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) c[u] = j0 + u < w ? __ldg(S.col + k0 + 32 * (j0 + u)) : -1;
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) v[u] = j0 + u < w ? __ldg(val + k0 + 32 * (j0 + u)) : 0.0;
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) xv[u] = c[u] >= 0 ? x[c[u]] : 0.0;
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) s += v[u] * xv[u];
    }
    return s;
}
#endif

// plan of an on-chip solve; P->on stays false where the system does not fit
fp_status resident_setup(fem_pic* ctx, int64_t n, const std::vector<int32_t>& width, ResidentPlan* P);

}  // namespace fempic
