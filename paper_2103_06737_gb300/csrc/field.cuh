// Internal declarations of the implicit field step (not part of the C ABI).
#pragma once

#include <cuda_bf16.h>

#include <cfloat>
#include <cmath>

#include "internal.cuh"

namespace fempic {

struct HostFields {
    std::vector<uint8_t> edge_fixed, node_fixed;   // PEC DOFs
    std::vector<int32_t> e_rp, e_col;              // edge-edge pattern (free DOFs)
    std::vector<double> M, S;                      // [*eps], [*S] on that pattern
    std::vector<int32_t> n_rp, n_col;              // node-node pattern
    std::vector<double> L;                         // D0^T [*eps] D0
};

// pec: boundary edges and nodes fixed at zero; else the natural boundary (nothing fixed)
void assemble_fields(const HostComplex& hc, double eps, double mu, bool pec, HostFields* hf);

// Largest eigenvalue of D^-1 A (A symmetric CSR with positive diagonal), estimated by
// `steps` Lanczos steps on D^-1/2 A D^-1/2 from a fixed start vector (a lower bound that
// converges quickly for the top of the spectrum).
double jacobi_lambda_max(const std::vector<int32_t>& rp, const std::vector<int32_t>& col,
                         const std::vector<double>& val, int steps);

struct LearnedDev;  // learned correction (learned.cu)

// A solve that ended with a squared residual norm rr has met its threshold.  Not where the residual is
// no finite number: such a solve stops (nothing is left to reduce) but has no solution.
__host__ __device__ inline bool solve_met(double rr, double thr) { return rr <= thr && rr <= DBL_MAX; }

// What a solve's output words (iterations, |r|^2, |reference|^2, refinements) say: the numbers of info,
// and FP_OK, or FP_ENOCONV where the relative residual is not within tol (NaN included).  FP_ECUDA
// where the refinements still are kAbandoned: a mixed solver writes {0, infinity, 1, kAbandoned} when
// it starts, so that one that gives up does not leave an earlier solve's numbers.  marked: an exchange
// of the handle was abandoned; FP_ECUDA too, since a block can give up on a last exchange that the
// others see complete, and its rows of the solution are then missing.
constexpr double kAbandoned = -1.0;
__host__ __device__ inline void solve_begin(double out[4]) {
    out[0] = 0.0, out[1] = HUGE_VAL, out[2] = 1.0, out[3] = kAbandoned;
}
fp_status solve_outcome(const double out[4], bool marked, double tol, fp_solve_info* info);

// launch shape of the on-chip mixed solver for one system (pcg_resident.cu)
struct ResidentPlan {
    bool on = false;            // a block's share of the FP32 operator fits in shared memory
    bool one = false;           // one block
    int grid = 0, threads = 0, spb = 0, pairs_max = 0;   // spb: slices per block
    size_t smem = 0, smem_poly = 0;   // with Jacobi or the learned correction; with the polynomial (0: does not fit)
    int32_t* pp = nullptr;      // device: slot pairs before each slice
};

// packed copies of one system's operator for the streamed mixed solver (pcg_stream.cu)
struct StreamPlan {
    bool on = false;
    int64_t n = 0;
    int ns = 0, nt = 0, nseg = 1, seg = 0, tpb = 0, grid = 0, ring = 0;   // slices, tiles, records per slice, their slots, tiles per block
    void* where = nullptr;                // device: places of the learned correction's records
    std::vector<uint32_t> width;          // per record: slots, and whether its columns are 32-bit
    unsigned char* rec[3] = {nullptr, nullptr, nullptr};   // FP32, learned correction, FP64
    uint2* meta[3] = {nullptr, nullptr, nullptr};
    int stage[3] = {0, 0, 0};
    size_t bytes[3] = {0, 0, 0};
};

struct FieldDev {
    double dt = 0, eps = 0, mu = 0;
    int bc = FP_BC_PEC;             // field boundary condition
    // natural boundary: the W0 integrals alpha (device) and their sum, for the projection's
    // zero-mean constraint; partial sums of its two reductions
    double* alpha = nullptr;
    double alpha_sum = 0.0;
    double* msum = nullptr;
    int64_t ne = 0, nn = 0, nf = 0;
    HostFields host;
    int32_t *e_rp = nullptr, *e_col = nullptr, *n_rp = nullptr, *n_col = nullptr;
    double *Adinv = nullptr, *Ldinv = nullptr;
    uint8_t *edge_fixed = nullptr, *node_fixed = nullptr;
    int32_t* face_edges = nullptr;  // [3 nf]: (i,j), (j,k), (i,k) of face (i<j<k)
    double *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr, *rhs = nullptr, *tmp = nullptr,
           *delta = nullptr, *qd = nullptr;
    float* Ldinv32 = nullptr;       // FP32 copy
    // sliced ELLPACK (slices of 32 rows, column-major inside a slice): coalesced loads of the
    // values and columns of 32 consecutive rows
    int32_t *se_ptr = nullptr, *se_w = nullptr, *se_col = nullptr, *sn_ptr = nullptr, *sn_w = nullptr,
            *sn_col = nullptr;
    double *se_M = nullptr, *se_S = nullptr, *se_A = nullptr, *sn_L = nullptr;
    float* sn_L32 = nullptr;        // FP32 copy, where the on-chip solver runs
    float *r32 = nullptr, *z32 = nullptr, *p32 = nullptr, *q32 = nullptr, *c32 = nullptr;
    float *s32 = nullptr, *d32[2] = {nullptr, nullptr};  // Chebyshev preconditioner scratch
    double lmax[2] = {2.0, 2.0};    // estimated largest eigenvalue of D^-1 A, Newmark and Gauss systems
    // column offsets col - row as int16 in the SELL layout, for the on-chip solver (null without it)
    int16_t *se_d16 = nullptr, *sn_d16 = nullptr;
    // The mixed solver's copy of the Newmark operator in its own row order: solver row r is
    // edge perm_e[r] (rows and columns renumbered alike).  A solve holds its solution in px in
    // this order, the streamed solver its right-hand side in pb (null without it); pe_A32 is null
    // without the on-chip solver.  se_d16 and hwidth of the Newmark system describe this copy.
    int32_t *pe_ptr = nullptr, *pe_w = nullptr, *pe_col = nullptr, *perm_e = nullptr;
    double* pe_A = nullptr;
    float *pe_A32 = nullptr, *pe_dinv32 = nullptr;
    double *pb = nullptr, *px = nullptr;
    int64_t sectors_e[2] = {0, 0};  // gathered 32-byte sectors per product: edge order, solver order
    std::vector<int32_t> hwidth[2];  // host copies of the SELL slice widths (Newmark, Gauss)
    double* red = nullptr;          // reduction partials
    double* out = nullptr;          // [8] output words of the last two solves (in sync's memory)
    int grid = 0;                   // co-resident blocks (cooperative launch limit)
    int grid_e = 0, grid_n = 0;     // grids of the edge and node systems
    int bs_e = 256, bs_n = 256;     // and their block sizes
    int last_fp64[2] = {0, 0};      // solver used by the last solve in each info slot
    bool exchanges[2] = {false, false};   // whether its blocks exchanged through memory
    ResidentPlan res[2];            // on-chip solver, Newmark and Gauss systems
    StreamPlan stream[2];           // streamed solver, Newmark and Gauss systems
    void* sync = nullptr;           // words of the mixed solvers' grid exchanges (grid_sync.cuh)
    LearnedDev* learned[2] = {nullptr, nullptr};  // per system (Newmark, Gauss)
    int learned_sys = FP_SYS_NEWMARK;              // system the fem_pic_learned_* calls address
    bool learned_used[2] = {false, false};         // the last solve in each info slot used its network
    int slot_sys[2] = {FP_SYS_NEWMARK, FP_SYS_GAUSS};  // system of the last solve in each info slot
};

#ifdef __CUDACC__
struct Sell {
    const int32_t* ptr;   // [slices] start of each slice
    const int32_t* w;     // [slices] width (longest row) of each slice
    const int32_t* col;   // padded entries point at the row itself with value 0
};

// row i of a SELL-32 matrix times x; the 32 lanes of a warp take the 32 rows of a slice.
// The entries are taken in chunks of kSellChunk: the column indices of a chunk are loaded
// together, then the values and the gathered x, so a thread has a chunk of independent
// loads in flight instead of one dependent index -> x pair at a time.
#ifndef FP_SELL_CHUNK
#define FP_SELL_CHUNK 8
#endif
constexpr int kSellChunk = FP_SELL_CHUNK;

// Operator entries are read once per product and streamed: with FP_SELL_STREAM (the default)
// they are loaded with the evict-first hint so that they do not push the gathered vector out
// of L2 (96^3 mesh: Gauss-law solve 5.6 -> 4.3 ms, Newmark 19.9 -> 19.4 ms).
#ifndef FP_SELL_STREAM
#define FP_SELL_STREAM 1
#endif
template <typename T>
__device__ __forceinline__ T ld_op(const T* p) {
#if FP_SELL_STREAM
    return __ldcs(p);
#else
    return __ldg(p);
#endif
}

template <typename V, typename X>
__device__ __forceinline__ X sell_row(const Sell& S, const V* __restrict__ val, const X* __restrict__ x,
                                      int64_t i) {
    const int64_t sl = i >> 5;
    const int32_t* cp = S.col + __ldg(S.ptr + sl) + (i & 31);
    const V* vp = val + __ldg(S.ptr + sl) + (i & 31);
    const int w = __ldg(S.w + sl);
    X s = X(0);
    for (int j0 = 0; j0 < w; j0 += kSellChunk) {
        int c[kSellChunk];
        V a[kSellChunk];
        X xv[kSellChunk];
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) c[u] = j0 + u < w ? ld_op(cp + 32 * (j0 + u)) : -1;
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) a[u] = j0 + u < w ? ld_op(vp + 32 * (j0 + u)) : V(0);
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) xv[u] = c[u] >= 0 ? __ldcg(x + c[u]) : X(0);
#pragma unroll
        for (int u = 0; u < kSellChunk; ++u) s += (X)a[u] * xv[u];
    }
    return s;
}

#endif

// learned correction hooks (learned.cu)
void learned_free(FieldDev* F);
void learned_free(FieldDev* F, int sys);
fp_status learned_guess(fem_pic* ctx, int sys, const double* rhs, double* x0, cudaStream_t s);
bool learned_active(const FieldDev* F, int sys);
int* learned_flag(FieldDev* F, int sys);
// the learned preconditioner's correction (solver SELL layout) when it is active and built, else null
const __nv_bfloat16* learned_precond(const FieldDev* F, int sys);
bool learned_precond_ready(const FieldDev* F, int sys);   // model FP_LEARNED_PRECOND, built
int learned_model(const FieldDev* F, int sys);            // -1: no network
void learned_set_active(FieldDev* F, int sys, bool on);

}  // namespace fempic
