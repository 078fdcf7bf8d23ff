// The mixed-precision solvers of the field step (field.cu): iterative refinement.  The residual
// r = b - A x and its norm are FP64; each correction A c = r / |r| is solved approximately by PCG
// on FP32 copies of A and of the vectors, with FP32 sums (until its own residual drops by
// inner_tol, or by less when that already meets the outer tolerance), then x += |r| c in FP64.
// A p is carried as q = A z + beta q: two grid sums per inner iteration.
//
// Preconditioners of the inner PCG: Jacobi; a learned correction, z = D^-1 r + Dl r with Dl on the
// operator's pattern (a solve in which r.z is not positive goes on with Jacobi); or z = P(r), P
// the Chebyshev polynomial of degree deg in B = D^-1 A applied to f = D^-1 r (three-term
// recurrence on [theta - delta, theta + delta]):
//   d_0 = f / theta, z = d_0, s = f;
//   k = 1..deg-1:  s <- s - B d_{k-1},  d_k = rho_k rho_{k-1} d_{k-1} + (2 rho_k / delta) s,
//                  z <- z + d_k,  rho_0 = delta / theta,  rho_k = 1 / (2 theta / delta - rho_{k-1}).
// P is positive on (0, theta + delta] and beyond it up to 2 theta, so PCG with it stays a
// symmetric positive definite method.  Each step's product needs the previous d of every block:
// one grid barrier per step, d in two buffers.
//
// One cooperative launch per solve; every block takes the same decisions from the same grid sums.
#pragma once

#include "field.cuh"

namespace fempic {

// fraction of the outer threshold an inner solve aims for when that needs less than inner_tol
// (the FP32 recurrence residual can differ slightly from the FP64 one)
constexpr double kInnerMargin = 0.2;
constexpr int kResMaxSlices = 96;   // slices of a block of the on-chip solver, at most

// ---- records of the streamed solver (pcg_stream.cu)
__host__ __device__ constexpr uint32_t align16(uint32_t b) { return (b + 15u) & ~15u; }
constexpr int kConsumers = 15;            // consumer warps = slices of a tile; one more warp copies
constexpr uint32_t kHeader = align16(8u * kConsumers);
constexpr uint32_t kWide = 0x80000000u;   // meta flag: 32-bit columns

enum { OP_F32, OP_LEARNED, OP_F64, OP_COUNT };
// bytes of the parts of a record of w slots: bases, columns, values
__host__ __device__ inline uint32_t base_bytes(uint32_t w, bool wide) { return wide ? 0u : align16(4u * w); }
__host__ __device__ inline uint32_t col_bytes(uint32_t w, bool wide) { return wide ? 128u * w : 128u * ((w + 1u) / 2u); }
__host__ __device__ inline uint32_t val_bytes(uint32_t w, int op) {
    return op == OP_F32 ? 128u * w : op == OP_F64 ? 256u * w : 128u * ((w + 1u) / 2u);
}
__host__ __device__ inline uint32_t rec_bytes(uint32_t w, bool wide, int op) {
    return w == 0 ? 0u : base_bytes(w, wide) + col_bytes(w, wide) + val_bytes(w, op);
}
// a tile's place in the ring
inline uint32_t tile_bytes(uint32_t bytes) { return (bytes + 127u) & ~127u; }

// The ring in shared memory.  A pass hides its copies behind its products only when two of its tiles
// fit, and what the ring leaves free is L1 for the gathered vector (64^3 mesh: 51 us per iteration with
// this much, 53 with all of it): as much as two FP64 tiles of the cube meshes' edge systems take
// (19 slots a row, 2 x 93,568 bytes), more where the operator's own tiles are larger.
constexpr size_t kStreamRing = 187392;

// Rows of up to wmax slots as nseg records of at most seg slots each, alike in size: as few as let two
// FP64 tiles fit in `room` bytes, whatever their column format (20 slots in the 230,656 bytes of
// sm_103a).  Each more record costs a wait on the ring per slice.
inline void stream_segments(int wmax, size_t room, int* nseg, int* seg) {
    int most = 1;
    auto two = [](int w) {
        const uint32_t narrow = rec_bytes(w, false, OP_F64), wide = rec_bytes(w, true, OP_F64);
        return (size_t)2 * tile_bytes(kHeader + kConsumers * (narrow > wide ? narrow : wide));
    };
    while (most < 0xffff && two(most + 1) <= room) ++most;
    const int w = wmax > 1 ? wmax : 1;
    *nseg = (w + most - 1) / most;
    *seg = (w + *nseg - 1) / *nseg;
}

#ifdef __CUDACC__
// FP64 scalars of a refinement, in shared memory: computed by one thread of each block from the
// grid's sums.  With every thread computing them (two square roots and two quotients, 16 cycles of the
// SM's FP64 pipe per warp and operation) a solve of two refinements took 83 instead of 68 us on the
// edge system of the 4^3 mesh and 391 instead of 367 us on that of 32^3.
struct Refinement {
    double rr, ref2, thr, root_thr, rnorm, rinv;   // |r|^2, |reference|^2, threshold, its root, |r|, 1 / |r|
    float red;                                     // by how much the inner solve reduces its residual
    int stop;                                      // the threshold is met (or r is not a number)

    // v: sums of r.r, b.b and the reference's square; the last two count at the first residual
    __device__ __forceinline__ void set(const double (&v)[3], bool first, bool scaled, double tol, double inner_tol) {
        rr = v[0];
        if (first) {
            ref2 = scaled ? v[2] : v[1];
            thr = tol * tol * ref2;
            root_thr = sqrt(thr);
        }
        stop = !(rr > thr);
        if (stop) return;
        rnorm = sqrt(rr);
        rinv = 1.0 / rnorm;
        const double need = kInnerMargin * (root_thr * rinv);
        red = (float)(need > inner_tol ? need : inner_tol);
    }
};

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
    const double* r0;       // null, or the start's residual, DOF order
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

struct StreamArgs {
    const unsigned char* rec[3];   // packed operators: FP32, learned correction, FP64
    const uint2* meta[3];          // per tile: offset in 16-byte units, bytes
    int stage[3], nst[3];          // bytes of a place in the ring, places
    int ns, nt, nseg, tpb;         // slices, tiles, records per slice, tiles per block
    bool evict_first, learned, x_zero;
    int64_t n;
    const float* dinv32;
    const int32_t* perm;    // row -> DOF (null: rows in DOF order)
    const double* b;        // right-hand side, DOF order
    double* x;              // start and solution, DOF order
    const double* r0;       // null, or the start's residual, DOF order
    double *pb, *px;        // both in row order (b and x themselves without a permutation)
    double* ax;             // null, or A x for the final x in DOF order
    const double* scale_vec;   // row order (no permutation with it)
    double* r64;
    float *r, *z, *p, *q, *c, *s, *d0, *d1;
    void* sync;
    int deg;
    float theta, delta;
    double tol, inner_tol;
    int max_iter, max_outer;
    double* out;
    int32_t* status;
    int* lflag;
};

// the streamed solver: packed copies of an operator (val: FP64, val32: FP32, both in SELL order),
// room for a learned correction's records and their packing, and a solve
fp_status stream_setup(fem_pic* ctx, const Sell& S, const double* val, const float* val32, int64_t n, int wmax,
                       StreamPlan* P);
fp_status stream_learned_room(fem_pic* ctx, StreamPlan* P);
fp_status stream_learned_pack(fem_pic* ctx, StreamPlan* P, const Sell& S, const double* val, const __nv_bfloat16* pre,
                              cudaStream_t s);
fp_status stream_solve(fem_pic* ctx, const StreamPlan& P, StreamArgs a, cudaStream_t s);

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

void stream_free(StreamPlan* P);

// plan of an on-chip solve; P->on stays false where the system does not fit
fp_status resident_setup(fem_pic* ctx, int64_t n, const std::vector<int32_t>& width, ResidentPlan* P);

}  // namespace fempic
