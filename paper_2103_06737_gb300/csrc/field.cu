// Implicit field step on the GPU (FP64): Newmark wave-equation update, Gauss-law
// projection, Faraday update (Sec. II.C, IV.A-B), with a Jacobi-preconditioned CG that
// runs as one cooperative kernel (convergence decided on the device, no host round trip).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>

#include "async_copy.cuh"
#include "field.cuh"
#include "grid_sync.cuh"
#include "pcg.cuh"

namespace cg = cooperative_groups;


namespace fempic {


namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBlock = 256;
// Cooperative solvers: up to 2 co-resident blocks per SM (1 for 1024-thread blocks); the block
// size is chosen per system from kSolverBlocks at setup.
constexpr int kSolverPerSm = 2;

__device__ __forceinline__ double as_f64(float x) { return f2d(x); }
__device__ __forceinline__ double as_f64(double x) { return x; }

// Deterministic grid-wide sum of NV values, result valid in every thread.  Warp sums go to
// sh[k][warp]; thread 0 writes the block's partial to part[NV * block + k]; after the grid
// barrier warp 0 of every block adds all partials in block order and broadcasts through
// sh[k][BS / 32].  Two block barriers and one grid barrier per call.  Consecutive calls must
// use different `part` buffers (a block may write the next partials while another block
// still reads these).
template <int BS, int NV, typename T>
__device__ __forceinline__ void grid_sum(T v[NV], T* part, cg::grid_group& g, T (*sh)[BS / 32 + 1]) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
    }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k][wid] = v[k];
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            T t = T(0);
#pragma unroll
            for (int w = 0; w < BS / 32; ++w) t += sh[k][w];
            part[NV * blockIdx.x + k] = t;
        }
    g.sync();
    if (wid == 0) {
        T t[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) t[k] = T(0);
        for (int b = lane; b < (int)gridDim.x; b += 32)
#pragma unroll
            for (int k = 0; k < NV; ++k) t[k] += __ldcg(part + NV * b + k);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(kFull, t[k], o);
        }
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < NV; ++k) sh[k][BS / 32] = t[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sh[k][BS / 32];
}

struct PcgArgs {
    Sell S;
    const double* val;
    const double* dinv;
    int64_t n;
    const double* b;
    double* x;
    double *r, *z, *p, *q;
    double* red;
    double tol;
    const double* scale_vec;  // non-null: stop at ||r|| <= tol ||scale_vec||, else at ||r|| <= tol ||b||
    int max_iter;
    double* out;     // [iterations, ||r||^2, ||b||^2]
    int32_t* status;
};

// Jacobi-preconditioned conjugate gradients in one cooperative launch (FP64).  Every
// block takes the same decisions from the same grid-wide sums (deterministic: partials
// summed in block order), so all blocks run the same number of grid barriers; the loop is
// bounded by max_iter.  A p is carried as q = A z + beta q, two barriers per iteration.
template <int BS>
__global__ void __launch_bounds__(BS, BS >= 1024 ? 1 : kSolverPerSm) k_pcg(PcgArgs a) {
    cg::grid_group g = cg::this_grid();
    __shared__ double sh[4][BS / 32 + 1];
    // rows [r0, r1) of this block: contiguous runs of whole 32-row slices, so the columns a
    // block gathers (neighbouring DOFs) stay within a window that its SM's L1 can hold
    const int64_t chunk = ((a.n + gridDim.x - 1) / gridDim.x + 31) & ~(int64_t)31;
    const int64_t r0 = min(a.n, (int64_t)blockIdx.x * chunk), r1 = min(a.n, r0 + chunk);
    const int64_t stride = BS;
    const int64_t t0 = r0 + threadIdx.x;
    double* part0 = a.red;                    // 4 values per block
    double* part1 = a.red + 4 * gridDim.x;    // 2 values per block
    double* part2 = a.red + 6 * gridDim.x;    // 2 values per block
    double v[4] = {0.0, 0.0, 0.0, 0.0};  // r.r, b.b, s.s
    for (int64_t i = t0; i < r1; i += stride) {
        const double bi = a.b[i];
        const double ri = bi - sell_row<double, double>(a.S, a.val, a.x, i);
        a.r[i] = ri;
        a.z[i] = a.dinv[i] * ri;
        v[0] += ri * ri;
        v[1] += bi * bi;
        if (a.scale_vec) v[2] += a.scale_vec[i] * a.scale_vec[i];
    }
    grid_sum<BS, 4, double>(v, part0, g, sh);  // also makes z visible to every block
    double rr = v[0];
    const double bb = a.scale_vec ? v[2] : v[1];
    const double thr = a.tol * a.tol * bb;
    int it = 0;
    if (rr > thr && a.max_iter > 0) {
        // p = z, q = A z; rz, pq
        double u[2] = {0.0, 0.0};
        for (int64_t i = t0; i < r1; i += stride) {
            const double w = sell_row<double, double>(a.S, a.val, a.z, i);
            const double zi = a.z[i];
            a.p[i] = zi;
            a.q[i] = w;
            u[0] += a.r[i] * zi;
            u[1] += zi * w;
        }
        grid_sum<BS, 2, double>(u, part1, g, sh);
        double rz = u[0], pq = u[1];
        for (;;) {
            if (!(pq > 0.0)) break;  // breakdown (same decision in every block)
            const double alpha = rz / pq;
            double w2[2] = {0.0, 0.0};  // r.z, r.r
            for (int64_t i = t0; i < r1; i += stride) {
                a.x[i] += alpha * a.p[i];
                const double ri = a.r[i] - alpha * a.q[i];
                const double zi = a.dinv[i] * ri;
                a.r[i] = ri;
                a.z[i] = zi;
                w2[0] += ri * zi;
                w2[1] += ri * ri;
            }
            grid_sum<BS, 2, double>(w2, part2, g, sh);
            ++it;
            rr = w2[1];
            if (!(rr > thr) || it >= a.max_iter) break;
            const double beta = w2[0] / rz;
            rz = w2[0];
            double u2[2] = {0.0, 0.0};
            for (int64_t i = t0; i < r1; i += stride) {
                const double w = sell_row<double, double>(a.S, a.val, a.z, i);
                const double pi = a.z[i] + beta * a.p[i];
                const double qi = w + beta * a.q[i];
                a.p[i] = pi;
                a.q[i] = qi;
                u2[0] += pi * qi;
            }
            grid_sum<BS, 2, double>(u2, part1, g, sh);
            pq = u2[0];
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[0] = (double)it;
        a.out[1] = rr;
        a.out[2] = bb;      // squared norm the residual is measured against
        a.out[3] = 0.0;
        if (!solve_met(rr, thr)) atomicOr(a.status, ST_NOCONV);
    }
}

// Newmark right-hand side, the extrapolated initial guess u = 2E^n - E^{n-1} and its residual.
// With A = [*eps] + dt^2/4 [*S] the right-hand side
//   [*eps] u - dt^2 [*S] (E^n / 2 + E^{n-1} / 4) - dG = A u - dt^2 [*S] E^n - dG,
// dG = dG^{n+1/2} - dG^{n-1/2}: so r0 = b - A u = -dt^2 [*S] E^n - dG comes with it, and the solver
// starts without an FP64 product of its own (field step on the 64^3 mesh 2423 -> 2383 us, 96^3
// 18.0 -> 17.5 ms).
// u is a pass of its own, so that the SELL pass does two FP64 multiply-adds per stored entry.
__global__ void k_newmark_guess(const uint8_t* __restrict__ fixed, const double* __restrict__ En,
                                const double* __restrict__ Em, int64_t n, double* __restrict__ u) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        u[i] = fixed[i] ? 0.0 : 2.0 * En[i] - Em[i];
}

template <typename Real>
__global__ void k_newmark_rhs(Sell Sl, const double* __restrict__ Av, const double* __restrict__ Sv,
                              const uint8_t* __restrict__ fixed, const double* __restrict__ u,
                              const double* __restrict__ En, double dt2, const Real* __restrict__ dGh,
                              const Real* __restrict__ dGp, int64_t n, double* __restrict__ rhs,
                              double* __restrict__ r0) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t sl = i >> 5;
        const int64_t base = __ldg(Sl.ptr + sl) + (i & 31);
        const int w = __ldg(Sl.w + sl);
        double s = 0.0, t = 0.0;
        for (int j0 = 0; j0 < w; j0 += kSellChunk) {   // chunks of independent loads, as in sell_row
            int c[kSellChunk];
#pragma unroll
            for (int q = 0; q < kSellChunk; ++q) c[q] = j0 + q < w ? __ldg(Sl.col + base + 32 * (j0 + q)) : -1;
#pragma unroll
            for (int q = 0; q < kSellChunk; ++q) {
                if (c[q] < 0) continue;
                const int64_t k = base + 32 * (int64_t)(j0 + q);
                s = fma(__ldg(Av + k), u[c[q]], s);
                t = fma(__ldg(Sv + k), __ldg(En + c[q]), t);
            }
        }
        if (fixed[i]) {
            rhs[i] = r0[i] = 0.0;
            continue;
        }
        const double gh = dGh ? as_f64(dGh[i]) : 0.0, gp = dGp ? as_f64(dGp[i]) : 0.0;
        const double r = -dt2 * t - (gh - gp);
        r0[i] = r;
        rhs[i] = s + r;
    }
}

__global__ void k_spmv(Sell Sl, const double* __restrict__ val, const double* __restrict__ x, int64_t n,
                       double* __restrict__ y) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        y[i] = sell_row<double, double>(Sl, val, x, i);
}

// g_n = (D0^T [*eps] E)_n + Q_n on free nodes (ME = [*eps] E), 0 on PEC nodes; and, where b is
// given, the Faraday update of the same step, b <- b - dt D1 (E1 + E0)/2 on face (i<j<k): +(i,j)
// +(j,k) -(i,k).  E1 is the Newmark solution before the projection: the projection subtracts a
// gradient (zero on PEC edges, whose nodes it leaves alone), and D1 D0 = 0, so its curl is that of
// the projected field.  One launch for both, and the projection then runs in place: a copy and a
// launch less (the field step's kernels beside the solves: 4^3 mesh 36 -> 30 us, 32^3 75 -> 62 us).
template <typename Real>
__global__ void k_gauss_rhs(const int32_t* __restrict__ ptr, const int32_t* __restrict__ col,
                            const int8_t* __restrict__ sgn, const uint8_t* __restrict__ fixed,
                            const double* __restrict__ ME, const Real* __restrict__ Q, int64_t nn,
                            double* __restrict__ g, double* __restrict__ qd, const int32_t* __restrict__ fe,
                            const double* __restrict__ E1, const double* __restrict__ E0, double half_dt, int64_t nf,
                            double* __restrict__ b) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, all = b ? nn + nf : nn;
    for (int64_t i = first; i < all; i += stride) {
        if (i >= nn) {
            const int64_t f = i - nn;
            const int ij = __ldg(fe + 3 * f), jk = __ldg(fe + 3 * f + 1), ik = __ldg(fe + 3 * f + 2);
            const double c = (__ldg(E1 + ij) + __ldg(E0 + ij)) + (__ldg(E1 + jk) + __ldg(E0 + jk)) -
                             (__ldg(E1 + ik) + __ldg(E0 + ik));
            b[f] -= half_dt * c;
            continue;
        }
        if (fixed[i]) {
            g[i] = 0.0;
            qd[i] = 0.0;
            continue;
        }
        double s = Q ? as_f64(Q[i]) : 0.0;
        qd[i] = s;
        for (int j = ptr[i]; j < ptr[i + 1]; ++j) s += sgn[j] > 0 ? ME[col[j]] : -ME[col[j]];
        g[i] = s;
    }
}

// E_e <- EN_e - (d_j - d_i) on free edges, 0 on PEC edges: the Gauss-law projection E - D0 d (E may be EN)
__global__ void k_project(const int32_t* __restrict__ edges, const uint8_t* __restrict__ fixed,
                          const double* __restrict__ d, const double* EN, int64_t ne, double* E) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += stride) {
        const int2 ij = __ldg(reinterpret_cast<const int2*>(edges) + e);
        E[e] = fixed[e] ? 0.0 : EN[e] - (__ldg(d + ij.y) - __ldg(d + ij.x));
    }
}

constexpr int kSolverBlocks[4] = {128, 256, 512, 1024};

void* solver_kernel(int bs) {
    switch (bs) {
        case 128: return (void*)k_pcg<128>;
        case 256: return (void*)k_pcg<256>;
        case 1024: return (void*)k_pcg<1024>;
        default: return (void*)k_pcg<512>;
    }
}

int grid_of(const fem_pic* ctx, int64_t n) {
    int64_t g = (n + kBlock - 1) / kBlock, cap = (int64_t)ctx->sm_count * 8;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

template <typename T>
fp_status up(fem_pic* ctx, T** d, const std::vector<T>& h) {
    FP_CUDA_TRY(ctx, cudaMalloc((void**)d, h.size() * sizeof(T) + 16));
    if (!h.empty()) FP_CUDA_TRY(ctx, cudaMemcpy(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
    return FP_OK;
}

// ax (Newmark system only, may be null): also A x for the final x, in DOF order, when the
// mixed solver ran (F->last_fp64[slot] == 0 afterwards); the FP64 solver leaves it alone.
// x_zero: the start is zero whatever x holds.
fp_status run_pcg(fem_pic* ctx, int system, const double* rhs, double* x, double tol, const double* scale_vec,
                  int max_iter, int slot, cudaStream_t s, double* ax = nullptr, bool x_zero = false,
                  const double* r0 = nullptr) {
    FieldDev* F = ctx->field;
    int use64 = ctx->solver_fp64;
    if (ctx->solver_sys[system] >= 0) use64 = ctx->solver_sys[system] == FP_PC_JACOBI_FP64;
    const int ph = system == FP_SYS_NEWMARK ? PH_CG_NEWMARK : PH_CG_GAUSS;
    F->last_fp64[slot] = use64;
    F->slot_sys[slot] = system;
    F->exchanges[slot] = false;
    if (!use64) {
        const bool nm = system == FP_SYS_NEWMARK;
        const __nv_bfloat16* dl16 = learned_precond(F, system);
        int* lflag = dl16 ? learned_flag(F, system) : nullptr;
        const int deg = dl16 ? 1 : ctx->poly_deg[system];   // the learned preconditioner replaces the polynomial
        // Chebyshev interval [b / ratio, b] with b 5% above the Lanczos estimate of lambda_max
        const double bmax = 1.05 * F->lmax[system], blo = bmax / ctx->poly_ratio[system];
        const float theta = (float)(0.5 * (bmax + blo)), delta = (float)(0.5 * (bmax - blo));
        const int32_t* perm = nm ? F->perm_e : nullptr;   // the Newmark system has its own row order
        const int max_outer = 12;
        PhaseTimer pt(ctx, ph, s);
        const ResidentPlan& P = F->res[system];
        const bool on_chip = P.on && (deg <= 1 || P.smem_poly);
        F->exchanges[slot] = !(on_chip && P.one);
        if (on_chip) {
            ResidentArgs a{};
            a.S = nm ? Sell{F->pe_ptr, F->pe_w, F->pe_col} : Sell{F->sn_ptr, F->sn_w, F->sn_col};
            a.val = nm ? F->pe_A : F->sn_L, a.val32 = nm ? F->pe_A32 : F->sn_L32;
            a.d16u = reinterpret_cast<const uint16_t*>(nm ? F->se_d16 : F->sn_d16);
            a.dinv32 = nm ? F->pe_dinv32 : F->Ldinv32, a.dl16 = dl16, a.perm = perm;
            a.n = nm ? F->ne : F->nn, a.ns = (int)((a.n + 31) / 32);
            a.b = rhs, a.x = x, a.px = perm ? F->px : x, a.ax = ax, a.x_zero = x_zero, a.scale_vec = scale_vec;
            a.r0 = x_zero ? rhs : r0, a.r64 = F->q, a.z = F->z32, a.d0 = F->d32[0], a.d1 = F->d32[1], a.sync = F->sync;
            a.deg = deg, a.theta = theta, a.delta = delta, a.tol = tol, a.inner_tol = ctx->inner_tol;
            a.max_iter = max_iter, a.max_outer = max_outer, a.out = F->out + 4 * slot, a.status = ctx->d_status;
            a.lflag = lflag;
            return resident_solve(ctx, P, a, s);
        }
        StreamArgs a{};
        a.learned = dl16 != nullptr, a.x_zero = x_zero;
        a.dinv32 = nm ? F->pe_dinv32 : F->Ldinv32, a.perm = perm;
        a.b = rhs, a.x = x, a.pb = perm ? F->pb : const_cast<double*>(rhs), a.px = perm ? F->px : x, a.ax = ax;
        a.scale_vec = scale_vec, a.r0 = x_zero ? rhs : r0, a.r64 = F->q;
        a.r = F->r32, a.z = F->z32, a.p = F->p32, a.q = F->q32, a.c = F->c32, a.s = F->s32;
        a.d0 = F->d32[0], a.d1 = F->d32[1], a.sync = F->sync;
        a.deg = deg, a.theta = theta, a.delta = delta, a.tol = tol, a.inner_tol = ctx->inner_tol;
        a.max_iter = max_iter, a.max_outer = max_outer, a.out = F->out + 4 * slot, a.status = ctx->d_status;
        a.lflag = lflag;
        return stream_solve(ctx, F->stream[system], a, s);
    }
    PcgArgs a;
    if (system == FP_SYS_NEWMARK) {
        a.S = Sell{F->se_ptr, F->se_w, F->se_col}, a.val = F->se_A, a.dinv = F->Adinv, a.n = F->ne;
    } else {
        a.S = Sell{F->sn_ptr, F->sn_w, F->sn_col}, a.val = F->sn_L, a.dinv = F->Ldinv, a.n = F->nn;
    }
    if (x_zero) FP_CUDA_TRY(ctx, cudaMemsetAsync(x, 0, a.n * sizeof(double), s));
    a.b = rhs, a.x = x, a.r = F->r, a.z = F->z, a.p = F->p, a.q = F->q, a.red = F->red;
    a.tol = tol, a.scale_vec = scale_vec, a.max_iter = max_iter, a.out = F->out + 4 * slot, a.status = ctx->d_status;
    void* args[] = {&a};
    PhaseTimer pt(ctx, ph, s);
    const int grid = system == FP_SYS_NEWMARK ? F->grid_e : F->grid_n;
    const int bs = system == FP_SYS_NEWMARK ? F->bs_e : F->bs_n;
    FP_CUDA_TRY(ctx, cudaLaunchCooperativeKernel(solver_kernel(bs), dim3(grid), dim3(bs), args, 0, s));
    return FP_OK;
}

// tol: the tolerance the solve had (FP_ENOCONV where it missed it); below 0: only the numbers
fp_status fill_info(fem_pic* ctx, int slot, double tol, fp_solve_info* info, cudaStream_t s, float ms) {
    if (!info) return FP_OK;
    GridReport r;
    FP_CUDA_TRY(ctx, cudaMemcpyAsync(&r, static_cast<const char*>(ctx->field->sync) + kGridMark, sizeof r,
                                     cudaMemcpyDeviceToHost, s));
    FP_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    fp_status met = solve_outcome(r.out + 4 * slot, r.mark != 0 && ctx->field->exchanges[slot], tol, info);
    if (tol < 0.0 && met == FP_ENOCONV) met = FP_OK;
    if (met == FP_ECUDA) ctx->err = "a field solve gave up waiting for its other blocks: no solution (fem_pic_status resets it)";
    info->ms = ms;
    info->precond = ctx->field->last_fp64[slot] ? FP_PC_JACOBI_FP64 : FP_PC_JACOBI;
    info->fell_back = 0;
    if (ctx->field->learned_used[slot]) {
        int fl = 0;
        if (const int* flag = learned_flag(ctx->field, ctx->field->slot_sys[slot])) {   // null: no network any more
            FP_CUDA_TRY(ctx, cudaMemcpyAsync(&fl, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
            FP_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        }
        info->precond = FP_PC_LEARNED;
        info->fell_back = fl;
    }
    return met;
}

// Natural boundary (Eq. zero_mean_constraint): the projection solves L d = g - (sum g / sum
// alpha) alpha (L is singular, its null space the constants; the net charge is spread as
// alpha) and takes the solution with alpha^T d = 0, the d = C_z y of the constrained system.
// Both use a deterministic reduction: per-block partial sums, then every block adds the
// partials in block order before it updates its entries.
constexpr int kMeanBlocks = 128;

// part[b] = sum over block b's entries of v (w == nullptr) or of w v
__global__ void __launch_bounds__(256) k_dot_partial(const double* __restrict__ v, const double* __restrict__ w,
                                                     int64_t n, double* __restrict__ part) {
    __shared__ double sh[8];
    double t = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        t += w ? w[i] * v[i] : v[i];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double u = 0.0;
        for (int k = 0; k < 8; ++k) u += sh[k];
        part[blockIdx.x] = u;
    }
}

// y -= (scale sum_b part[b]) dir  (dir == nullptr: the constant vector 1)
__global__ void __launch_bounds__(256) k_sub_scaled(const double* __restrict__ part, int np, double scale,
                                                    const double* __restrict__ dir, int64_t n, double* __restrict__ y) {
    __shared__ double c;
    if (threadIdx.x == 0) {
        double u = 0.0;
        for (int k = 0; k < np; ++k) u += part[k];
        c = scale * u;
    }
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] -= dir ? c * dir[i] : c;
}

// the projection's right-hand side made consistent (natural boundary only)
fp_status neumann_rhs(fem_pic* ctx, cudaStream_t s) {
    FieldDev* F = ctx->field;
    if (F->bc != FP_BC_NEUMANN) return FP_OK;
    k_dot_partial<<<kMeanBlocks, 256, 0, s>>>(F->rhs, nullptr, F->nn, F->msum);
    k_sub_scaled<<<kMeanBlocks, 256, 0, s>>>(F->msum, kMeanBlocks, 1.0 / F->alpha_sum, F->alpha, F->nn, F->rhs);
    FP_CUDA_TRY(ctx, cudaGetLastError());
    return FP_OK;
}

// the projection's solution shifted to alpha^T d = 0 (natural boundary only)
fp_status neumann_gauge(fem_pic* ctx, cudaStream_t s) {
    FieldDev* F = ctx->field;
    if (F->bc != FP_BC_NEUMANN) return FP_OK;
    k_dot_partial<<<kMeanBlocks, 256, 0, s>>>(F->delta, F->alpha, F->nn, F->msum);
    k_sub_scaled<<<kMeanBlocks, 256, 0, s>>>(F->msum, kMeanBlocks, 1.0 / F->alpha_sum, nullptr, F->nn, F->delta);
    FP_CUDA_TRY(ctx, cudaGetLastError());
    return FP_OK;
}

fp_status field_step_impl(fem_pic_t* ctx, const double* E_prev, const double* E_cur, double* E_next,
                          double* b, const void* dG_half, const void* dG_prev, const void* Q_new, double tol,
                          int max_iter, cudaStream_t s) {
    FieldDev* F = ctx->field;
    const bool f32 = dG_f32(ctx), q32 = Q_f32(ctx);   // dG, Q are float arrays
    const int ge = grid_of(ctx, F->ne);
    {
        PhaseTimer pt(ctx, PH_SOLVE, s);
        // u = 2E^n - E^{n-1} goes straight into E_next: it is also the solver's starting guess
        const double dt2 = F->dt * F->dt;
        k_newmark_guess<<<ge, kBlock, 0, s>>>(F->edge_fixed, E_cur, E_prev, F->ne, E_next);
        if (f32)
            k_newmark_rhs<float><<<ge, kBlock, 0, s>>>(Sell{F->se_ptr, F->se_w, F->se_col}, F->se_A, F->se_S,
                                                       F->edge_fixed, E_next, E_cur, dt2, (const float*)dG_half,
                                                       (const float*)dG_prev, F->ne, F->rhs, F->z);
        else
            k_newmark_rhs<double><<<ge, kBlock, 0, s>>>(Sell{F->se_ptr, F->se_w, F->se_col}, F->se_A, F->se_S,
                                                        F->edge_fixed, E_next, E_cur, dt2, (const double*)dG_half,
                                                        (const double*)dG_prev, F->ne, F->rhs, F->z);
        FP_CUDA_TRY(ctx, cudaGetLastError());
    }
    // learned correction of the guess (with fallback), and/or collection of its residual
    if (learned_active(F, FP_SYS_NEWMARK)) {
        fp_status sl = learned_guess(ctx, FP_SYS_NEWMARK, F->rhs, E_next, s);
        if (sl != FP_OK) return sl;
    }
    // Newmark solve for E^N from the guess 2E^n - E^{n-1} (written into E_next above), whose residual
    // is known unless the learned correction may have replaced it
    const bool replaced = learned_active(F, FP_SYS_NEWMARK) && learned_model(F, FP_SYS_NEWMARK) == FP_LEARNED_GUESS;
    fp_status st = run_pcg(ctx, FP_SYS_NEWMARK, F->rhs, E_next, tol, nullptr, max_iter, 0, s, F->tmp, false,
                           replaced ? nullptr : F->z);
    if (st != FP_OK) return st;
    // Gauss-law projection: L d = D0^T M E^N + Q on interior nodes, to ||r|| <= tol ||Q||.
    // D0^T M E^N = D0^T A E^N, since D0^T S = (S D0)^T = 0 (curl grad = 0) on the rows the
    // interior nodes touch; the mixed solver hands back A E^N = b - r from its last residual,
    // so M E^N needs its own product only after the FP64 solver.
    {
        PhaseTimer pt(ctx, PH_SOLVE, s);
        if (F->last_fp64[0])
            k_spmv<<<ge, kBlock, 0, s>>>(Sell{F->se_ptr, F->se_w, F->se_col}, F->se_M, E_next, F->ne, F->tmp);
        // and the Faraday update of b, from E^N
        const int gf = grid_of(ctx, b ? F->nn + F->nf : F->nn);
        if (q32)
            k_gauss_rhs<float><<<gf, kBlock, 0, s>>>(ctx->d_n2e_ptr, ctx->d_n2e_col, ctx->d_n2e_sgn, F->node_fixed,
                                                     F->tmp, (const float*)Q_new, F->nn, F->rhs, F->qd, F->face_edges,
                                                     E_next, E_cur, 0.5 * F->dt, F->nf, b);
        else
            k_gauss_rhs<double><<<gf, kBlock, 0, s>>>(ctx->d_n2e_ptr, ctx->d_n2e_col, ctx->d_n2e_sgn,
                                                      F->node_fixed, F->tmp, (const double*)Q_new, F->nn, F->rhs,
                                                      F->qd, F->face_edges, E_next, E_cur, 0.5 * F->dt, F->nf, b);
        FP_CUDA_TRY(ctx, cudaGetLastError());
        fp_status sn = neumann_rhs(ctx, s);
        if (sn != FP_OK) return sn;
    }
    // learned correction of the projection's zero starting point (node graph), with fallback
    const bool corrected = learned_active(F, FP_SYS_GAUSS) && learned_model(F, FP_SYS_GAUSS) == FP_LEARNED_GUESS;
    if (learned_active(F, FP_SYS_GAUSS)) {
        FP_CUDA_TRY(ctx, cudaMemsetAsync(F->delta, 0, F->nn * sizeof(double), s));
        fp_status sl = learned_guess(ctx, FP_SYS_GAUSS, F->rhs, F->delta, s);
        if (sl != FP_OK) return sl;
    }
    st = run_pcg(ctx, FP_SYS_GAUSS, F->rhs, F->delta, tol, F->qd, max_iter, 1, s, nullptr, !corrected);
    if (st != FP_OK) return st;
    {
        PhaseTimer pt(ctx, PH_SOLVE, s);
        st = neumann_gauge(ctx, s);
        if (st != FP_OK) return st;
        k_project<<<ge, kBlock, 0, s>>>(ctx->d_edges, F->edge_fixed, F->delta, E_next, F->ne, E_next);
        FP_CUDA_TRY(ctx, cudaGetLastError());
    }
    return FP_OK;
}

}  // namespace

// a block that joins an exchange of two and is alone in it
static __global__ void k_exchange_selftest(void* sync, int32_t* status, uint64_t limit_ns) {
    __shared__ GridSyncShared sh;
    GridSync<false> g;
    g.init(sync, &sh, status);
    g.nb = 2;
    g.limit1 = limit_ns;
    g.barrier();
}
fp_status launch_exchange_selftest(fem_pic* ctx, double limit_s, cudaStream_t s) {
    if (!ctx->field || !ctx->field->sync) return FP_OK;
    k_exchange_selftest<<<1, 32, 0, s>>>(ctx->field->sync, ctx->d_status, (uint64_t)(limit_s * 1e9));
    FP_CUDA_TRY(ctx, cudaGetLastError());
    return FP_OK;
}

// after a wait of a mixed solver ran out: the words of its grid exchanges start afresh
cudaError_t field_reset_sync(fem_pic* ctx, cudaStream_t s) {
    if (!ctx->field || !ctx->field->sync) return cudaSuccess;
    char* m = static_cast<char*>(ctx->field->sync);
    const cudaError_t e = cudaMemsetAsync(m, 0, kGridOut, s);   // (not the output words)
    return e != cudaSuccess ? e : cudaMemsetAsync(m + kGridLine, 0, grid_sync_bytes(ctx->sm_count) - kGridLine, s);
}

void field_free(fem_pic* ctx) {
    FieldDev* F = ctx->field;
    if (!F) return;
    learned_free(F);
    void* ptrs[] = {F->e_rp, F->e_col, F->n_rp, F->n_col, F->Adinv, F->Ldinv,
                    F->edge_fixed, F->node_fixed, F->face_edges, F->r, F->z, F->p, F->q, F->rhs, F->tmp,
                    F->delta, F->qd, F->red, F->Ldinv32, F->r32,
                    F->z32, F->p32, F->q32, F->c32, F->s32, F->d32[0], F->d32[1], F->se_d16, F->sn_d16, F->pe_ptr, F->pe_w, F->pe_col, F->perm_e, F->pe_A, F->pe_A32, F->pe_dinv32, F->pb, F->px, F->alpha, F->msum, F->se_ptr, F->se_w, F->se_col, F->sn_ptr, F->sn_w,
                    F->sn_col, F->se_M, F->se_S, F->se_A, F->sn_L, F->sn_L32, F->sync, F->res[0].pp, F->res[1].pp};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    for (StreamPlan& P : F->stream) stream_free(&P);
    delete F;
    ctx->field = nullptr;
}

}  // namespace fempic

using namespace fempic;

static fp_status field_setup(fem_pic_t* ctx, double dt, double eps, double mu, int bc) {
    FieldDev* F = new FieldDev();
    ctx->field = F;
    const HostComplex& hc = ctx->hc;
    F->dt = dt, F->eps = eps, F->mu = mu, F->ne = hc.ne, F->nn = hc.nn, F->nf = hc.nf, F->bc = bc;
    assemble_fields(hc, eps, mu, bc == FP_BC_PEC, &F->host);
    const HostFields& H = F->host;
    std::vector<double> A(H.M.size()), Ad(hc.ne), Ld(hc.nn);
    for (size_t k = 0; k < A.size(); ++k) A[k] = H.M[k] + 0.25 * dt * dt * H.S[k];
    for (int64_t i = 0; i < hc.ne; ++i)
        for (int32_t j = H.e_rp[i]; j < H.e_rp[i + 1]; ++j)
            if (H.e_col[j] == i) Ad[i] = 1.0 / A[j];
    for (int64_t i = 0; i < hc.nn; ++i)
        for (int32_t j = H.n_rp[i]; j < H.n_rp[i + 1]; ++j)
            if (H.n_col[j] == i) Ld[i] = 1.0 / H.L[j];
    // top of the Jacobi-scaled spectra, for the Chebyshev preconditioner of the inner solves
    F->lmax[FP_SYS_NEWMARK] = jacobi_lambda_max(H.e_rp, H.e_col, A, 40);
    F->lmax[FP_SYS_GAUSS] = jacobi_lambda_max(H.n_rp, H.n_col, H.L, 40);
    // face -> edges (i,j), (j,k), (i,k)
    std::vector<int32_t> fe(3 * hc.nf);
    {
        std::vector<int32_t> rp, col;
        std::vector<int8_t> val;
        incidence_csr(hc, 1, &rp, &col, &val);  // columns sorted: (i,j) < (i,k) < (j,k)
        for (int64_t f = 0; f < hc.nf; ++f) {
            fe[3 * f] = col[3 * f];
            fe[3 * f + 1] = col[3 * f + 2];
            fe[3 * f + 2] = col[3 * f + 1];
        }
    }
    fp_status st = FP_OK;
    if (st == FP_OK) st = up(ctx, &F->e_rp, H.e_rp);
    if (st == FP_OK) st = up(ctx, &F->e_col, H.e_col);
    if (st == FP_OK) st = up(ctx, &F->n_rp, H.n_rp);
    if (st == FP_OK) st = up(ctx, &F->n_col, H.n_col);
    if (st == FP_OK) st = up(ctx, &F->Adinv, Ad);
    if (st == FP_OK) st = up(ctx, &F->Ldinv, Ld);
    if (st == FP_OK) st = up(ctx, &F->edge_fixed, H.edge_fixed);
    if (st == FP_OK) st = up(ctx, &F->node_fixed, H.node_fixed);
    if (st == FP_OK) st = up(ctx, &F->face_edges, fe);
    {
        std::vector<float> ld32(Ld.begin(), Ld.end());
        if (st == FP_OK) st = up(ctx, &F->Ldinv32, ld32);
    }
    {
        // SELL-32 copies of the operators (the CSR stays on the host for export)
        auto sell = [](const std::vector<int32_t>& rp, const std::vector<int32_t>& col, int64_t n,
                       std::vector<int32_t>* ptr, std::vector<int32_t>* w, std::vector<int32_t>* scol,
                       std::vector<int64_t>* map) {
            const int64_t ns = (n + 31) / 32;
            ptr->assign(ns, 0);
            w->assign(ns, 0);
            int64_t off = 0;
            for (int64_t sl = 0; sl < ns; ++sl) {
                int wmax = 0;
                for (int64_t r = 32 * sl; r < 32 * sl + 32 && r < n; ++r) wmax = std::max(wmax, rp[r + 1] - rp[r]);
                (*ptr)[sl] = (int32_t)off;
                (*w)[sl] = wmax;
                off += 32 * (int64_t)wmax;
            }
            scol->assign(off, 0);
            map->assign(off, -1);
            for (int64_t sl = 0; sl < ns; ++sl)
                for (int64_t lane = 0; lane < 32; ++lane) {
                    const int64_t r = 32 * sl + lane;
                    const int64_t base = (*ptr)[sl] + lane;
                    for (int j = 0; j < (*w)[sl]; ++j) {
                        const int64_t k = base + 32 * (int64_t)j;
                        if (r < n && j < rp[r + 1] - rp[r]) {
                            (*scol)[k] = col[rp[r] + j];
                            (*map)[k] = rp[r] + j;
                        } else {
                            (*scol)[k] = (int32_t)(r < n ? r : 0);  // padding: zero value
                        }
                    }
                }
        };
        auto gather = [](const std::vector<int64_t>& map, const std::vector<double>& v) {
            std::vector<double> o(map.size(), 0.0);
            for (size_t k = 0; k < map.size(); ++k)
                if (map[k] >= 0) o[k] = v[map[k]];
            return o;
        };
        std::vector<int32_t> ptr, w, scol;
        std::vector<int64_t> map;
        // column offsets col - row as int16 (empty when some offset does not fit)
        // (the lanes past the last row of a partial slice are never computed: offset 0)
        auto offsets16 = [](const std::vector<int32_t>& scol, const std::vector<int32_t>& sptr,
                            const std::vector<int32_t>& sw, int64_t n) {
            std::vector<int16_t> d(scol.size());
            for (size_t sl = 0; sl < sptr.size(); ++sl)
                for (int64_t j = 0; j < sw[sl]; ++j)
                    for (int64_t lane = 0; lane < 32; ++lane) {
                        const int64_t k = sptr[sl] + 32 * j + lane;
                        const int64_t row = (int64_t)(32 * sl + lane);
                        const int64_t off = row < n ? (int64_t)scol[k] - row : 0;
                        if (off < -32768 || off > 32767) return std::vector<int16_t>();
                        d[k] = (int16_t)off;
                    }
            return d;
        };
        sell(H.e_rp, H.e_col, hc.ne, &ptr, &w, &scol, &map);
        std::vector<double> sM = gather(map, H.M), sS = gather(map, H.S), sA = gather(map, A);
        if (st == FP_OK) st = up(ctx, &F->se_ptr, ptr);
        if (st == FP_OK) st = up(ctx, &F->se_w, w);
        if (st == FP_OK) st = up(ctx, &F->se_col, scol);
        if (st == FP_OK) st = up(ctx, &F->se_M, sM);
        if (st == FP_OK) st = up(ctx, &F->se_S, sS);
        if (st == FP_OK) st = up(ctx, &F->se_A, sA);
        {
            // Row order of the mixed solver's Newmark operator.  Edge ids are lexicographic in
            // (i, j), so the edges leaving a node are consecutive and a 32-row slice mixes edges
            // of several directions: lane l's k-th neighbour lies far from lane l+1's, and a
            // product gathers about one useful value per 32-byte sector of x.  Renumbered by
            // (block of kPermNodes first nodes, rank of the edge among its first node's edges,
            // first node), a slice holds same-rank edges of consecutive nodes, whose neighbours
            // are again consecutive.  Of the two orders the one whose products gather fewer
            // sectors (counted over its SELL layout) is kept, so a mesh without that structure
            // keeps the edge order; so is the edge order when the other's column offsets do
            // not fit in 16 bits.
            constexpr int32_t kPermNodes = 256;
            const int64_t ne = hc.ne;
            std::vector<int32_t> ident(ne), blocked(ne), rank(ne, 0);
            for (int64_t k = 0; k < ne; ++k) {
                ident[k] = (int32_t)k;
                if (k > 0 && hc.edges[2 * k] == hc.edges[2 * (k - 1)]) rank[k] = rank[k - 1] + 1;
            }
            blocked = ident;
            std::sort(blocked.begin(), blocked.end(), [&](int32_t a, int32_t b) {
                const int32_t ia = hc.edges[2 * a], ib = hc.edges[2 * b];
                if (ia / kPermNodes != ib / kPermNodes) return ia / kPermNodes < ib / kPermNodes;
                if (rank[a] != rank[b]) return rank[a] < rank[b];
                return ia != ib ? ia < ib : a < b;
            });
            // CSR of P A P^T (columns sorted) for perm (solver row -> edge)
            auto permuted = [&](const std::vector<int32_t>& perm, std::vector<int32_t>* rp2, std::vector<int32_t>* col2,
                                std::vector<double>* val2) {
                std::vector<int32_t> inv(ne);
                for (int64_t r = 0; r < ne; ++r) inv[perm[r]] = (int32_t)r;
                rp2->assign(ne + 1, 0);
                col2->resize(H.e_col.size());
                val2->resize(H.e_col.size());
                std::vector<std::pair<int32_t, double>> row;
                int64_t o = 0;
                for (int64_t r = 0; r < ne; ++r) {
                    const int32_t e0 = perm[r];
                    row.clear();
                    for (int32_t j = H.e_rp[e0]; j < H.e_rp[e0 + 1]; ++j) row.emplace_back(inv[H.e_col[j]], A[j]);
                    std::sort(row.begin(), row.end(),
                              [](const std::pair<int32_t, double>& a, const std::pair<int32_t, double>& b) {
                                  return a.first < b.first;
                              });
                    for (const auto& pr : row) (*col2)[o] = pr.first, (*val2)[o] = pr.second, ++o;
                    (*rp2)[r + 1] = (int32_t)o;
                }
            };
            // distinct 32-byte sectors of x that the lanes of each slice gather per entry
            auto sectors = [](const std::vector<int32_t>& rp, const std::vector<int32_t>& col, int64_t n) {
                int64_t total = 0;
                int32_t sec[32];
                for (int64_t r0 = 0; r0 < n; r0 += 32) {
                    const int64_t r1 = std::min<int64_t>(n, r0 + 32);
                    int w = 0;
                    for (int64_t r = r0; r < r1; ++r) w = std::max(w, rp[r + 1] - rp[r]);
                    for (int j = 0; j < w; ++j) {
                        int m = 0;
                        for (int64_t r = r0; r < r1; ++r)
                            if (j < rp[r + 1] - rp[r]) sec[m++] = col[rp[r] + j] >> 3;
                        std::sort(sec, sec + m);
                        total += (int64_t)(std::unique(sec, sec + m) - sec);
                    }
                }
                return total;
            };
            std::vector<int32_t> rp2, col2;
            std::vector<double> val2;
            permuted(blocked, &rp2, &col2, &val2);
            F->sectors_e[0] = sectors(H.e_rp, H.e_col, ne);
            F->sectors_e[1] = sectors(rp2, col2, ne);
            const std::vector<int32_t>* perm = &blocked;
            std::vector<int16_t> d16;
#ifndef FP_SOLVER_ORDER
#define FP_SOLVER_ORDER 1
#endif
            bool blocked_order = false;
            if (FP_SOLVER_ORDER && F->sectors_e[1] < F->sectors_e[0]) {
                // the solver order gathers fewer sectors; its 16-bit column offsets (for the
                // shared-memory operator) may not fit on large meshes, the order is kept anyway
                sell(rp2, col2, ne, &ptr, &w, &scol, &map);
                d16 = offsets16(scol, ptr, w, ne);
                blocked_order = true;
            }
            if (!blocked_order) {   // the edge order
                perm = &ident;
                F->sectors_e[1] = F->sectors_e[0];
                permuted(ident, &rp2, &col2, &val2);
                sell(rp2, col2, ne, &ptr, &w, &scol, &map);
                d16 = offsets16(scol, ptr, w, ne);
            }
            std::vector<double> pA = gather(map, val2);
            std::vector<float> pA32(pA.begin(), pA.end()), pdinv(ne);
            for (int64_t r = 0; r < ne; ++r) pdinv[r] = (float)Ad[(*perm)[r]];
            if (!d16.empty() && st == FP_OK) st = up(ctx, &F->se_d16, d16);
            F->hwidth[FP_SYS_NEWMARK] = w;
            if (st == FP_OK) st = up(ctx, &F->perm_e, *perm);
            if (st == FP_OK) st = up(ctx, &F->pe_ptr, ptr);
            if (st == FP_OK) st = up(ctx, &F->pe_w, w);
            if (st == FP_OK) st = up(ctx, &F->pe_col, scol);
            if (st == FP_OK) st = up(ctx, &F->pe_A, pA);
            if (st == FP_OK) st = up(ctx, &F->pe_A32, pA32);
            if (st == FP_OK) st = up(ctx, &F->pe_dinv32, pdinv);
            if (st == FP_OK) FP_CUDA_TRY(ctx, cudaMalloc((void**)&F->px, ne * sizeof(double)));
        }
        sell(H.n_rp, H.n_col, hc.nn, &ptr, &w, &scol, &map);
        std::vector<double> sL = gather(map, H.L);
        std::vector<float> sL32(sL.begin(), sL.end());
        {
            const std::vector<int16_t> d16 = offsets16(scol, ptr, w, hc.nn);
            if (!d16.empty() && st == FP_OK) st = up(ctx, &F->sn_d16, d16);
            F->hwidth[FP_SYS_GAUSS] = w;
        }
        if (st == FP_OK) st = up(ctx, &F->sn_ptr, ptr);
        if (st == FP_OK) st = up(ctx, &F->sn_w, w);
        if (st == FP_OK) st = up(ctx, &F->sn_col, scol);
        if (st == FP_OK) st = up(ctx, &F->sn_L, sL);
        if (st == FP_OK) st = up(ctx, &F->sn_L32, sL32);
    }
    const int64_t nmax = hc.ne > hc.nn ? hc.ne : hc.nn;
    float** vecs32[] = {&F->r32, &F->z32, &F->p32, &F->q32, &F->c32, &F->s32, &F->d32[0], &F->d32[1]};
    for (float** v : vecs32)
        if (st == FP_OK) FP_CUDA_TRY(ctx, cudaMalloc((void**)v, nmax * sizeof(float)));
    double** vecs[] = {&F->r, &F->z, &F->p, &F->q, &F->rhs, &F->tmp, &F->delta, &F->qd};
    for (double** v : vecs)
        if (st == FP_OK) FP_CUDA_TRY(ctx, cudaMalloc((void**)v, nmax * sizeof(double)));
    // cooperative grids: all blocks co-resident, at most kSolverPerSm per SM.  Per system the
    // block size whose block count (one row per thread) is closest to one block per SM: the
    // grid barriers and reductions cost more with more blocks, the SpMV and vector passes
    // less with more SMs busy.
    auto pick = [&](int64_t rows, int force, int* bs, int* grid) -> fp_status {
        double best = 1e30;
        for (int b : kSolverBlocks) {
            const double d = std::fabs(std::log((double)((rows + b - 1) / b) / (double)ctx->sm_count));
            if (d < best) best = d, *bs = b;
        }
        if (force > 0) *bs = force;
        int per_sm = 0;
        FP_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, solver_kernel(*bs), *bs, 0));
        per_sm = std::min(per_sm, kSolverPerSm);
        if (per_sm < 1) {
            ctx->err = "fem_pic_field_setup: the solver kernel cannot be co-resident";
            return FP_ECUDA;
        }
        const int64_t need = std::max<int64_t>(1, (rows + *bs - 1) / *bs);
        *grid = (int)std::min<int64_t>(need, (int64_t)ctx->sm_count * per_sm);
        return FP_OK;
    };
#ifndef FP_SOLVER_BS_E
#define FP_SOLVER_BS_E 0
#endif
#ifndef FP_SOLVER_BS_N
#define FP_SOLVER_BS_N 0
#endif
    if (st == FP_OK) st = pick(hc.ne, FP_SOLVER_BS_E, &F->bs_e, &F->grid_e);
    if (st == FP_OK) st = pick(hc.nn, FP_SOLVER_BS_N, &F->bs_n, &F->grid_n);
    // The mixed solver: on chip where a block's share of the operator fits in shared memory
    // (pcg_resident.cu), streamed otherwise (pcg_stream.cu); both where the polynomial's two more
    // vectors are what does not fit.
    for (int sys = 0; sys < 2 && st == FP_OK; ++sys)
        if (sys == FP_SYS_NEWMARK ? F->se_d16 : F->sn_d16)
            st = resident_setup(ctx, sys == FP_SYS_NEWMARK ? hc.ne : hc.nn, F->hwidth[sys], &F->res[sys]);
    for (int sys = 0; sys < 2 && st == FP_OK; ++sys) {
        if (F->res[sys].on && F->res[sys].smem_poly) continue;
        const bool nm = sys == FP_SYS_NEWMARK;
        const int wmax = F->hwidth[sys].empty() ? 0 : *std::max_element(F->hwidth[sys].begin(), F->hwidth[sys].end());
        st = stream_setup(ctx, nm ? Sell{F->pe_ptr, F->pe_w, F->pe_col} : Sell{F->sn_ptr, F->sn_w, F->sn_col},
                          nm ? F->pe_A : F->sn_L, nm ? F->pe_A32 : F->sn_L32, nm ? hc.ne : hc.nn, wmax, &F->stream[sys]);
        if (st == FP_OK && nm) FP_CUDA_TRY(ctx, cudaMalloc((void**)&F->pb, hc.ne * sizeof(double)));
        if (F->res[sys].on) continue;
        // only the on-chip solver reads the unpacked FP32 operator and its 16-bit offsets
        cudaFree(nm ? F->pe_A32 : F->sn_L32);
        cudaFree(nm ? F->se_d16 : F->sn_d16);
        (nm ? F->pe_A32 : F->sn_L32) = nullptr;
        (nm ? F->se_d16 : F->sn_d16) = nullptr;
    }
    if (st == FP_OK) {
        FP_CUDA_TRY(ctx, cudaMalloc(&F->sync, grid_sync_bytes(ctx->sm_count)));
        FP_CUDA_TRY(ctx, cudaMemset(F->sync, 0, grid_sync_bytes(ctx->sm_count)));
        F->out = reinterpret_cast<double*>(static_cast<char*>(F->sync) + kGridOut);
    }
    if (st == FP_OK) {
        F->grid = std::max(F->grid_e, F->grid_n);
        FP_CUDA_TRY(ctx, cudaMalloc((void**)&F->red, 9 * (size_t)F->grid * sizeof(double)));
    }
    if (st == FP_OK && bc == FP_BC_NEUMANN) {
        std::vector<double> a(hc.nn);
        st = fem_pic_whitney0_integrals(ctx, a.data());
        F->alpha_sum = 0.0;
        for (double v : a) F->alpha_sum += v;
        if (st == FP_OK) st = up(ctx, &F->alpha, a);
        if (st == FP_OK) FP_CUDA_TRY(ctx, cudaMalloc((void**)&F->msum, kMeanBlocks * sizeof(double)));
    }
    return st;
}

extern "C" {

fp_status fem_pic_field_setup(fem_pic_t* ctx, double dt, double eps, double mu) {
    return fem_pic_field_setup_bc(ctx, dt, eps, mu, FP_BC_PEC);
}

fp_status fem_pic_field_setup_bc(fem_pic_t* ctx, double dt, double eps, double mu, int bc) {
    if (!ctx || !(dt > 0.0) || !(eps > 0.0) || !(mu > 0.0) || (bc != FP_BC_PEC && bc != FP_BC_NEUMANN)) {
        if (ctx) ctx->err = "fem_pic_field_setup: dt, eps and mu must be positive, bc FP_BC_PEC or FP_BC_NEUMANN";
        return FP_EINVAL;
    }
    field_free(ctx);
    fp_status st;
    try {
        st = field_setup(ctx, dt, eps, mu, bc);
    } catch (const std::bad_alloc&) {   // no exception crosses the C ABI
        ctx->err = "fem_pic_field_setup: out of host memory";
        st = FP_EINVAL;
    }
    if (st != FP_OK) {   // nothing half-built: the handle is as before its first field setup
        field_free(ctx);
        (void)cudaGetLastError();
    }
    return st;
}

fp_status fem_pic_field_options(fem_pic_t* ctx, int newmark_solver, int gauss_solver, double inner_tol) {
    if (!ctx) return FP_EINVAL;
    auto ok = [](int v) { return v == -1 || v == FP_PC_JACOBI || v == FP_PC_JACOBI_FP64; };
    if (!ok(newmark_solver) || !ok(gauss_solver) || !(inner_tol > 0.0 && inner_tol < 1.0)) {
        ctx->err = "fem_pic_field_options: bad solver code or inner tolerance";
        return FP_EINVAL;
    }
    ctx->solver_sys[FP_SYS_NEWMARK] = newmark_solver;
    ctx->solver_sys[FP_SYS_GAUSS] = gauss_solver;
    ctx->inner_tol = inner_tol;
    return FP_OK;
}

fp_status fem_pic_field_poly(fem_pic_t* ctx, int system, int degree, double ratio) {
    if (!ctx || (system != FP_SYS_NEWMARK && system != FP_SYS_GAUSS) || degree < 1 || degree > 16 ||
        !(ratio > 1.0)) {
        if (ctx) ctx->err = "fem_pic_field_poly: system, degree in [1, 16] or ratio > 1 out of range";
        return FP_EINVAL;
    }
    ctx->poly_deg[system] = degree;
    ctx->poly_ratio[system] = ratio;
    return FP_OK;
}

fp_status fem_pic_field_last_info(fem_pic_t* ctx, fp_solve_info info[2], void* stream) {
    if (!ctx || !ctx->field || !info) return FP_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    fp_status st = fill_info(ctx, 0, -1.0, &info[0], s, 0.f);
    if (st == FP_OK) st = fill_info(ctx, 1, -1.0, &info[1], s, 0.f);
    return st;
}

fp_status fem_pic_whitney0_integrals(const fem_pic_t* ctx, double* alpha) {
    if (!ctx || !alpha) return FP_EINVAL;
    const HostComplex& hc = ctx->hc;
    std::vector<double> a(hc.nn, 0.0);
    for (int64_t t = 0; t < hc.nt; ++t) {
        const double* g = hc.geo[t].g;
        // |T| = 1 / (6 |det G|), G = rows grad l1..3
        const double det = g[0] * (g[4] * g[8] - g[5] * g[7]) - g[1] * (g[3] * g[8] - g[5] * g[6]) +
                           g[2] * (g[3] * g[7] - g[4] * g[6]);
        const double q = 1.0 / (24.0 * std::fabs(det));  // |T| / 4
        for (int k = 0; k < 4; ++k) a[hc.tv[4 * t + k]] += q;
    }
    std::memcpy(alpha, a.data(), a.size() * sizeof(double));
    return FP_OK;
}

fp_status fem_pic_field_nnz(const fem_pic_t* ctx, int64_t nnz[2]) {
    if (!ctx || !ctx->field || !nnz) return FP_EINVAL;
    nnz[0] = (int64_t)ctx->field->host.e_col.size();
    nnz[1] = (int64_t)ctx->field->host.n_col.size();
    return FP_OK;
}

fp_status fem_pic_field_matrix(const fem_pic_t* ctx, int which, int32_t* row_ptr, int32_t* col, double* val) {
    if (!ctx || !ctx->field || which < 0 || which > 3) return FP_EINVAL;
    const FieldDev* F = ctx->field;
    const HostFields& H = F->host;
    const bool node = which == 3;
    const std::vector<int32_t>& rp = node ? H.n_rp : H.e_rp;
    const std::vector<int32_t>& c = node ? H.n_col : H.e_col;
    if (row_ptr) std::memcpy(row_ptr, rp.data(), rp.size() * 4);
    if (col) std::memcpy(col, c.data(), c.size() * 4);
    if (val) {
        for (size_t k = 0; k < c.size(); ++k) {
            double v = which == 0 ? H.M[k] : which == 1 ? H.S[k] : which == 2 ? H.M[k] + 0.25 * F->dt * F->dt * H.S[k]
                                                                             : H.L[k];
            val[k] = v;
        }
    }
    return FP_OK;
}

fp_status fem_pic_field_solve(fem_pic_t* ctx, int system, const double* rhs, double* x, double tol,
                              int max_iter, int precond, fp_solve_info* info, void* stream) {
    if (!ctx || !ctx->field || !rhs || !x || (system != FP_SYS_NEWMARK && system != FP_SYS_GAUSS) ||
        !(tol > 0.0) || max_iter < 0 ||
        (precond != FP_PC_JACOBI && precond != FP_PC_JACOBI_FP64 && precond != FP_PC_LEARNED)) {
        if (ctx) ctx->err = "fem_pic_field_solve: bad argument (or fem_pic_field_setup not called)";
        return FP_EINVAL;
    }
    if (precond == FP_PC_LEARNED && !learned_precond_ready(ctx->field, system)) {
        ctx->err = "fem_pic_field_solve: FP_PC_LEARNED needs a built FP_LEARNED_PRECOND network for the system";
        return FP_EINVAL;
    }
    ctx->solver_fp64 = precond == FP_PC_JACOBI_FP64;
    learned_set_active(ctx->field, system, precond == FP_PC_LEARNED);
    ctx->field->learned_used[0] = precond == FP_PC_LEARNED;
    cudaStream_t s = (cudaStream_t)stream;
    cudaEvent_t a = nullptr, b = nullptr;
    if (info) {
        FP_CUDA_TRY(ctx, cudaEventCreate(&a));
        FP_CUDA_TRY(ctx, cudaEventCreate(&b));
        FP_CUDA_TRY(ctx, cudaEventRecord(a, s));
    }
    fp_status st = run_pcg(ctx, system, rhs, x, tol, nullptr, max_iter, 0, s);
    if (info && st == FP_OK) {
        float ms = 0.f;
        cudaEventRecord(b, s);
        cudaEventSynchronize(b);
        cudaEventElapsedTime(&ms, a, b);
        st = fill_info(ctx, 0, tol, info, s, ms);
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    return st;
}

fp_status fem_pic_field_step(fem_pic_t* ctx, const double* E_prev, const double* E_cur, double* E_next,
                             double* b, const void* dG_half, const void* dG_prev, const void* Q_new, double tol,
                             int max_iter, int precond, fp_solve_info info[2], void* stream) {
    if (!ctx || !ctx->field || !E_prev || !E_cur || !E_next || !Q_new || !(tol > 0.0) || max_iter < 0 ||
        (precond & ~(FP_PC_LEARNED | FP_PC_JACOBI_FP64 | FP_PC_LEARNED_GAUSS)) != 0 ||
        E_next == E_cur || E_next == E_prev) {
        if (ctx) ctx->err = "fem_pic_field_step: bad argument (or fem_pic_field_setup not called)";
        return FP_EINVAL;
    }
    const bool use[2] = {(precond & FP_PC_LEARNED) != 0, (precond & FP_PC_LEARNED_GAUSS) != 0};
    for (int k = 0; k < 2; ++k)
        if (use[k] && (!ctx->field->learned[k] || (learned_model(ctx->field, k) == FP_LEARNED_PRECOND &&
                                                    !learned_precond_ready(ctx->field, k)))) {
            ctx->err = "fem_pic_field_step: a learned correction needs fem_pic_learned_init for its system "
                       "(and fem_pic_learned_build for a learned preconditioner)";
            return FP_EINVAL;
        }
    ctx->solver_fp64 = (precond & FP_PC_JACOBI_FP64) != 0;
    for (int k = 0; k < 2; ++k) {
        learned_set_active(ctx->field, k, use[k]);
        ctx->field->learned_used[k] = use[k];
    }
    cudaStream_t s = (cudaStream_t)stream;
    fp_status st = field_step_impl(ctx, E_prev, E_cur, E_next, b, dG_half, dG_prev, Q_new, tol, max_iter, s);
    if (st != FP_OK || !info) return st;
    st = fill_info(ctx, 0, tol, &info[0], s, 0.f);
    const fp_status gs = fill_info(ctx, 1, tol, &info[1], s, 0.f);
    return st != FP_OK && (st != FP_ENOCONV || gs == FP_OK) ? st : gs;   // the graver of the two
}

fp_status fem_pic_field_initial(fem_pic_t* ctx, const void* Q, double* E, double tol, int max_iter,
                                fp_solve_info* info, void* stream) {
    if (!ctx || !ctx->field || !Q || !E || !(tol > 0.0) || max_iter < 0) {
        if (ctx) ctx->err = "fem_pic_field_initial: bad argument (or fem_pic_field_setup not called)";
        return FP_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    FieldDev* F = ctx->field;
    const bool f32 = Q_f32(ctx);   // Q is a float array
    const int gn = grid_of(ctx, F->nn), ge = grid_of(ctx, F->ne);
    FP_CUDA_TRY(ctx, cudaMemsetAsync(F->tmp, 0, F->ne * sizeof(double), s));
    if (f32)
        k_gauss_rhs<float><<<gn, kBlock, 0, s>>>(ctx->d_n2e_ptr, ctx->d_n2e_col, ctx->d_n2e_sgn, F->node_fixed, F->tmp,
                                                 (const float*)Q, F->nn, F->rhs, F->qd, nullptr, nullptr, nullptr,
                                                 0.0, 0, nullptr);
    else
        k_gauss_rhs<double><<<gn, kBlock, 0, s>>>(ctx->d_n2e_ptr, ctx->d_n2e_col, ctx->d_n2e_sgn, F->node_fixed,
                                                  F->tmp, (const double*)Q, F->nn, F->rhs, F->qd, nullptr, nullptr, nullptr,
                                                  0.0, 0, nullptr);
    fp_status st = neumann_rhs(ctx, s);
    if (st == FP_OK)
        st = run_pcg(ctx, FP_SYS_GAUSS, F->rhs, F->delta, tol, F->qd, max_iter, 1, s, nullptr, true);
    if (st == FP_OK) st = neumann_gauge(ctx, s);
    if (st != FP_OK) return st;
    k_project<<<ge, kBlock, 0, s>>>(ctx->d_edges, F->edge_fixed, F->delta, F->tmp, F->ne, E);
    FP_CUDA_TRY(ctx, cudaGetLastError());
    if (info) {
        st = fill_info(ctx, 1, tol, info, s, 0.f);
    }
    return st;
}

}  // extern "C"
