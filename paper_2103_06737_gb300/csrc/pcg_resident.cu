// Mixed-precision field solve with everything an iteration touches held on chip.
//
// The method is pcg.cuh's, here for systems of which a block's share of the FP32 operator and of
// the solver's vectors fits in its shared memory.  A solve of such a system
// moves almost no memory; its time is the latency of each iteration's chain: products that wait
// on gathered entries, and grid-wide sums.  So here
//  - a lane owns the same rows through the whole solve and keeps their r, z, p, q, c and D^-1
//    (and the polynomial's two vectors) in shared memory; only the vector that the next
//    product gathers is written out to global memory;
//  - operator entries lie in shared memory in pairs of a row's consecutive slots (8 bytes of
//    values, 4 bytes of 16-bit column offsets), copied by the lane that uses them;
//  - sums and barriers take one trip through L2 (grid_sync.cuh);
//  - a system of at most 1024 rows runs in one block, with the gathered vectors in shared
//    memory too and block barriers only;
//  - right-hand side, starting point and solution are read and written in DOF order through
//    the row permutation, without separate gather and scatter launches.
// Bound by latency: per Jacobi iteration two exchanges (1.5 us each on 152 blocks), one product
// (about 1 us for one slice a warp, 4 us for two slices a warp of the edge system).  Measured on
// the 32^3 mesh, per solve, against a kernel with the same operator in shared memory, vectors in
// global memory and cooperative-groups barriers: edge system 565 -> 352 us (17 iterations of degree
// 3), node system 253 -> 175 us (7 of degree 8); 4^3 mesh (one block) 141 -> 59 us and 52 -> 19 us.
// Two or three rows a lane in registers instead of shared memory spilled at the 80 registers that
// 800 threads leave; vectors in shared memory cost no time that shows.
#include <algorithm>
#include <cmath>

#include "field.cuh"
#include "grid_sync.cuh"
#include "pcg.cuh"

namespace fempic {
namespace {

// The two signed 16-bit column offsets of a slot pair, in 32-bit registers throughout.  Earlier builds
// that held them in 16-bit registers, and spilled those, read out of range; the spill is the
// suspected cause, not a proven one.  Every offset is range-checked where it enters shared memory.
__device__ __forceinline__ int offset_lo(int d) {
    int o;
    asm("bfe.s32 %0, %1, 0, 16;" : "=r"(o) : "r"(d));
    return o;
}
__device__ __forceinline__ int offset_hi(int d) { return d >> 16; }

// Row of an operator times x, xr = x + row: the lane's slot pairs are d[32 u] (column offsets) and
// v(u) (values), u < pairs.  PC pairs are gathered before any is used; the last pairs % PC, where
// there are any, in one more round.
template <int PC, class V>
__device__ __forceinline__ float row_dot(const int* d, const V& v, int pairs, const float* xr) {
    float s = 0.f, t = 0.f;
    int u0 = 0;
    for (; u0 + PC <= pairs; u0 += PC) {
        float xa[PC], xb[PC];
#pragma unroll
        for (int u = 0; u < PC; ++u) {
            const int o = d[32 * (u0 + u)];
            xa[u] = xr[offset_lo(o)];
            xb[u] = xr[offset_hi(o)];
        }
#pragma unroll
        for (int u = 0; u < PC; ++u) {
            const float2 a = v(u0 + u);
            s = fmaf(a.x, xa[u], s);
            t = fmaf(a.y, xb[u], t);
        }
    }
    if (u0 < pairs) {
        float xa[PC - 1], xb[PC - 1];
#pragma unroll
        for (int u = 0; u < PC - 1; ++u) {
            const int o = u0 + u < pairs ? d[32 * (u0 + u)] : 0;
            xa[u] = xr[offset_lo(o)];
            xb[u] = xr[offset_hi(o)];
        }
#pragma unroll
        for (int u = 0; u < PC - 1; ++u)
            if (u0 + u < pairs) {
                const float2 a = v(u0 + u);
                s = fmaf(a.x, xa[u], s);
                t = fmaf(a.y, xb[u], t);
            }
    }
    return s + t;
}

struct SharedValues {   // the operator's slot pairs in shared memory
    const float2* v;
    __device__ __forceinline__ float2 operator()(int u) const { return v[32 * u]; }
};
struct LearnedValues {  // the learned correction's slots, from global memory (SELL order)
    const __nv_bfloat16* l;
    int w;
    __device__ __forceinline__ float2 operator()(int u) const {
        return make_float2(__bfloat162float(__ldg(l + 64 * u)),
                           2 * u + 1 < w ? __bfloat162float(__ldg(l + 64 * u + 32)) : 0.f);
    }
};

// per-row vectors of a block in shared memory, in this order (the last two for the polynomial only)
enum { RV_R, RV_Z, RV_P, RV_Q, RV_C, RV_DI, RV_JACOBI, RV_S = RV_JACOBI, RV_D, RV_COUNT };

template <int THREADS, bool ONE>
struct Resident {
    static constexpr int PC = THREADS <= 512 ? 8 : 4;   // slot pairs of a row in flight
    const ResidentArgs& a;
    GridSync<ONE>& g;
    int lane, warp, W, s0, nsl, rows_pb;
    const int* sp;          // shared: slot pairs before each of the block's slices
    float2* sv;
    int* sd;                // two 16-bit column offsets per word
    float* vec;             // shared: RV_COUNT vectors of rows_pb rows
    float *xz, *x0, *x1;    // gathered vectors by solver row (one block: shared)

    __device__ __forceinline__ float* at(int v) const { return vec + v * rows_pb; }

    // z = P(r), published in xz (the next exchange makes it visible), after the step c += alpha p,
    // r -= alpha q of the inner CG where `step`; this lane's share of r.z and r.r is added to w
    __device__ __forceinline__ bool precondition(bool use_l, bool step, float alpha, float (&w)[2]) {
        float *r = at(RV_R), *z = at(RV_Z), *p = at(RV_P), *q = at(RV_Q), *c = at(RV_C), *di = at(RV_DI);
        auto residual = [&](int i) {
            float ri = r[i];
            if (step) {
                c[i] += alpha * p[i];
                ri -= alpha * q[i];
                r[i] = ri;
            }
            return ri;
        };
        if (!use_l && a.deg <= 1) {
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row >= a.n) continue;
                const float ri = residual(i), zi = di[i] * ri;
                xz[row] = z[i] = zi;
                w[0] += ri * zi;
                w[1] += ri * ri;
            }
            return true;
        }
        if (use_l) {
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row < a.n) x0[row] = residual(i);
            }
            if (!g.barrier()) return false;
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row >= a.n) continue;
                const LearnedValues lv{a.dl16 + __ldg(a.S.ptr + s0 + s) + lane, __ldg(a.S.w + s0 + s)};
                const float t = row_dot<PC>(sd + 32 * sp[s] + lane, lv, sp[s + 1] - sp[s], x0 + row);
                const float ri = r[i], zi = di[i] * ri + t;
                xz[row] = z[i] = zi;
                w[0] += ri * zi;
                w[1] += ri * ri;
            }
            return true;
        }
        // Chebyshev recurrence (pcg.cuh)
        float *sr = at(RV_S), *d = at(RV_D);
        const float sig = a.theta / a.delta;
        float rho = 1.f / sig;
        for (int s = warp; s < nsl; s += W) {
            const int i = 32 * s + lane, row = 32 * s0 + i;
            if (row >= a.n) continue;
            const float f = di[i] * residual(i), d0 = f / a.theta;
            sr[i] = f;
            z[i] = d0;
            d[i] = d0;
            x0[row] = d0;
        }
        for (int k = 1; k < a.deg; ++k) {
            if (!g.barrier()) return false;
            const float rn = 1.f / (2.f * sig - rho), c1 = rn * rho, c2 = 2.f * rn / a.delta;
            const float* x = (k & 1) ? x0 : x1;
            const bool last = k + 1 == a.deg;                     // publishes z instead of d
            float* nx = last ? xz : (k & 1) ? x1 : x0;
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row >= a.n) continue;
                const int o = 32 * sp[s] + lane;
                const float t = row_dot<PC>(sd + o, SharedValues{sv + o}, sp[s + 1] - sp[s], x + row);
                const float sn = sr[i] - di[i] * t;
                const float dk = c1 * d[i] + c2 * sn;
                const float zk = z[i] + dk;
                sr[i] = sn;
                d[i] = dk;
                z[i] = zk;
                nx[row] = last ? zk : dk;
                if (last) {
                    const float ri = r[i];
                    w[0] += ri * zk;
                    w[1] += ri * ri;
                }
            }
            rho = rn;
        }
        return true;
    }

    // q = A z + beta q, p = z + beta p (first: q = A z, p = z); this lane's share of p.q
    __device__ __forceinline__ float direction(bool first, float beta) {
        float *z = at(RV_Z), *p = at(RV_P), *q = at(RV_Q);
        float pq = 0.f;
        for (int s = warp; s < nsl; s += W) {
            const int i = 32 * s + lane, row = 32 * s0 + i;
            if (row >= a.n) continue;
            const int o = 32 * sp[s] + lane;
            const float w = row_dot<PC>(sd + o, SharedValues{sv + o}, sp[s + 1] - sp[s], xz + row);
            const float zi = z[i];
            const float pi = first ? zi : zi + beta * p[i];
            const float qi = first ? w : w + beta * q[i];
            p[i] = pi;
            q[i] = qi;
            pq += pi * qi;
        }
        return pq;
    }

    // the whole solve; false when a wait ran out (in every thread of the block alike)
    __device__ bool solve(int& total, int& outer, Refinement& f) {
        const bool b0t0 = blockIdx.x == 0 && threadIdx.x == 0;
        bool use_l = a.dl16 != nullptr;   // every block takes the same decisions (grid sums)
        if (use_l && a.lflag && b0t0) *a.lflag = 0;
        double* px = a.px;
        float *r = at(RV_R), *c = at(RV_C);
        if (a.x_zero || a.perm) {
            for (int s = warp; s < nsl; s += W) {
                const int row = 32 * (s0 + s) + lane;
                if (row < a.n) px[row] = a.x_zero ? 0.0 : a.x[a.perm ? __ldg(a.perm + row) : row];
            }
            if (!a.r0 && !g.barrier()) return false;
        }
        for (;;) {
            // ---- outer residual in FP64
            double v[3] = {0.0, 0.0, 0.0};
            for (int s = warp; s < nsl; s += W) {
                const int row = 32 * (s0 + s) + lane;
                if (row >= a.n) continue;
                const int k = a.perm ? __ldg(a.perm + row) : row;
                const double b = __ldg(a.b + k);
                const double ri = a.r0 && outer == 0 ? __ldg(a.r0 + k) : b - sell_row_cached(a.S, a.val, px, row);
                a.r64[row] = ri;
                v[0] += ri * ri;
                if (outer == 0) {
                    v[1] += b * b;
                    if (a.scale_vec) {
                        const double sc = __ldg(a.scale_vec + k);
                        v[2] += sc * sc;
                    }
                }
            }
            if (!g.sum64(v, [&](const double (&t)[3]) { f.set(t, outer == 0, a.scale_vec, a.tol, a.inner_tol); }))
                return false;
            if (f.stop || total >= a.max_iter || outer >= a.max_outer) return true;
            ++outer;
            // ---- inner FP32 PCG on A c = r / ||r||
            const double rinv = f.rinv;
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row >= a.n) continue;
                r[i] = d2f(a.r64[row] * rinv);
                c[i] = 0.f;
            }
            // r.z, r.r, then p.q; ||r|| is 1, the others are not known yet
            float w[2] = {0.f, 0.f}, y[1];
            const float start[2] = {0.f, 1.f}, none[1] = {0.f};
            if (!precondition(use_l, false, 0.f, w) || !g.sum(w, start)) return false;
            if (use_l && !(w[0] > 0.f)) {   // the learned operator is not positive on r: Jacobi from here on
                use_l = false;
                if (a.lflag && b0t0) *a.lflag = 1;
                continue;                   // c is still 0: the refinement restarts with Jacobi
            }
            y[0] = direction(true, 0.f);
            if (!g.sum(y, none)) return false;
            float rz = w[0], rr = w[1], pq = y[0];
            // by how much each sum changed last, for what to expect of the next
            float g_rz = 1.f, g_rr = 1.f, g_pq = 1.f;
            const float ithr = f.red * f.red * rr;
            for (;;) {
                if (!(pq > 0.f) || total >= a.max_iter) break;
                const float alpha = rz / pq;
                w[0] = w[1] = 0.f;
                if (!precondition(use_l, true, alpha, w)) return false;
                const float ew[2] = {rz * g_rz, rr * g_rr};
                if (!g.sum(w, ew)) return false;
                g_rz = w[0] / rz, g_rr = w[1] / rr, rr = w[1];
                ++total;
                if (!(w[1] > ithr)) break;
                if (use_l && !(w[0] > 0.f)) {   // not positive on this r: keep c, Jacobi from here on
                    use_l = false;
                    if (a.lflag && b0t0) *a.lflag = 1;
                    break;
                }
                const float beta = w[0] / rz;
                rz = w[0];
                y[0] = direction(false, beta);
                const float ey[1] = {pq * g_pq};
                if (!g.sum(y, ey)) return false;
                g_pq = y[0] / pq;
                pq = y[0];
            }
            const double rnorm = f.rnorm;
            for (int s = warp; s < nsl; s += W) {
                const int i = 32 * s + lane, row = 32 * s0 + i;
                if (row < a.n) px[row] += rnorm * f2d(c[i]);
            }
            if (!g.barrier()) return false;
        }
    }
};

template <int THREADS, bool ONE>
__global__ void __launch_bounds__(THREADS, 1) k_pcg_resident(ResidentArgs a) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ GridSyncShared shs;
    __shared__ int sp[kResMaxSlices + 1];
    __shared__ Refinement f;
    if (!ONE && blockIdx.x == 0 && threadIdx.x == blockDim.x - 1) solve_begin(a.out);   // (one block does not give up)
    GridSync<ONE> g;
    g.init(a.sync, &shs, a.status);
    Resident<THREADS, ONE> S{a, g};
    S.lane = g.lane, S.warp = g.wid, S.W = g.warps;
    S.s0 = min(a.ns, (int)blockIdx.x * a.spb);
    S.nsl = min(a.ns, S.s0 + a.spb) - S.s0;
    S.rows_pb = 32 * a.spb;
    S.sp = sp;
    S.sv = reinterpret_cast<float2*>(dsm);
    S.sd = reinterpret_cast<int*>(dsm + (size_t)a.pairs_max * 32 * 8);
    S.vec = reinterpret_cast<float*>(dsm + (size_t)a.pairs_max * 32 * 12);
    S.xz = a.z, S.x0 = a.d0, S.x1 = a.d1;
    if (ONE) {
        float* v = S.vec + (a.deg > 1 ? RV_COUNT : RV_JACOBI) * S.rows_pb;
        S.xz = v, S.x0 = v + S.rows_pb, S.x1 = v + 2 * S.rows_pb;
    }
    for (int s = threadIdx.x; s <= S.nsl; s += blockDim.x) sp[s] = __ldg(a.pp + S.s0 + s) - __ldg(a.pp + S.s0);
    __syncthreads();
    // the operator's entries: each lane copies the rows it will use
    for (int s = S.warp; s < S.nsl; s += S.W) {
        const int i = 32 * s + S.lane, row = 32 * S.s0 + i;
        if (row >= a.n) continue;
        S.vec[RV_DI * S.rows_pb + i] = __ldg(a.dinv32 + row);
        const int o = 32 * sp[s] + S.lane, w = __ldg(a.S.w + S.s0 + s), pairs = sp[s + 1] - sp[s];
        const int64_t k0 = (int64_t)__ldg(a.S.ptr + S.s0 + s) + S.lane;
#pragma unroll 4
        for (int u = 0; u < pairs; ++u) {
            const int64_t k = k0 + 64 * (int64_t)u;
            const bool two = 2 * u + 1 < w;
            int d = (int)__ldg(a.d16u + k) | (two ? (int)__ldg(a.d16u + k + 32) << 16 : 0);
            // the only place that sets a gathered index: it stays inside the vector
            if ((unsigned)(row + offset_lo(d)) >= (unsigned)a.n || (unsigned)(row + offset_hi(d)) >= (unsigned)a.n) {
                atomicOr(a.status, ST_INVAL);
                d = 0;
            }
            S.sv[o + 32 * u] = make_float2(__ldg(a.val32 + k), two ? __ldg(a.val32 + k + 32) : 0.f);
            S.sd[o + 32 * u] = d;
        }
    }
    int total = 0, outer = 0;
    const bool done = S.solve(total, outer, f);
    if (done) {
        for (int s = S.warp; s < S.nsl; s += S.W) {
            const int row = 32 * (S.s0 + s) + S.lane;
            if (row >= a.n) continue;
            const int k = a.perm ? __ldg(a.perm + row) : row;
            if (a.perm) a.x[k] = a.px[row];
            if (a.ax) a.ax[k] = __ldg(a.b + k) - a.r64[row];
        }
    }
    if (done && blockIdx.x == 0 && threadIdx.x == 0) {
        g.finish();
        a.out[0] = (double)total;
        a.out[1] = f.rr;
        a.out[2] = f.ref2;
        a.out[3] = (double)outer;
        if (!solve_met(f.rr, f.thr)) atomicOr(a.status, ST_NOCONV);
    }
}

// threads of a block at most: 80 registers each without spills
constexpr int kResThreads = 800;

void* resident_kernel(int threads, bool one) {
    if (one) return (void*)k_pcg_resident<640, true>;
    return threads <= 512 ? (void*)k_pcg_resident<512, false> : (void*)k_pcg_resident<kResThreads, false>;
}

}  // namespace

// A block takes at least this many slices (fewer blocks for small systems: each exchange then has
// fewer words to wait for).
constexpr int kResMinSlices = 4;
fp_status resident_setup(fem_pic* ctx, int64_t n, const std::vector<int32_t>& width, ResidentPlan* P) {
    *P = ResidentPlan();
    const int64_t ns = (int64_t)width.size();
    if (ns < 1) return FP_OK;
    std::vector<int32_t> pp(ns + 1, 0);
    for (int64_t s = 0; s < ns; ++s) pp[s + 1] = pp[s] + (width[s] + 1) / 2;
    const bool one = n <= 1024;
    const int64_t nb0 = one ? 1 : std::min<int64_t>(std::min(ctx->sm_count, 255), (ns + kResMinSlices - 1) / kResMinSlices);
    const int64_t spb = (ns + nb0 - 1) / nb0;
    if (spb > kResMaxSlices) return FP_OK;
    const int64_t warps = one ? 20 : kResThreads / 32, rounds = (spb + warps - 1) / warps;   // slices per warp
    const int threads = 32 * (int)((spb + rounds - 1) / rounds);
    int64_t most = 0;
    for (int64_t s = 0; s < ns; s += spb) most = std::max<int64_t>(most, pp[std::min(ns, s + spb)] - pp[s]);
    int optin = 0;
    FP_CUDA_TRY(ctx, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    void* k = resident_kernel(threads, one);
    cudaFuncAttributes fa;
    FP_CUDA_TRY(ctx, cudaFuncGetAttributes(&fa, k));
    const size_t room = (size_t)optin - fa.sharedSizeBytes;
    const size_t op = (size_t)most * 32 * 12, vec = 32 * (size_t)spb * sizeof(float);
    const size_t plain = op + (RV_JACOBI + (one ? 3 : 0)) * vec, poly = op + (RV_COUNT + (one ? 3 : 0)) * vec;
    if (plain > room) return FP_OK;
    // the attribute is per kernel, shared by every context: the device's limit, so that no
    // context lowers it below what another one launches with
    FP_CUDA_TRY(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room));
    P->one = one;
    P->grid = (int)((ns + spb - 1) / spb);
    P->spb = (int)spb;
    P->threads = threads;
    P->pairs_max = (int)most;
    P->smem = plain;
    P->smem_poly = poly <= room ? poly : 0;
    FP_CUDA_TRY(ctx, cudaMalloc((void**)&P->pp, pp.size() * sizeof(int32_t)));
    FP_CUDA_TRY(ctx, cudaMemcpy(P->pp, pp.data(), pp.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
    P->on = true;
    return FP_OK;
}

fp_status resident_solve(fem_pic* ctx, const ResidentPlan& P, ResidentArgs a, cudaStream_t s) {
    a.pp = P.pp, a.spb = P.spb, a.pairs_max = P.pairs_max;
    void* args[] = {&a};
    FP_CUDA_TRY(ctx, cudaLaunchCooperativeKernel(resident_kernel(P.threads, P.one), dim3(P.grid), dim3(P.threads),
                                                 args, a.deg > 1 ? P.smem_poly : P.smem, s));
    return FP_OK;
}

}  // namespace fempic
