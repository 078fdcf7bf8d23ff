// Mixed-precision field solve whose operator is streamed from HBM (or L2) once per product.
//
// The method is pcg.cuh's, here for systems whose FP32 operator does not fit in the SMs' shared
// memory (cube meshes on 152 SMs: the edge system from 34^3, 33^3 with the polynomial's two more
// vectors; the node system from about 66^3, 64^3 with them).  A product reads its operator once,
// so it is bound by the operator's bytes and, behind them, by the latency of the chain
// column -> gathered entry.  So here
//  - the operator is packed into one record per 32-row slice: per slot a 32-bit base column, per
//    entry a 16-bit column offset (relative to base + lane) and the value: 6.1 bytes per FP32
//    entry instead of 8 (the learned correction 4.1 instead of 6, the FP64 operator 10.1
//    instead of 12); a slice whose offsets do not fit keeps 32-bit columns;
//  - a producer warp streams the block's records, a tile of one slice per consumer warp at a time,
//    into a ring in shared memory with bulk copies (evict-first in L2 where the operator is
//    larger than L2), so that columns and values cost a shared-memory read and only the gather
//    waits; the copies of the next product start before the grid sum that precedes it;
//  - the vectors' own rows are loaded one tile ahead of their use;
//  - c += alpha p waits for the next product, which reads p anyway, and vector passes move 16
//    bytes per lane.
// Measured per Jacobi iteration, against a kernel that read columns and values from global memory
// with an L2 prefetch one step ahead: edge system of the 64^3 mesh (1.9M rows) 67 -> 49 us, of
// 96^3 (6.3M rows) 235 -> 184 us (945 MB: 75% of a 6.8 TB/s copy), node system of 96^3 31 -> 24 us.
// With only the copies (no gather, no vectors) a 64^3 pass takes 36 us; the rest is the
// instructions per entry and the gather's latency.  Tried and slower: a ring per warp with
// its own copies (58 us), two slices per warp at once on 12 warps (67 us), 19 or 23 consumer warps
// (spills, 58 us), chunks of 8 gathers (52 us).
#include <algorithm>
#include <cmath>

#include "async_copy.cuh"
#include "field.cuh"
#include "grid_sync.cuh"
#include "pcg.cuh"

namespace fempic {
namespace {

constexpr int kStreamThreads = 32 * (kConsumers + 1);
constexpr int kStreamBars = 4;                       // tiles in flight, at most
constexpr uint64_t kCopyWaitNs = 2000000000ull;

// rows that a pass reads once: past L1, whose room the gathered vector needs
template <typename T>
__device__ __forceinline__ T ld_row(const T* p) {
    if constexpr (sizeof(T) == 4) {
        float v;
        asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    } else {
        double v;
        asm volatile("ld.global.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
        return v;
    }
}
__device__ __forceinline__ float4 ld_row4(const float* p) {
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint64_t evict_first_policy() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// shared-memory loads by 32-bit address
__device__ __forceinline__ uint32_t lds32(uint32_t p) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(p));
    return v;
}
__device__ __forceinline__ int2 lds64(uint32_t p) {
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(p));
    return v;
}
__device__ __forceinline__ void lds_val(uint32_t p, float* v) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(*v) : "r"(p)); }
__device__ __forceinline__ void lds_val(uint32_t p, double* v) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(*v) : "r"(p)); }

// The block's walk over its tiles of an operator.  A tile is kConsumers consecutive slices, one per
// consumer warp: a header {offset, slots} per slice, then their records, copied by one bulk copy.
// The last warp (its lane 0) issues the copies as the consumers free their places; tile n uses
// barrier n mod kStreamBars, phase n / kStreamBars.  Items are (tile, segment) pairs: slices of more
// than seg slots are stored as several records.
struct Ring {
    const StreamArgs& a;
    unsigned char* buf;
    uint64_t *full, *empty;        // kStreamBars each
    unsigned long long* fail;      // shared: a wait ran out, the block leaves at its next exchange
    uint64_t policy;
    int lane, warp, t0, nt;        // the block's tiles
    uint32_t count;                // items so far, over the whole launch: issued (producer) or used (consumer)
    int op, items, next, slot;     // of the current pass; next: items issued or used
    bool producer, dead;

    __device__ __forceinline__ bool wait(uint64_t* bars, uint32_t n) {
        if (dead) return false;
        if (mbar_wait_bounded(bars + (n & (kStreamBars - 1)), (n / kStreamBars) & 1u, kCopyWaitNs)) return true;
        dead = true;
        *fail = 1;
        return false;
    }
    // producer's lane 0: the next item's copy
    __device__ __forceinline__ void issue() {
        const uint2 m = __ldg(a.meta[op] + (size_t)t0 * a.nseg + next);
        uint64_t* b = full + (count & (kStreamBars - 1));
        mbar_arrive_expect_tx(b, m.y);
        unsigned char* dst = buf + slot * a.stage[op];
        const unsigned char* src = a.rec[op] + (size_t)m.x * 16;
        if (a.evict_first) bulk_g2s_hint(dst, src, m.y, b, policy);
        else bulk_g2s(dst, src, m.y, b);
        ++count;
        ++next;
        slot = slot + 1 == a.nst[op] ? 0 : slot + 1;
    }
    // begins a pass over operator o: the first copies, once the pass before has been read
    __device__ __forceinline__ void start(int o) {
        op = o;
        items = nt * a.nseg;
        next = slot = 0;
        if (!producer || lane != 0) return;
        for (uint32_t n = count > kStreamBars ? count - kStreamBars : 0; n < count; ++n) wait(empty, n);
        fence_proxy_async_smem();
        while (!dead && next < items && next < a.nst[op]) issue();
    }
    // producer: the rest of the pass
    __device__ __forceinline__ void feed() {
        if (lane == 0)
            while (!dead && next < items)
                if (wait(empty, count - (uint32_t)a.nst[op])) issue();
        __syncwarp();
    }
    // consumer: the record of this warp's slice in the next item (shared address; w: slots and kWide)
    __device__ __forceinline__ uint32_t get(uint32_t* w) {
        const bool ok = wait(full, count);
        const uint32_t st = smem_u32(buf) + slot * a.stage[op];
        const int2 h = lds64(st + 8 * warp);
        *w = ok ? (uint32_t)h.y : 0u;
        return st + (uint32_t)h.x;
    }
    __device__ __forceinline__ void release() {
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + (count & (kStreamBars - 1)));
        ++count;
        slot = slot + 1 == a.nst[op] ? 0 : slot + 1;
    }
    // gives back what start() began and no pass has read
    __device__ __forceinline__ void drain() {
        const int begun = min(items, a.nst[op]);
        if (!producer)
            for (int k = 0; k < begun; ++k) {
                wait(full, count);
                release();
            }
        __syncwarp();
    }
};

template <int OP>
struct OpTypes;
template <>
struct OpTypes<OP_F32> {
    using X = float;
};
template <>
struct OpTypes<OP_LEARNED> {
    using X = float;
};
template <>
struct OpTypes<OP_F64> {
    using X = double;
};

// N slots of a record in shared memory: B its bases and C its columns (the lane's) from the first of
// them on, V the lane's values; xl: the gathered vector, already at the lane.  All N are gathered
// before any is used.  Of the last four slots only those below `left` exist (left >= N: all).
template <int OP, int N, bool WIDE, typename X>
__device__ __forceinline__ X slots(uint32_t B, uint32_t C, uint32_t V, const X* xl, int left, X s) {
    X xv[N];
#pragma unroll
    for (int u = 0; u < N; u += 2) {
        const bool in0 = u < N - 4 || u < left, in1 = u + 1 < N - 4 || u + 1 < left;
        xv[u] = xv[u + 1] = X(0);
        if constexpr (WIDE) {
            if (in0) xv[u] = xl[(int)lds32(C + 128 * u)];
            if (in1) xv[u + 1] = xl[(int)lds32(C + 128 * (u + 1))];
        } else if (in0) {
            const uint32_t d = lds32(C + 64 * u);
            const int2 b = lds64(B + 4 * u);
            xv[u] = xl[b.x + (int)(d & 0xffffu)];
            if (in1) xv[u + 1] = xl[b.y + (int)(d >> 16)];
        }
    }
#pragma unroll
    for (int u = 0; u < N; u += 2) {
        const bool in0 = u < N - 4 || u < left, in1 = u + 1 < N - 4 || u + 1 < left;
        if constexpr (OP == OP_LEARNED) {
            if (in0) {
                const uint32_t l = lds32(V + 64 * u);
                s = fmaf(__uint_as_float(l << 16), xv[u], s);
                s = fmaf(__uint_as_float(l & 0xffff0000u), xv[u + 1], s);   // an odd width's last half is zero
            }
        } else {
            X v0, v1;
            constexpr int kBytes = 32 * (int)sizeof(X);
            if (in0) {
                lds_val(V + kBytes * u, &v0);
                s = fma(v0, xv[u], s);
            }
            if (in1) {
                lds_val(V + kBytes * (u + 1), &v1);
                s = fma(v1, xv[u + 1], s);
            }
        }
    }
    return s;
}
// a whole record of w slots
template <int OP, bool WIDE, typename X>
__device__ __forceinline__ X record_dot(uint32_t st, uint32_t w, const X* x, int lane, X s) {
    constexpr int kVal = OP == OP_LEARNED ? 64 : 32 * (int)sizeof(X), kCol = WIDE ? 128 : 64;   // bytes per slot
    const X* xl = WIDE ? x : x + lane;
    uint32_t B = st, C = st + base_bytes(w, WIDE) + 4 * lane;
    uint32_t V = st + base_bytes(w, WIDE) + col_bytes(w, WIDE) + (OP == OP_F64 ? 8 : 4) * lane;
    int left = (int)w;
    for (; left > 16; left -= 16) {
        s = slots<OP, 16, WIDE>(B, C, V, xl, 16, s);
        B += 64, C += 16 * kCol, V += 16 * kVal;
    }
    if (left > 12) return slots<OP, 16, WIDE>(B, C, V, xl, left, s);
    if (left > 8) return slots<OP, 12, WIDE>(B, C, V, xl, left, s);
    if (left > 4) return slots<OP, 8, WIDE>(B, C, V, xl, left, s);
    return slots<OP, 4, WIDE>(B, C, V, xl, left, s);
}

// A pass over the block's tiles: for each row, F::load (its own vectors' entries, one tile ahead),
// then F::apply with the row's product.  start(OP) came before.
template <int OP, class F>
__device__ __forceinline__ void stream_pass(Ring& R, const typename OpTypes<OP>::X* x, F& f) {
    using X = typename OpTypes<OP>::X;
    const StreamArgs& a = R.a;
    if (R.producer) {
        R.feed();
        return;
    }
    constexpr int kStep = 32 * kConsumers;
    int64_t row = (int64_t)kStep * R.t0 + 32 * R.warp + R.lane;
    typename F::Row next{};
    if (R.nt > 0 && row < a.n) next = f.load(row);
    for (int t = 0; t < R.nt; ++t, row += kStep) {
        const typename F::Row mine = next;
        if (t + 1 < R.nt && row + kStep < a.n) next = f.load(row + kStep);
        X s = X(0);
        for (int g = 0; g < a.nseg; ++g) {
            uint32_t w;
            const uint32_t st = R.get(&w);
            if (row < a.n && w != 0u)
                s = (w & kWide) ? record_dot<OP, true>(st, w & 0xffffu, x, R.lane, s)
                                : record_dot<OP, false>(st, w, x, R.lane, s);
            R.release();
        }
        if (row < a.n) f.apply(row, mine, s);
    }
}

// ---- what a row does with its product
struct DirectionRows {       // q = A z + beta q, p = z + beta p, and the deferred c += alpha p of the step before
    const StreamArgs& a;
    bool first, c_first;     // first: q = A z, p = z; c_first: c holds nothing yet
    float beta, alpha, pq;
    struct Row {
        float z, p, q, c;
    };
    __device__ __forceinline__ Row load(int64_t i) const {
        Row r;
        r.z = a.z[i];
        r.p = first ? 0.f : ld_row(a.p + i);
        r.q = first ? 0.f : ld_row(a.q + i);
        r.c = first || c_first ? 0.f : ld_row(a.c + i);
        return r;
    }
    __device__ __forceinline__ void apply(int64_t i, const Row& r, float w) {
        const float pi = first ? r.z : r.z + beta * r.p, qi = first ? w : w + beta * r.q;
        if (!first) a.c[i] = r.c + alpha * r.p;
        a.p[i] = pi;
        a.q[i] = qi;
        pq += pi * qi;
    }
};
struct LearnedRows {         // z = D^-1 r + Dl r
    const StreamArgs& a;
    float rz, rr;
    struct Row {
        float r, di;
    };
    __device__ __forceinline__ Row load(int64_t i) const { return Row{a.r[i], ld_row(a.dinv32 + i)}; }
    __device__ __forceinline__ void apply(int64_t i, const Row& r, float t) {
        const float zi = r.di * r.r + t;
        a.z[i] = zi;
        rz += r.r * zi;
        rr += r.r * r.r;
    }
};
struct ChebyshevRows {       // one step of the recurrence (pcg.cuh)
    const StreamArgs& a;
    const float* dc;         // the step before
    float* dn;               // this step (null for the last)
    float c1, c2, rz, rr;
    struct Row {
        float di, s, d, z, r;
    };
    __device__ __forceinline__ Row load(int64_t i) const {
        return Row{ld_row(a.dinv32 + i), ld_row(a.s + i), dc[i], ld_row(a.z + i), dn ? 0.f : ld_row(a.r + i)};
    }
    __device__ __forceinline__ void apply(int64_t i, const Row& r, float t) {
        const float sn = r.s - r.di * t, dk = c1 * r.d + c2 * sn, zk = r.z + dk;
        a.s[i] = sn;
        a.z[i] = zk;
        if (dn) {
            dn[i] = dk;
        } else {
            rz += r.r * zk;
            rr += r.r * r.r;
        }
    }
};
struct ResidualRows {        // r64 = b - A x
    const StreamArgs& a;
    bool ref;                // also the norms the tolerance refers to
    double rr, bb, ss;
    struct Row {
        double b, s;
    };
    __device__ __forceinline__ Row load(int64_t i) const { return Row{ld_row(a.pb + i), ref && a.scale_vec ? ld_row(a.scale_vec + i) : 0.0}; }
    __device__ __forceinline__ void apply(int64_t i, const Row& r, double t) { take(i, r, r.b - t); }
    __device__ __forceinline__ void take(int64_t i, const Row& r, double ri) {
        a.r64[i] = ri;
        rr += ri * ri;
        if (ref) bb += r.b * r.b, ss += r.s * r.s;
    }
};

__global__ void __launch_bounds__(kStreamThreads, 1) k_pcg_stream(StreamArgs a) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ GridSyncShared shs;
    __shared__ __align__(8) uint64_t full[kStreamBars], empty[kStreamBars];
    if (blockIdx.x == 0 && threadIdx.x == blockDim.x - 1) solve_begin(a.out);
    GridSync<false> g;
    g.init(a.sync, &shs, a.status);
    const int lane = g.lane, warp = g.wid;
    const int t0 = min(a.nt, (int)blockIdx.x * a.tpb), nt = min(a.nt, t0 + a.tpb) - t0;
    const int s0 = t0 * kConsumers, nsl = min(a.ns, s0 + nt * kConsumers) - s0;
    if (threadIdx.x == 0) {
        for (int k = 0; k < kStreamBars; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], kConsumers);
        }
        mbar_fence_init();
    }
    __syncthreads();
    Ring R{a, dsm, full, empty, &shs.rest[kFail]};
    R.policy = evict_first_policy();
    R.lane = lane, R.warp = warp, R.t0 = t0, R.nt = nt;
    R.count = 0;
    R.op = OP_F32, R.items = R.next = R.slot = 0;
    R.producer = warp == kConsumers, R.dead = false;
    // rows of the block, four per lane in the vector passes (vectors have room for whole slices)
    const int64_t r0 = (int64_t)32 * s0, r1 = min(a.n, (int64_t)32 * (s0 + nsl));
    const int64_t q0 = r0 / 4 + threadIdx.x, q1 = r1 / 4, qs = blockDim.x;
    const int64_t rest = 4 * q1 + threadIdx.x;   // the last rows of a count that is no multiple of 4
    const bool b0t0 = blockIdx.x == 0 && threadIdx.x == 0;
    __shared__ Refinement ref;
    int total = 0, outer = 0;
    bool use_l = a.learned;   // every block takes the same decisions (grid sums)
    if (use_l && a.lflag && b0t0) *a.lflag = 0;
    auto product_op = [&]() { return use_l ? OP_LEARNED : OP_F32; };   // the first product of an iteration

    // one entry of a vector step: r (and z or the recurrence's start) from r or r64
    float alpha = 0.f, w[2] = {0.f, 0.f};
    double rinv = 0.0;
    auto step1 = [&](float r, float di, float* z, float* s, float* d) {
        if (!use_l) {
            if (a.deg <= 1) {
                *z = di * r;
                w[0] += r * *z;
                w[1] += r * r;
            } else {
                *s = di * r;
                *z = *d = *s / a.theta;
            }
        }
    };
    // the vector step before a preconditioner: r <- r64 / ||r|| (init) or r - alpha q
    auto vectors = [&](bool init) {
        w[0] = w[1] = 0.f;
        const bool jac = !use_l && a.deg <= 1, poly = !use_l && a.deg > 1;
        // two groups of four rows in flight: their loads before any store
        for (int64_t qa = q0; qa < q1; qa += 2 * qs) {
            float4 r[2], di[2];
            float4 o[2], y[2];
            double2 x0[2], x1[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int64_t q = qa + k * qs;
                di[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (q >= q1) continue;
                if (!use_l) di[k] = ld_row4(a.dinv32 + 4 * q);
                if (init) {
                    x0[k] = reinterpret_cast<const double2*>(a.r64)[2 * q];
                    x1[k] = reinterpret_cast<const double2*>(a.r64)[2 * q + 1];
                } else {
                    o[k] = ld_row4(a.r + 4 * q);
                    y[k] = ld_row4(a.q + 4 * q);
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int64_t q = qa + k * qs;
                if (q >= q1) continue;
                if (init)
                    r[k] = make_float4(d2f(x0[k].x * rinv), d2f(x0[k].y * rinv), d2f(x1[k].x * rinv), d2f(x1[k].y * rinv));
                else
                    r[k] = make_float4(o[k].x - alpha * y[k].x, o[k].y - alpha * y[k].y, o[k].z - alpha * y[k].z,
                                       o[k].w - alpha * y[k].w);
                float4 z = make_float4(0.f, 0.f, 0.f, 0.f), s = z, d = z;
                reinterpret_cast<float4*>(a.r)[q] = r[k];
                step1(r[k].x, di[k].x, &z.x, &s.x, &d.x);
                step1(r[k].y, di[k].y, &z.y, &s.y, &d.y);
                step1(r[k].z, di[k].z, &z.z, &s.z, &d.z);
                step1(r[k].w, di[k].w, &z.w, &s.w, &d.w);
                if (jac || poly) reinterpret_cast<float4*>(a.z)[q] = z;
                if (poly) {
                    reinterpret_cast<float4*>(a.s)[q] = s;
                    reinterpret_cast<float4*>(a.d0)[q] = d;
                }
            }
        }
        if (rest < r1) {
            const float r = init ? d2f(a.r64[rest] * rinv) : a.r[rest] - alpha * a.q[rest];
            float z = 0.f, s = 0.f, d = 0.f;
            a.r[rest] = r;
            step1(r, use_l ? 0.f : __ldg(a.dinv32 + rest), &z, &s, &d);
            if (jac || poly) a.z[rest] = z;
            if (poly) a.s[rest] = s, a.d0[rest] = d;
        }
    };
    // z = P(r) after the vector step; w: this lane's r.z and r.r
    auto precondition = [&](bool init) -> bool {
        vectors(init);
        if (use_l) {
            if (!g.barrier()) return false;
            LearnedRows f{a, 0.f, 0.f};
            stream_pass<OP_LEARNED>(R, a.r, f);
            w[0] = f.rz, w[1] = f.rr;
            R.start(OP_F32);
        } else if (a.deg > 1) {
            const float sig = a.theta / a.delta;
            float rho = 1.f / sig;
            for (int k = 1; k < a.deg; ++k) {
                if (!g.barrier()) return false;
                const float rn = 1.f / (2.f * sig - rho);
                ChebyshevRows f{a, (k & 1) ? a.d0 : a.d1, k + 1 < a.deg ? ((k & 1) ? a.d1 : a.d0) : nullptr,
                                rn * rho, 2.f * rn / a.delta, 0.f, 0.f};
                stream_pass<OP_F32>(R, f.dc, f);
                w[0] = f.rz, w[1] = f.rr;
                R.start(OP_F32);
                rho = rn;
            }
        }
        return true;
    };

    auto solve = [&]() -> bool {
        // right-hand side and start in row order
        if (a.perm) {
            for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
                const int k = __ldg(a.perm + i);
                a.pb[i] = __ldg(a.b + k);
                a.px[i] = a.x_zero ? 0.0 : a.x[k];
            }
        } else if (a.x_zero) {
            for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) a.px[i] = 0.0;
        }
        if (!a.r0) R.start(OP_F64);
        if (!g.barrier()) return false;
        for (;;) {
            // ---- outer residual in FP64
            double v[3];
            {
                ResidualRows f{a, outer == 0, 0.0, 0.0, 0.0};
                if (a.r0 && outer == 0) {
                    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x)
                        f.take(i, f.load(i), __ldg(a.r0 + (a.perm ? __ldg(a.perm + i) : i)));
                } else {
                    stream_pass<OP_F64>(R, a.px, f);
                }
                v[0] = f.rr, v[1] = f.bb, v[2] = f.ss;
            }
            R.start(product_op());
            if (!g.sum64(v, [&](const double (&t)[3]) { ref.set(t, outer == 0, a.scale_vec, a.tol, a.inner_tol); }))
                return false;
            if (ref.stop || total >= a.max_iter || outer >= a.max_outer) return true;
            ++outer;
            // ---- inner FP32 PCG on A c = r / ||r||
            rinv = ref.rinv;
            float rz = 0.f, rr = 0.f, pq = 0.f, ithr = 0.f;
            float g_rz = 1.f, g_rr = 1.f, g_pq = 1.f;   // by how much each sum changed last
            // init: the first direction; c_first: c holds nothing yet; step: c += alpha p is still to
            // be done; restart: the learned operator is not positive on the first r
            bool init = true, c_first = true, step = false, restart = false;
            for (;;) {
                if (!precondition(init)) return false;
                const float ew[2] = {init ? 0.f : rz * g_rz, init ? 1.f : rr * g_rr};   // ||r|| is 1 at first
                if (!g.sum(w, ew)) return false;
                if (!init) {
                    g_rz = w[0] / rz, g_rr = w[1] / rr;
                    ++total;
                    if (!(w[1] > ithr)) break;
                }
                if (use_l && !(w[0] > 0.f)) {   // not positive on this r: keep c, Jacobi from here on
                    use_l = false;
                    if (a.lflag && b0t0) *a.lflag = 1;
                    restart = init;
                    break;
                }
                DirectionRows f{a, init, c_first, init ? 0.f : w[0] / rz, alpha, 0.f};
                rz = w[0], rr = w[1];
                if (init) ithr = ref.red * ref.red * rr;
                stream_pass<OP_F32>(R, a.z, f);
                R.start(product_op());
                float y[1] = {f.pq};
                const float ey[1] = {init ? 0.f : pq * g_pq};
                if (!g.sum(y, ey)) return false;
                if (!init) {
                    g_pq = y[0] / pq;
                    c_first = false;
                }
                step = init = false;
                pq = y[0];
                if (!(pq > 0.f) || total >= a.max_iter) break;
                alpha = rz / pq;
                step = true;
            }
            R.drain();
            R.start(OP_F64);
            if (restart) continue;   // x is unchanged: the refinement starts again with Jacobi
            // x += ||r|| c, with the last step's alpha p
            const double rnorm = ref.rnorm;
            if (!c_first || step)
                for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
                    const float ci = c_first ? 0.f : a.c[i];
                    a.px[i] += rnorm * f2d(step ? ci + alpha * a.p[i] : ci);
                }
            if (!g.barrier()) return false;
        }
    };
    const bool done = solve();
    R.drain();
    if (R.dead) atomicOr(a.status, ST_TIMEOUT);
    if (!done) return;
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
        const int64_t k = a.perm ? __ldg(a.perm + i) : i;
        if (a.perm) a.x[k] = a.px[i];
        if (a.ax) a.ax[k] = a.pb[i] - a.r64[i];
    }
    if (b0t0) {
        g.finish();
        a.out[0] = (double)total;
        a.out[1] = ref.rr;
        a.out[2] = ref.ref2;
        a.out[3] = (double)outer;
        if (!solve_met(ref.rr, ref.thr)) atomicOr(a.status, ST_NOCONV);
    }
}

// ---- packing (at setup, a warp per item)
// entry of lane `lane` (row i) at slot j of its slice: its column; padding entries keep the row itself
__device__ __forceinline__ bool real_entry(const Sell& S, const double* val, int64_t k, int64_t i) {
    return !(__ldg(S.col + k) == (int32_t)i && __ldg(val + k) == 0.0);
}
// range of col - lane over the real entries of slot k0 (lane 0's position); lo > hi: none
__device__ __forceinline__ void slot_range(const Sell& S, const double* val, int64_t k0, int64_t row0, int64_t n,
                                           int lane, int* lo, int* hi) {
    int l = INT32_MAX, h = INT32_MIN;
    if (row0 + lane < n && real_entry(S, val, k0 + lane, row0 + lane)) l = h = __ldg(S.col + k0 + lane) - lane;
    *lo = __reduce_min_sync(0xffffffffu, l);
    *hi = __reduce_max_sync(0xffffffffu, h);
}
// column written for lane: its own, or for padding one inside the slot's range and the vector
__device__ __forceinline__ int packed_col(const Sell& S, const double* val, int64_t k0, int64_t row0, int64_t n,
                                          int lane, int lo) {
    if (row0 + lane >= n) return lo + lane;   // never gathered
    if (real_entry(S, val, k0 + lane, row0 + lane)) return __ldg(S.col + k0 + lane);
    const int64_t c = (int64_t)lo + lane;
    return c >= 0 && c < n ? (int)c : (int)(row0 + lane);
}
__global__ void k_stream_widths(Sell S, const double* __restrict__ val, int64_t n, int ns, int nseg, int seg,
                                uint32_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t items = (int64_t)ns * nseg, stride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t it = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < items; it += stride) {
        const int s = (int)(it / nseg), g = (int)(it - (int64_t)s * nseg);
        const int w = min(seg, max(0, __ldg(S.w + s) - g * seg));
        bool wide = false;
        for (int u = 0; u < w; ++u) {
            const int64_t k0 = (int64_t)__ldg(S.ptr + s) + 32 * (int64_t)(g * seg + u), row0 = (int64_t)32 * s;
            int lo, hi;
            slot_range(S, val, k0, row0, n, lane, &lo, &hi);
            if (lo > hi) lo = hi = (int)row0;
            const int c = packed_col(S, val, k0, row0, n, lane, lo) - lane - lo;
            wide = wide || __any_sync(0xffffffffu, c < 0 || c > 65535);
        }
        if (lane == 0) out[it] = (uint32_t)w | (wide ? kWide : 0u);
    }
}
// where an item's record and its entry of the tile's header {offset inside the tile, slots and kWide} go
struct PackItem {
    unsigned long long rec, head;   // byte offsets
    uint32_t inside, w;
};
template <int OP, typename V>
__global__ void k_stream_pack(Sell S, const double* __restrict__ val, const V* __restrict__ v, int64_t n, int ns,
                              int nseg, int seg, const PackItem* __restrict__ where, unsigned char* __restrict__ rec) {
    const int lane = threadIdx.x & 31;
    const int64_t items = (int64_t)ns * nseg, stride = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t it = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); it < items; it += stride) {
        const int s = (int)(it / nseg), g = (int)(it - (int64_t)s * nseg);
        const PackItem m = where[it];
        const uint32_t w = m.w & 0xffffu;
        const bool wide = (m.w & kWide) != 0;
        unsigned char* st = rec + m.rec;
        if (lane == 0) *reinterpret_cast<uint2*>(rec + m.head) = make_uint2(m.inside, m.w);
        uint32_t* C = reinterpret_cast<uint32_t*>(st + base_bytes(w, wide)) + lane;
        unsigned char* vals = st + base_bytes(w, wide) + col_bytes(w, wide);
        const int64_t row0 = (int64_t)32 * s;
        uint32_t pair = 0, lpair = 0;
        for (uint32_t u = 0; u < w; ++u) {
            const int64_t k0 = (int64_t)__ldg(S.ptr + s) + 32 * (int64_t)(g * seg + (int)u);
            int lo, hi;
            slot_range(S, val, k0, row0, n, lane, &lo, &hi);
            if (lo > hi) lo = (int)row0;
            const int c = packed_col(S, val, k0, row0, n, lane, lo);
            if (wide) {
                C[32 * u] = row0 + lane < n ? (uint32_t)c : 0u;
            } else {
                if (lane == 0) reinterpret_cast<int*>(st)[u] = lo;
                const uint32_t d = (uint32_t)(c - lane - lo) & 0xffffu;
                pair = (u & 1u) ? pair | (d << 16) : d;
                if ((u & 1u) || u + 1 == w) C[32 * (u >> 1)] = pair;
            }
            if constexpr (OP == OP_LEARNED) {
                const uint32_t b = (uint32_t)__bfloat16_as_ushort(v[k0 + lane]);
                lpair = (u & 1u) ? lpair | (b << 16) : b;
                if ((u & 1u) || u + 1 == w) reinterpret_cast<uint32_t*>(vals)[32 * (u >> 1) + lane] = lpair;
            } else {
                reinterpret_cast<V*>(vals)[32 * u + lane] = v[k0 + lane];
            }
        }
    }
}

int pack_grid(const fem_pic* ctx) { return ctx->sm_count * 8; }

}  // namespace

void stream_free(StreamPlan* P) {
    for (int k = 0; k < OP_COUNT; ++k) {
        cudaFree(P->rec[k]);
        cudaFree(P->meta[k]);
        P->rec[k] = nullptr, P->meta[k] = nullptr;
    }
    cudaFree(P->where);
    P->where = nullptr;
    P->on = false;
}

// one operator's tiles: where its records go (the item of slice s, segment g is s nseg + g), the
// tiles' places and sizes, and room for them
static fp_status stream_layout(fem_pic* ctx, StreamPlan* P, int op, std::vector<PackItem>* where) {
    where->assign(P->width.size(), PackItem());
    std::vector<uint2> meta((size_t)P->nt * P->nseg);
    size_t off = 0;
    uint32_t most = 16;
    for (int t = 0; t < P->nt; ++t)
        for (int g = 0; g < P->nseg; ++g) {
            uint32_t in = kHeader;
            for (int k = 0; k < kConsumers && t * kConsumers + k < P->ns; ++k) {
                const size_t it = (size_t)(t * kConsumers + k) * P->nseg + g;
                (*where)[it] = PackItem{off + in, off + 8 * (size_t)k, in, P->width[it]};
                in += rec_bytes(P->width[it] & 0xffffu, (P->width[it] & kWide) != 0, op);
            }
            meta[(size_t)t * P->nseg + g] = make_uint2((uint32_t)(off / 16), in);
            off += in;
            most = std::max(most, in);
        }
    if (off / 16 > UINT32_MAX) {
        ctx->err = "fem_pic_field_setup: the operator is too large for the streamed solver";
        return FP_EINVAL;
    }
    P->bytes[op] = off;
    P->stage[op] = (int)tile_bytes(most);
    FP_CUDA_TRY(ctx, cudaMalloc((void**)&P->rec[op], off + 128));
    FP_CUDA_TRY(ctx, cudaMemset(P->rec[op], 0, off + 128));   // headers of slices past the last: no slots
    FP_CUDA_TRY(ctx, cudaMalloc((void**)&P->meta[op], meta.size() * sizeof(uint2) + 16));
    FP_CUDA_TRY(ctx, cudaMemcpy(P->meta[op], meta.data(), meta.size() * sizeof(uint2), cudaMemcpyHostToDevice));
    return FP_OK;
}

template <int OP, typename V>
static fp_status stream_pack(fem_pic* ctx, StreamPlan* P, const Sell& S, const double* val, const V* v,
                             const std::vector<PackItem>& where) {
    PackItem* d = nullptr;
    FP_CUDA_TRY(ctx, cudaMalloc((void**)&d, where.size() * sizeof(PackItem) + 16));
    cudaError_t e = cudaMemcpy(d, where.data(), where.size() * sizeof(PackItem), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        k_stream_pack<OP, V><<<pack_grid(ctx), 256>>>(S, val, v, P->n, P->ns, P->nseg, P->seg, d, P->rec[OP]);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d);
    FP_CUDA_TRY(ctx, e);
    return FP_OK;
}

fp_status stream_setup(fem_pic* ctx, const Sell& S, const double* val, const float* val32, int64_t n, int wmax,
                       StreamPlan* P) {
    stream_free(P);
    P->n = n;
    P->ns = (int)((n + 31) / 32);
    P->nt = (P->ns + kConsumers - 1) / kConsumers;
    int optin = 0;
    FP_CUDA_TRY(ctx, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    cudaFuncAttributes fa;
    FP_CUDA_TRY(ctx, cudaFuncGetAttributes(&fa, (const void*)k_pcg_stream));
    const size_t room = ((size_t)optin - fa.sharedSizeBytes) & ~(size_t)127;
    stream_segments(wmax, room, &P->nseg, &P->seg);
    const size_t items = (size_t)P->ns * P->nseg;
    uint32_t* d = nullptr;
    FP_CUDA_TRY(ctx, cudaMalloc((void**)&d, items * 4 + 16));
    k_stream_widths<<<pack_grid(ctx), 256>>>(S, val, n, P->ns, P->nseg, P->seg, d);
    P->width.resize(items);
    const cudaError_t e = cudaMemcpy(P->width.data(), d, items * 4, cudaMemcpyDeviceToHost);
    cudaFree(d);
    FP_CUDA_TRY(ctx, e);
    std::vector<PackItem> where;
    fp_status st = stream_layout(ctx, P, OP_F32, &where);
    if (st == FP_OK) st = stream_pack<OP_F32, float>(ctx, P, S, val, val32, where);
    if (st == FP_OK) st = stream_layout(ctx, P, OP_F64, &where);
    if (st == FP_OK) st = stream_pack<OP_F64, double>(ctx, P, S, val, val, where);
    if (st != FP_OK) return st;
    FP_CUDA_TRY(ctx, cudaFuncSetAttribute((const void*)k_pcg_stream, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room));
    P->ring = (int)std::min(room, std::max(kStreamRing, (size_t)2 * P->stage[OP_F64]));
    if (P->ring < P->stage[OP_F64]) {
        ctx->err = "fem_pic_field_setup: a tile does not fit in the streamed solver's ring";
        return FP_ECUDA;
    }
    const int nb = std::min(ctx->sm_count, 255);
    P->tpb = (P->nt + nb - 1) / nb;
    P->grid = (P->nt + P->tpb - 1) / P->tpb;
    P->on = true;
    return FP_OK;
}

fp_status stream_learned_room(fem_pic* ctx, StreamPlan* P) {
    if (!P->on || P->rec[OP_LEARNED]) return FP_OK;
    std::vector<PackItem> where;
    fp_status st = stream_layout(ctx, P, OP_LEARNED, &where);
    if (st == FP_OK) {
        const size_t bytes = where.size() * sizeof(PackItem);
        cudaError_t e = cudaMalloc(&P->where, bytes + 16);
        if (e == cudaSuccess) e = cudaMemcpy(P->where, where.data(), bytes, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            ctx->err = std::string("fem_pic_learned_init: the streamed solver's records: ") + cudaGetErrorString(e);
            st = FP_ECUDA;
        }
    }
    if (st != FP_OK) {   // all of it or nothing: the packing takes records for complete
        cudaFree(P->rec[OP_LEARNED]);
        cudaFree(P->meta[OP_LEARNED]);
        cudaFree(P->where);
        P->rec[OP_LEARNED] = nullptr, P->meta[OP_LEARNED] = nullptr, P->where = nullptr;
    }
    return st;
}

fp_status stream_learned_pack(fem_pic* ctx, StreamPlan* P, const Sell& S, const double* val, const __nv_bfloat16* pre,
                              cudaStream_t s) {
    if (!P->on || !P->rec[OP_LEARNED]) return FP_OK;
    k_stream_pack<OP_LEARNED, __nv_bfloat16><<<pack_grid(ctx), 256, 0, s>>>(
        S, val, pre, P->n, P->ns, P->nseg, P->seg, static_cast<const PackItem*>(P->where), P->rec[OP_LEARNED]);
    FP_CUDA_TRY(ctx, cudaGetLastError());
    return FP_OK;
}

fp_status stream_solve(fem_pic* ctx, const StreamPlan& P, StreamArgs a, cudaStream_t s) {
    int l2 = 0;
    FP_CUDA_TRY(ctx, cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, ctx->device));
    for (int k = 0; k < OP_COUNT; ++k) {
        a.rec[k] = P.rec[k], a.meta[k] = P.meta[k], a.stage[k] = std::max(P.stage[k], 16);
        a.nst[k] = std::max(1, std::min(kStreamBars, P.ring / a.stage[k]));
    }
    a.ns = P.ns, a.nt = P.nt, a.nseg = P.nseg, a.tpb = P.tpb, a.n = P.n;
    // operators that stay in L2 beside the vectors are read from it; larger ones go through without
    // displacing the vectors
    const size_t held = P.bytes[OP_F32] + (a.learned ? P.bytes[OP_LEARNED] : 0) + (size_t)6 * P.n * sizeof(float);
    a.evict_first = held > (size_t)l2 * 3 / 4;
    void* args[] = {&a};
    FP_CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)k_pcg_stream, dim3(P.grid), dim3(kStreamThreads), args,
                                                 (size_t)P.ring, s));
    return FP_OK;
}

}  // namespace fempic
