// Grid-wide sums and barriers of the cooperative solvers.
//
// A grid barrier is one trip to L2 to arrive and one to see the last arrival, about 1.2 us on
// 152 blocks; reading every block's partial sum after it is another trip (2.1-2.6 us for such a
// sum).  Here the sum rides on the arrival: a block adds {its partial as an integer, 1 arrival}
// to one 64-bit word, and the poll that sees the last arrival reads the total with it (1.5-1.7 us
// with the block's own reduction).  Integer addition is associative, so the total does not
// depend on the order of arrival and every block and every run gets the same bits.
//
//   bits 0-7 arrivals, 8-15 blocks whose partial does not fit, 16-63 signed sum of the partials
//   scaled by a power of two that all blocks choose alike from the sum's previous values, so
//   that the expected total lies near 2^36: partials below 2^39 fit, and the roundings of at most
//   255 partials, half a unit each, stay below 2^-24 of a total of at least 2^31, a float's own
//   rounding.  Otherwise (a sum that grew or fell more than that, a value that is not
//   finite) all blocks see it in the same word and add the floats, which came with the
//   exchange, themselves in block order.
//
// Words are never cleared: a block subtracts what the word held at its last exchange.  Two words
// are used in turn, since a block may arrive at the next exchange before another has read this
// one; it cannot arrive at the one after.  (Polling one array of all blocks' partials, or a
// mailbox of partials per block, measured 2.7-5 us: 152 blocks' words per exchange are more
// traffic than the trip they save.)
//
// Every wait is bounded: a block that does not see the others within the limit sets ST_EXCHANGE in
// the status word and a mark beside the words, and leaves (all its threads together); the others
// see the mark and follow.  The words then hold arrivals that belong to no exchange, so a launch
// that finds the mark leaves at its first exchange; fem_pic_status clears words and mark.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstring>

#include "internal.cuh"
#ifdef __CUDACC__
#include "async_copy.cuh"
#endif

namespace fempic {

// Limit of a wait.  A launch's first exchange also waits for blocks that have not started because a
// kernel of another stream still holds their SMs (30 s); the later ones only for blocks at work (2 s).
constexpr uint64_t kGridStartNs = 30000000000ull, kGridWaitNs = 2000000000ull;
// device memory of one handle's exchanges (zeroed at setup): the words at rest, the mark of an
// abandoned exchange and the solves' output words, read with it by one copy (GridReport); the words
// in use (two exchanges; a line each), then the blocks' partials for the sums that are added one by
// one (two copies of three doubles per block)
constexpr size_t kGridLine = 128, kGridMark = 32, kGridOut = 64;
struct GridReport {
    unsigned long long mark, pad[3];
    double out[8];               // four per info slot
};
static_assert(sizeof(GridReport) == kGridLine - kGridMark && offsetof(GridReport, out) == kGridOut - kGridMark,
              "GridReport layout");
constexpr int kFail = 4;
inline size_t grid_sync_bytes(int blocks) { return 3 * kGridLine + (size_t)2 * blocks * 3 * 8; }

// A sum's word: the exponent of its scale, a block's increment, and the total that the increments
// of all blocks stand for (false: to be added one by one).
constexpr int kWordExpect = 36;
constexpr float kWordFits = 549755813888.f;              // 2^39
constexpr long long kWordLeast = 1ll << 31;
__host__ __device__ inline float word_pow2(int e) {
    const uint32_t b = (uint32_t)(e + 127) << 23;
    float f;
    memcpy(&f, &b, 4);
    return f;
}
// power of two that takes a total of about `expect` near 2^kWordExpect (0: no expectation)
__host__ __device__ inline int word_exp(float expect) {
    uint32_t b;
    memcpy(&b, &expect, 4);
    const int e = (int)((b >> 23) & 0xffu), s = kWordExpect - (e - 127);
    return expect > 0.f && e > 0 && e < 255 ? (s < -96 ? -96 : s > 96 ? 96 : s) : 0;
}
__host__ __device__ inline unsigned long long word_put(float v, int e) {
    const float x = v * word_pow2(e);
    return (fabsf(x) < kWordFits ? (unsigned long long)llrintf(x) << 16 : 256ull) + 1ull;   // (a NaN does not fit)
}
__host__ __device__ inline bool word_total(unsigned long long d, int e, float* total) {
    const long long t = (long long)d >> 16;
    *total = (float)t * word_pow2(-e);
    return ((d >> 8) & 255ull) == 0 && (t >= kWordLeast || t <= -kWordLeast);
}

#ifdef __CUDACC__

struct GridSyncShared {
    double part64[3][32];
    float part[2][3][33];        // per-warp partials, by the exchange's parity
    float tot[2][2];
    // [2 par + k]: what each word held after this block's last exchange on it; [kFail]: not 0, the
    // block does not arrive any more (its own wait ran out, or the mark is set)
    unsigned long long rest[5];
    int state[2];                // bit 0: a wait ran out, bit 1: add the partials one by one
};

template <bool ONE>   // ONE: a single block, no exchange through memory
struct GridSync {
    char* mem;
    GridSyncShared* sh;
    int32_t* status;
    uint64_t limit, limit1;    // of a wait, ns; of the first
    uint32_t turn;             // exchanges so far
    int nb, lane, wid, warps;

    __device__ __forceinline__ void init(void* m, GridSyncShared* s, int32_t* st) {
        mem = static_cast<char*>(m);
        sh = s;
        status = st;
        limit = kGridWaitNs;
        limit1 = kGridStartNs;
        turn = 0;
        nb = gridDim.x;
        lane = threadIdx.x & 31;
        wid = threadIdx.x >> 5;
        warps = blockDim.x >> 5;
        // nothing changes the words at rest before every block's first arrival; the mark comes with them
        if (!ONE && threadIdx.x < 5) s->rest[threadIdx.x] =
            *reinterpret_cast<volatile unsigned long long*>(mem + 8 * threadIdx.x);
        if (ONE && threadIdx.x == 0) s->rest[kFail] = 0;
        __syncthreads();
    }
    __device__ __forceinline__ volatile int* mark() { return reinterpret_cast<volatile int*>(mem + kGridMark); }
    // one thread: the exchange is abandoned
    __device__ __forceinline__ void abandon() {
        atomicOr(status, ST_EXCHANGE);
        *mark() = 1;
    }
    // by one thread at the end of a launch whose waits all ended: the next launch starts here
    __device__ __forceinline__ void finish() {
        if constexpr (!ONE)
            for (int k = 0; k < 4; ++k)
                *reinterpret_cast<volatile unsigned long long*>(mem + 8 * k) = sh->rest[k];
    }
    __device__ __forceinline__ unsigned long long* word(int par) {
        return reinterpret_cast<unsigned long long*>(mem + kGridLine * (1 + par));
    }
    // one thread: adds q[0..NW) to the words of this exchange and waits until every block has;
    // the words' increments in d.  Makes what the block wrote before (ordered by the block
    // barrier) visible to the blocks that leave the exchange.
    template <int NW>
    __device__ __forceinline__ bool arrive_wait(int par, const unsigned long long (&q)[NW], unsigned long long (&d)[NW]) {
        unsigned long long* w = word(par);
        unsigned long long p[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) p[k] = sh->rest[2 * par + k];
        // the last addition releases, the load of that word acquires
#pragma unroll
        for (int k = 1; k < NW; ++k)
            asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(w + k), "l"(q[k]) : "memory");
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"(q[0]) : "memory");
        uint64_t t0 = 0;
        for (uint32_t spin = 0;; ++spin) {
            unsigned long long c[NW];
            bool all = true;
            // the acquire last: the loads are in flight together (a word whose arrivals are not
            // complete yet shows it in its own count)
#pragma unroll
            for (int k = 1; k < NW; ++k)
                asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(c[k]) : "l"(w + k) : "memory");
            asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(c[0]) : "l"(w) : "memory");
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                d[k] = c[k] - p[k];
                all = all && (int)(d[k] & 255ull) == nb;
            }
            if (all) {
#pragma unroll
                for (int k = 0; k < NW; ++k) sh->rest[2 * par + k] = c[k];
                return true;
            }
            if ((spin & 1023u) == 1023u) {
                if (t0 == 0) t0 = global_ns();
                if (*mark() != 0 || global_ns() - t0 > (turn == 1 ? limit1 : limit)) return false;
            }
        }
    }

    // grid barrier: what any thread wrote before is visible to every thread after
    __device__ __forceinline__ bool barrier() {
        if (ONE) {
            __syncthreads();
            return true;
        }
        const int par = (int)(turn++ & 1u);
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long q[1] = {1ull};
            unsigned long long d[1];
            const bool ok = sh->rest[kFail] == 0 && arrive_wait<1>(par, q, d);
            if (!ok) abandon();
            sh->state[par] = ok ? 0 : 1;
        }
        __syncthreads();
        return sh->state[par] == 0;
    }

    // v[k] <- sum over the grid, the same bits in every thread; expect[k]: about what the sums
    // will be (any value, the same in every block; it only decides how fast the sum is).  Also
    // a grid barrier.
    template <int NV>
    __device__ __forceinline__ bool sum(float (&v)[NV], const float (&expect)[NV]) {
        static_assert(NV <= 2, "two words per exchange");
        const int par = (int)(turn++ & 1u);
#pragma unroll
        for (int k = 0; k < NV; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < NV; ++k) sh->part[par][k][wid] = v[k];
        __syncthreads();
        const bool alive = ONE || sh->rest[kFail] == 0;   // early: its latency beside the shuffles'
        if (ONE || wid == 0) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                v[k] = lane < warps ? sh->part[par][k][lane] : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
            }
        }
        if (ONE) return true;
        float* parts = reinterpret_cast<float*>(mem + 3 * kGridLine + (size_t)par * nb * 24);
        if (threadIdx.x == 0) {
            unsigned long long q[NV], d[NV] = {};
            int e[NV];
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                e[k] = word_exp(expect[k]);
                q[k] = word_put(v[k], e[k]);
                parts[k * nb + blockIdx.x] = v[k];             // for the sums added one by one
            }
            const bool ok = alive && arrive_wait<NV>(par, q, d);
            bool exact = false;
#pragma unroll
            for (int k = 0; k < NV; ++k) exact = !word_total(d[k], e[k], &sh->tot[par][k]) || exact;
            if (!ok) abandon();
            sh->state[par] = ok ? (exact ? 2 : 0) : 1;
        }
        __syncthreads();
        if (sh->state[par] == 2) {   // the same in every block
            if (wid == 0) {
                float t[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) t[k] = 0.f;
                for (int b = lane; b < nb; b += 32)
#pragma unroll
                    for (int k = 0; k < NV; ++k) t[k] += __ldcg(parts + k * nb + b);
#pragma unroll
                for (int k = 0; k < NV; ++k) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
                    if (lane == 0) sh->tot[par][k] = t[k];
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = sh->tot[par][k];
        return sh->state[par] != 1;
    }

    // v[0..2] summed over the lanes of a warp: the totals in lanes 0, 8 and 16.  The values share the
    // first two steps, six additions instead of fifteen: an FP64 instruction of a warp takes the
    // SM's FP64 pipe 16 cycles, and every warp of a block issues these.
    __device__ __forceinline__ double warp_sum3(const double (&v)[3]) const {
        const bool h = lane & 16, q = lane & 8;
        const double a = (h ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h ? v[0] : v[2], 16);
        const double up = __shfl_xor_sync(0xffffffffu, v[1], 16), b = h ? 0.0 : v[1] + up;
        double t = (q ? b : a) + __shfl_xor_sync(0xffffffffu, q ? a : b, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    }

    // FP64 sums of three values over the grid (once per refinement), added in block order, handed to
    // post(v) in one thread of each block; what it writes to shared memory every thread sees
    // after.  Scalar FP64 work belongs there: a square root or a quotient that every warp
    // computes for itself keeps the FP64 pipe of the SM for microseconds.
    template <class Post>
    __device__ __forceinline__ bool sum64(double (&v)[3], Post post) {
        const double t = warp_sum3(v);
        if ((lane & 7) == 0 && lane < 24) sh->part64[lane >> 3][wid] = t;
        __syncthreads();
        double* parts = reinterpret_cast<double*>(mem + 3 * kGridLine + (size_t)(turn & 1u) * nb * 24);
        if (wid == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k) v[k] = lane < warps ? sh->part64[k][lane] : 0.0;
            const double b = warp_sum3(v);
            if (ONE)
                v[0] = b;
            else if ((lane & 7) == 0 && lane < 24)
                parts[(lane >> 3) * nb + blockIdx.x] = b;
        }
        if (!ONE && !barrier()) return false;
        if (wid == 0) {
            if (!ONE) {
                v[0] = v[1] = v[2] = 0.0;
                for (int b = lane; b < nb; b += 32)
#pragma unroll
                    for (int k = 0; k < 3; ++k) v[k] += __ldcg(parts + k * nb + b);
                v[0] = warp_sum3(v);
            }
            const double all[3] = {v[0], __shfl_sync(0xffffffffu, v[0], 8), __shfl_sync(0xffffffffu, v[0], 16)};
            if (lane == 0) post(all);
        }
        __syncthreads();
        return true;
    }
};

#endif
}  // namespace fempic
