// Host-side decisions of the field solvers with a small C interface.  Test infrastructure: built by
// tests/test_host_solver.py with g++.
#include "../paper_2103_06737_gb300/csrc/field.cuh"
#include "../paper_2103_06737_gb300/csrc/grid_sync.cuh"
#include "../paper_2103_06737_gb300/csrc/pcg.cuh"

using namespace fempic;

extern "C" {

// the status and {rel_res, abs_res, iters, outer} that a solve's output words stand for
int hs_outcome(const double* out, int marked, double tol, double* r) {
    fp_solve_info info{};
    const int st = (int)solve_outcome(out, marked != 0, tol, &info);
    r[0] = info.rel_res, r[1] = info.abs_res, r[2] = info.iters, r[3] = info.outer;
    return st;
}

int hs_met(double rr, double thr) { return solve_met(rr, thr) ? 1 : 0; }

double hs_wait_seconds(int first) { return 1e-9 * (double)(first ? kGridStartNs : kGridWaitNs); }

// the total of n blocks' partials as one grid exchange sums them; 0: the blocks add the floats instead
int hs_word_sum(const float* v, int n, float expect, float* total) {
    const int e = word_exp(expect);
    unsigned long long d = 0;
    for (int k = 0; k < n; ++k) d += word_put(v[k], e);
    return (int)(d & 255ull) == n && word_total(d, e, total);
}

// r: records per slice, their slots, bytes of an FP64 tile of full records with 16- and 32-bit columns
void hs_segments(int wmax, int64_t room, int64_t* r) {
    int nseg = 0, seg = 0;
    stream_segments(wmax, (size_t)room, &nseg, &seg);
    r[0] = nseg, r[1] = seg;
    for (int wide = 0; wide < 2; ++wide)
        r[2 + wide] = tile_bytes(kHeader + kConsumers * rec_bytes((uint32_t)seg, wide != 0, OP_F64));
}

}  // extern "C"
