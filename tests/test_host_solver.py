"""Host-side decisions of the field solvers, on the library's own source compiled with g++."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_host_assembly import CSRC, HERE, ROOT, _cuda_include

OK, ECUDA, ENOCONV = 0, 2, 4
INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module")
def hs(tmp_path_factory):
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("hs") / "libhs.so")
    cmd = [cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + inc, "-I" + os.path.join(ROOT, "include"),
           os.path.join(HERE, "host_solver.cpp"), os.path.join(CSRC, "field_build.cpp"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    lib.hs_outcome.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_void_p]
    lib.hs_segments.argtypes = [ctypes.c_int, ctypes.c_int64, ctypes.c_void_p]
    lib.hs_word_sum.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_float, ctypes.c_void_p]
    lib.hs_wait_seconds.restype = ctypes.c_double
    lib.hs_met.argtypes = [ctypes.c_double, ctypes.c_double]
    return lib


# iterations, |r|^2, |reference|^2, refinements -> status at a tolerance of 1e-10
@pytest.mark.parametrize("words,status", [
    ((12, 1e-22, 1.0, 2), OK), ((0, 0.0, 0.0, 0), OK),             # within it; a zero right-hand side
    ((9, 1e-18, 1.0, 2), ENOCONV),                                  # the iteration cap
    ((0, NAN, 1.0, 0), ENOCONV), ((0, NAN, NAN, 0), ENOCONV),       # a NaN in the start, in the right-hand side
    ((0, INF, 1.0, 0), ENOCONV), ((0, INF, INF, 0), ENOCONV),       # a norm that overflows
    ((0, INF, 1.0, -1), ECUDA)])                                    # as a solve writes them when it starts
def test_outcome_of_a_solve(hs, words, status):
    w, r = np.array(words, np.float64), np.zeros(4)
    assert hs.hs_outcome(w.ctypes.data, 0, 1e-10, r.ctypes.data) == status
    assert (r[2], r[3]) == (words[0], max(words[3], 0))
    # the device sets the status word's bit by the same rule
    assert hs.hs_met(w[1], 1e-20 * w[2]) == (status == OK)
    # whatever they say, an exchange was abandoned: a block may have left without its rows
    assert hs.hs_outcome(w.ctypes.data, 1, 1e-10, r.ctypes.data) == ECUDA


def test_first_exchange_waits_for_blocks_that_start_late(hs):
    """A block can start only when a kernel of another stream has left its SM: the wait for all blocks
    to be there is many times the wait for blocks at work, and still bounded."""
    assert 2.0 <= hs.hs_wait_seconds(0) <= 5.0
    assert 10.0 * hs.hs_wait_seconds(0) <= hs.hs_wait_seconds(1) <= 60.0


@pytest.mark.parametrize("blocks", [2, 152, 255])
@pytest.mark.parametrize("kind", ["alike", "one_large", "signs"])
def test_exchange_sums_are_as_fine_as_float_sums(hs, blocks, kind):
    """The total that an exchange takes from its integer word is within 2^-23 of the exact one: half a
    unit per block, at most 2^-24 of it, and its own rounding to a float.  Totals near their
    expectation, and up to 16 times above or below, come from the word."""
    rng = np.random.default_rng(blocks)
    for log_ratio in range(-40, 16):
        expect = np.float32(rng.uniform(1e-6, 1e-3))
        total = float(expect) * 2.0 ** log_ratio
        unit = 2.0 ** (np.frexp(expect)[1] - 1 - 36)      # of the word: the expectation's power of two is 2^36
        if kind == "one_large":     # all the others rounded the same way, by nearly half a unit
            v = np.full(blocks, 0.49 * unit)
            v[0] = total
        else:
            v = rng.uniform(0.5, 1.5, blocks) * total / blocks
            if kind == "signs":
                v[1::2] *= -0.5
        v = v.astype(np.float32)
        got = np.zeros(1, np.float32)
        used = hs.hs_word_sum(v.ctypes.data, blocks, expect, got.ctypes.data)
        exact = float(v.astype(np.float64).sum())
        if used:
            assert abs(float(got[0]) - exact) <= 2.0 ** -23 * abs(exact), (log_ratio, got[0], exact)
        assert used or abs(log_ratio) > 4 or (kind, blocks) != ("alike", 152)


def test_exchange_sums_that_do_not_fit_are_left_to_the_floats(hs):
    got = np.zeros(1, np.float32)
    for bad in (NAN, INF, -INF, 1e30):
        v = np.array([1.0, bad, 1.0], np.float32)
        assert not hs.hs_word_sum(v.ctypes.data, 3, 1.0, got.ctypes.data)
    for expect in (0.0, NAN, INF, -1.0, 1e-42):           # no expectation: units of one
        v = np.full(3, 0.25, np.float32)
        assert not hs.hs_word_sum(v.ctypes.data, 3, expect, got.ctypes.data)


def test_records_of_wide_rows_fit_twice(hs):
    """However wide the rows, two FP64 tiles fit in the shared memory of an SM (227 KB less the kernel's
    own 1,792 bytes), so that copies run beside products; rows of up to 20 slots (19 in the cube
    meshes' edge systems) are one record; the records of a row are alike."""
    room = 232448 - 1792
    r = np.zeros(4, np.int64)
    for wmax in [1, 2, 15, 18, 19, 20, 21, 22, 37, 38, 39, 57, 58, 64, 100, 1000, 1501, 30000]:
        hs.hs_segments(wmax, room, r.ctypes.data)
        nseg, seg, narrow, wide = (int(x) for x in r)
        assert nseg * seg >= wmax > (nseg - 1) * seg
        assert 2 * narrow <= room and 2 * wide <= room, wmax
        assert nseg * seg - wmax < nseg
        assert (nseg == 1) == (wmax <= 20)
