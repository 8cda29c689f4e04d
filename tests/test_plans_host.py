"""Host decisions of csrc/plan.h, compiled by themselves: the row-per-lane
layout, the products that read it, the ways of a solve and the SMs of a sweep's
systems."""

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "plan.h"
using namespace hz;
extern "C" int slices(const int *rp, int n, int *base, unsigned *longs, long long *slots) {
    const SlicePlan p = slice_plan(rp, n, rp[n]);
    std::copy(p.base.begin(), p.base.end(), base);
    std::copy(p.longs.begin(), p.longs.end(), longs);
    *slots = p.slots;
    return p.fits;
}
extern "C" int product(int nsl, int width, int binary64, int sms) { return slice_product(nsl, width, binary64, sms); }
extern "C" int sweep(int ns, const int *nsl, int sms, int max_cta, int max_slices, int *ncta) {
    std::vector<int> c;
    const bool ok = sweep_plan(std::vector<int>(nsl, nsl + ns), sms, max_cta, max_slices, &c);
    std::copy(c.begin(), c.end(), ncta);
    return ok;
}
extern "C" int ways(int *way, const int *answers, int *tried, int *n) {
    Way w = (Way)*way;
    *n = 0;
    const bool ok = first_way(w, [&](Way v) {
        tried[*n] = (int)v;
        return (Launch)answers[(*n)++];
    });
    *way = (int)w;
    return ok;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, lib = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2112_06465_gb300", "csrc"), src, "-o", lib], check=True)
    return C.CDLL(lib)


def pointers(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


def slices(plan, lens):
    rp, n = pointers(lens), len(lens)
    ns = (n + 31) // 32
    base, longs, slots = np.zeros(ns + 1, np.int32), np.zeros(ns, np.uint32), C.c_longlong()
    fits = plan.slices(rp.ctypes.data_as(C.c_void_p), n, base.ctypes.data_as(C.c_void_p),
                       longs.ctypes.data_as(C.c_void_p), C.byref(slots))
    return bool(fits), base, longs, slots.value


@pytest.mark.parametrize("n", [1, 31, 32, 33, 95, 4099])
@pytest.mark.parametrize("lo,hi,far", [(7, 7, 0), (0, 9, 0), (9, 17, 0), (5, 9, 100), (64, 64, 0), (65, 65, 0)])
def test_slice_widths_and_long_rows(plan, n, lo, hi, far):
    """Widths, long rows and slots against their definition, row by row."""
    rng = np.random.default_rng(n + hi)
    lens = rng.integers(lo, hi + 1, n)
    if far:
        lens[rng.integers(0, n, 1 + n // 100)] = far
    if lens.sum() == 0:
        lens[0] = 1
    fits, base, longs, slots = slices(plan, lens)
    lim = max(32.0, 2.0 * lens.sum() / n)
    pad = np.zeros((len(longs), 32), int)
    pad.reshape(-1)[:n] = lens
    isl = pad > lim
    assert np.array_equal((isl * (1 << np.arange(32, dtype=np.uint64))).sum(1), longs)
    width = np.where(isl, 0, pad).max(1)
    assert np.array_equal(np.concatenate([[0], np.cumsum(width)]), base) and slots == 32 * width.sum()
    if width.max() > 64 or slots * 5 > 7 * (lens.sum() - pad[isl].sum()):
        assert not fits


@pytest.mark.parametrize("count,length,fits", [
    (1, 33, True), (1, 512, True), (1, 513, False), (2, 256, True), (2, 257, False), (1, 257, True),
    (3, 33, False), (8, 400, False), (32, 100, False)])
def test_long_rows_that_lie_together(plan, count, length, fits):
    """A warp sums its slice's long rows one after the other: at most two
    passes of 256 entries over them, wherever the slice lies."""
    for n in (8000, 600000):
        for first in (0, 64, n - count):
            lens = np.full(n, 7)
            lens[first:first + count] = length
            assert slices(plan, lens)[0] == fits
        lens = np.full(n, 7)
        lens[:128 * count:128] = 100   # one in a slice, any number of slices
        assert slices(plan, lens)[0]
    lens = np.full(8000, 7)
    lens[:64 * 63:64] = 100            # more than one row in 128
    assert not slices(plan, lens)[0]


def test_products_of_few_wide_slices(plan):
    """Edges of the rule on 152 SMs: which products by themselves read the slices."""
    f = lambda nsl, width, b64: bool(plan.product(nsl, width, b64, 152))
    assert all(f(nsl, w, 1) for nsl in (1, 100, 100000) for w in (1, 15, 39))
    assert [f(nsl, 40, 1) for nsl in (1, 228, 229, 380, 381)] == [False, False, True, True, True]
    assert [f(nsl, 53, 1) for nsl in (1, 228, 229, 380, 381)] == [False, False, False, False, True]
    assert [f(nsl, 40, 0) for nsl in (1, 760)] == [True, True]
    assert [f(nsl, 41, 0) for nsl in (1, 760, 761)] == [False, False, True]


def shares(plan, nsl, sms=152, max_cta=160, max_slices=60):
    a, out = np.array(nsl, np.int32), np.zeros(len(nsl), np.int32)
    ok = plan.sweep(len(nsl), a.ctypes.data_as(C.c_void_p), sms, max_cta, max_slices, out.ctypes.data_as(C.c_void_p))
    return bool(ok), [int(c) for c in out]


@pytest.mark.parametrize("nsl,fits", [
    ([2000] + [32] * 100, True), ([1500] + [10] * 60, True), ([2, 626, 1, 22], True), ([626, 1, 153, 22, 10], True),
    ([32] * 152, True), ([32] * 153, False), ([626] + [1] * 150, False), ([153] + [1] * 140, True),
    ([9121], False), ([9120], True), ([0, 5, 0, 9], True), ([7628] + [61] * 12, True), ([0, 0], True), ([1], True)])
def test_sweep_shares(plan, nsl, fits):
    """A sweep runs on chip exactly where one CTA for each system and enough
    for the large ones fit on the SMs together; then no SM stays idle that a
    system could use, and no CTA holds more than its slices."""
    ok, c = shares(plan, nsl)
    assert ok == fits == (sum(-(-n // 60) for n in nsl) <= 152)
    if not ok:
        return
    assert sum(c) <= 152 and all((n > 0) == (k > 0) and k <= n for n, k in zip(nsl, c))
    assert sum(c) == 152 or all(k == n for n, k in zip(nsl, c))
    assert all(-(-n // k) <= 60 for n, k in zip(nsl, c) if k)


def test_sweep_shares_of_even_systems(plan):
    assert shares(plan, [100, 100, 100, 100]) == (True, [38, 38, 38, 38])
    assert shares(plan, [432, 432, 106, 106], sms=100) == (True, [40, 40, 10, 10])


@pytest.mark.parametrize("start,answers,way,tried,ok", [
    (0, [0], 0, [0], 1), (0, [1, 0], 1, [0, 1], 1), (0, [1, 1], 2, [0, 1], 1), (1, [0], 1, [1], 1),
    (1, [1], 2, [1], 1), (0, [2], 0, [0], 0), (0, [1, 2], 1, [0, 1], 0), (2, [], 2, [], 1)])
def test_ways_of_a_solve(plan, start, answers, way, tried, ok):
    """Launches that the device answers with done (0), no room (1) or another
    error (2): a refused cluster goes to every SM, that to the graph, and an
    error to the caller."""
    a, t, n, w = (C.c_int * 4)(*answers), (C.c_int * 4)(), C.c_int(), C.c_int(start)
    assert plan.ways(C.byref(w), a, t, C.byref(n)) == ok
    assert w.value == way and list(t[:n.value]) == tried
