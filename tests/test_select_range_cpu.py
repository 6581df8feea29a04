"""The ranges that the layer-wide selection narrows its keys down to: the kernel's own arithmetic (csrc/select_range.h, compiled here for
the host) walked through the kernel's passes, on keys up to 2^64 - 1.  Whatever the keys, the walk ends within the stated passes, and the
range it ends at holds the budgeted key."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_00596_b200", "csrc")

# the passes of prune_select_kernel on one thread: what is counted, picked and left
WALK = r"""
#include <vector>
#include "select_range.h"
using namespace npas;
extern "C" int walk(const uint64_t *keys, long long n, uint64_t base, uint64_t top, long long n_keep, unsigned rank_limit,
                    uint64_t *lo_out, uint64_t *hi_out, long long *need_out, long long *have_out)
{
    uint64_t lo = 0, hi = ~0ull;
    long long need = n_keep, have = n;
    int shift = sel_first_shift(base, top), pass = 0;
    for (; need != have && have > (long long)rank_limit && lo != hi; ++pass) {
        if (pass == 64) return -1;
        std::vector<long long> hist(kSelBins, 0);
        if (pass) shift = sel_shift(hi - lo);
        for (long long i = 0; i < n; ++i) {
            const uint64_t k = keys[i];
            if (pass && (k < lo || k > hi)) continue;
            const unsigned b = pass ? sel_bin(k, lo, shift) : sel_first_bin(k, base, shift);
            if (b >= kSelBins) return -2;
            ++hist[b];
        }
        long long above = 0;
        int bin = (int)kSelBins - 1;
        while (bin >= 0 && above + hist[bin] < need) above += hist[bin--];
        if (bin < 0) return -3;
        need -= above; have = hist[bin];
        if (pass) sel_range((unsigned)bin, shift, lo, hi);
        else sel_first_range((unsigned)bin, base, shift, lo, hi);
    }
    *lo_out = lo; *hi_out = hi; *need_out = need; *have_out = have;
    return pass;
}
extern "C" int passes() { return kSelPasses; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("select")
    src, so = d / "walk.cpp", d / "walk.so"
    src.write_text(WALK)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", str(so), str(src)])
    return ctypes.CDLL(str(so))


def _walk(lib, keys, n_keep, base, top, rank_limit):
    keys = np.ascontiguousarray(keys, dtype=np.uint64)
    lo, hi, need, have = ctypes.c_uint64(), ctypes.c_uint64(), ctypes.c_longlong(), ctypes.c_longlong()
    p = lib.walk(keys.ctypes.data_as(ctypes.c_void_p), ctypes.c_longlong(len(keys)), ctypes.c_uint64(int(base)), ctypes.c_uint64(int(top)),
                 ctypes.c_longlong(n_keep), ctypes.c_uint(rank_limit), ctypes.byref(lo), ctypes.byref(hi), ctypes.byref(need), ctypes.byref(have))
    return p, lo.value, hi.value, need.value, have.value


def _keys(kind, rng, n=3000):
    top = 2 ** 64 - 1
    if kind == "numbers":
        return (rng.standard_normal(n) ** 2).view(np.uint64)
    if kind == "numbers and one pattern":                 # what weights of the bits 0xFFFFFFFF leave, beside ordinary ones
        return np.where(rng.random(n) < 0.7, np.uint64(0xFFFFFFFFE0000000), (rng.standard_normal(n) ** 2).view(np.uint64))
    if kind == "top end":                                 # neighbouring keys up to the last one there is
        return np.array([top - int(v) for v in rng.integers(0, 1500, n)], dtype=np.uint64)
    if kind == "top end of wide steps":
        return np.array([top - (int(v) << int(s)) for v, s in zip(rng.integers(0, 700, n), rng.integers(0, 52, n))], dtype=np.uint64)
    if kind == "both ends":
        return np.where(rng.random(n) < 0.5, np.uint64(top) - rng.integers(0, 40, n).astype(np.uint64), rng.integers(0, 40, n).astype(np.uint64))
    if kind == "one value at the end":
        return np.full(n, top, dtype=np.uint64)
    assert kind == "any bits"
    return rng.integers(0, 2 ** 64, n, dtype=np.uint64)


@pytest.mark.parametrize("kind", ["numbers", "numbers and one pattern", "top end", "top end of wide steps", "both ends", "one value at the end", "any bits"])
@pytest.mark.parametrize("rank_limit", [0, 1, 16, 512])
def test_every_selection_ends_at_the_budgeted_key(lib, kind, rank_limit):
    rng = np.random.default_rng(11)
    for trial in range(6):
        keys = _keys(kind, rng)
        order = np.sort(keys)[::-1]
        n = len(keys)
        samples = [(keys[::max(1, n // 256)].min(), keys[::max(1, n // 256)].max()),         # as the kernel samples
                   (keys.min(), keys.max()), (keys[0], keys[0]), (order[n // 2], keys.max())]
        for base, top in samples:
            base, top = min(int(base), int(top)), max(int(base), int(top))
            for n_keep in (1, n // 3, n // 2 + 1, n - 1, n):
                passes, lo, hi, need, have = _walk(lib, keys, n_keep, base, top, rank_limit)
                assert 0 <= passes <= lib.passes(), (trial, base, top, n_keep, passes)
                assert lo <= int(order[n_keep - 1]) <= hi
                assert have == int(((keys >= np.uint64(lo)) & (keys <= np.uint64(hi))).sum()) and need == n_keep - int((keys > np.uint64(hi)).sum())
                assert need == have or have <= rank_limit or lo == hi
