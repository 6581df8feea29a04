"""Host-only checks of the kernel choice: the committed (case, path) table and the plan cache."""
import ctypes
import os
import random
import subprocess

import pytest

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import binding as B
from dispatch_table import (CONV_AUTO, CONV_CASES, CONV_TAKES, LINEAR_AUTO, LINEAR_CASES, LINEAR_TAKES, UNSUPPORTED)


def _conv_query(kw, path, variant=0):
    R, S = kw.get("R", 3), kw.get("S", 3)
    keep = kw["keep"]
    max_taps = R * S if callable(keep) else min(keep, R * S)
    blob = B.BpBlob(None, B.BpDesc(kw["K"], kw["C"], R, S, kw["Mb"], kw["Nb"], B.BF16, B.BF16, max_taps))
    return npas.conv2d_bp_kernel((kw["N"], kw["H"], kw["W"], kw["C"]), blob, stride=kw.get("stride", 1),
                                 pad=kw.get("pad", 1), relu=True, bias=True, residual=True, path=path, variant=variant)


def _linear_query(kw, path, residual=False, variant=0):
    kc = kw["keep_cols"]
    blob = B.BbBlob(None, B.BbDesc(kw["O"], kw["I"], kw["Bo"], kw["Bi"], B.BF16, B.BF16, kw["Bi"] if callable(kc) else kc))
    return npas.linear_bb_kernel(kw["M"], blob, relu=True, bias=True, residual=residual, path=path, variant=variant)


@pytest.mark.parametrize("path", sorted(CONV_TAKES))
def test_conv_forced_paths_take_exactly_the_listed_cases(path):
    for i, kw in enumerate(CONV_CASES):
        if i in CONV_TAKES[path]:
            assert _conv_query(kw, path) == path, (i, path)
        else:
            with pytest.raises(npas.NpasError) as e:
                _conv_query(kw, path)
            assert e.value.code == UNSUPPORTED, (i, path)


def test_conv_automatic_choice():
    for i, kw in enumerate(CONV_CASES):
        assert _conv_query(kw, 0) == CONV_AUTO[i], i
        assert _conv_query(kw, 2) == CONV_AUTO[i], i          # every case has a tensor-core kernel


@pytest.mark.parametrize("path", sorted(LINEAR_TAKES))
def test_linear_forced_paths_take_exactly_the_listed_cases(path):
    for i, kw in enumerate(LINEAR_CASES):
        for residual in (False, True):
            if i in LINEAR_TAKES[path]:
                assert _linear_query(kw, path, residual) == path, (i, path)
            else:
                with pytest.raises(npas.NpasError) as e:
                    _linear_query(kw, path, residual)
                assert e.value.code == UNSUPPORTED, (i, path)


def test_linear_automatic_choice():
    for i, kw in enumerate(LINEAR_CASES):
        assert _linear_query(kw, 0) == LINEAR_AUTO[i], i


@pytest.mark.parametrize("O,Bo,takes", [(1000, 40, [16, 32, 48, 64, 80, 128, 144, 192, 240, 256]), (1024, 64, [16, 32, 64, 128, 192, 256]),
                                        (1008, 48, [16]), (8, 8, [16, 128])])
def test_linear_column_tile_is_whole_chunks_for_every_output_width(O, Bo, takes):
    """`variant` of path 5: what the header promises for each width O and nothing else (a tile of 40 columns left 8 of 40 unwritten)."""
    kw = dict(M=512, I=512, O=O, Bo=Bo, Bi=64, keep_cols=32)
    for v in (1, 8, 15, 17, 20, 24, 40, 72, 100, 200, 250, 257, 264, 512, *takes):
        if v in takes:
            assert _linear_query(kw, 5, variant=v) == 5, v
        else:
            for path in (5, 6):
                with pytest.raises(npas.NpasError) as e:
                    _linear_query(kw, path, variant=v)
                assert e.value.code == UNSUPPORTED, v
            assert _linear_query(kw, 0, variant=v) not in (5, 6), v


def test_sweep_shape_choices():
    """64x28x28x512 -> 512: kept pairs only where measured faster (up to 3 of 9 taps at 16x16 blocks, up to 4
    of 9 at 32x32), the CTA-pair dense-image kernel elsewhere, also for the block sizes below 16."""
    def q(Mb, Nb, taps):
        return _conv_query(dict(N=64, H=28, W=28, C=512, K=512, Mb=Mb, Nb=Nb, keep=taps), 0)
    assert [q(16, 16, t) for t in (1, 2, 3, 4, 5, 9)] == [8, 8, 8, 7, 7, 7]
    assert [q(32, 32, t) for t in (1, 2, 3, 4, 5, 9)] == [8, 8, 8, 8, 7, 7]
    assert [q(8, 8, t) for t in (1, 9)] == [7, 7] and [q(4, 4, t) for t in (1, 9)] == [7, 7]
    # the tile-shape variant of the pair kernel: only combinations the geometry allows
    kw = dict(N=64, H=28, W=28, C=512, K=512, Mb=16, Nb=16, keep=3)
    for nt, mt in ((128, 1), (128, 2), (256, 1), (256, 2)):
        assert _conv_query(kw, 7, nt | (mt << 16)) == 7
    with pytest.raises(npas.NpasError):
        _conv_query(kw, 7, 64 | (1 << 16))


def _pair_plan(N, H, W, C, K, R, stride, pad, Nb, variant):
    d = B.ConvDesc(N, H, W, C, K, R, R, stride, pad, B.BF16, B.BF16, 1, 1, 0, 7, variant)
    shape = (ctypes.c_int32 * 8)()
    s = npas.load().npas_internal_conv_d2_plan(ctypes.byref(d), ctypes.byref(B.BpDesc(K, C, R, R, 16, Nb, B.BF16, B.BF16, 0)), shape)
    assert s in (0, UNSUPPORTED)
    return list(shape) if s == 0 else None


@pytest.mark.parametrize("wide", [0, 1 << 24])
def test_plan_of_the_pair_kernel_is_that_of_its_shape_alone(wide):
    """The item shape the planner picks among all is planned as when it is the only one allowed: no candidate leaves anything behind for
    the ones after it (slabs of two tiles had left their rows and strides to shapes of one tile)."""
    rng = random.Random(17)
    layers = [(30, 11, 43, 16, 368, 1, 1, 0)]
    while len(layers) < 4000:
        R = rng.choice([1, 1, 3, 3, 4])
        layers.append((rng.randint(1, 64), rng.randint(3, 64), rng.randint(3, 100), 16 * rng.randint(1, 32), 16 * rng.randint(1, 32), R, rng.choice([1, 1, 2]),
                       rng.randint(0, R // 2)))
    planned = 0
    for lay in layers:
        free = _pair_plan(*lay, 8, wide)
        if free is not None:
            planned += 1
            assert free == _pair_plan(*lay, 8, wide | free[0] | (free[1] << 16)), lay
    assert planned > (1500 if wide else 60)


def test_tiles_of_filters_ask_for_nothing_past_the_last_and_store_every_filter_once(tmp_path):
    """The last tiles of the wide pair kernel (two halves of whole filter groups) and of the split kernel, through the arithmetic that both
    kernels use (csrc/tail_start.h, compiled here for the host): weights past the last filter are not asked for, which a tensor copy
    would touch unmapped memory for, and what tiles share is stored by one of them."""
    csrc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_00596_b200", "csrc")
    src, so = tmp_path / "tail.cpp", tmp_path / "tail.so"
    src.write_text('#include "tail_start.h"\nextern "C" int start_of(int s, int w, int t) { return npas::tail_start(s, w, t); }\n')
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-fPIC", "-shared", "-I", csrc, "-o", str(so), str(src)])
    start_of = ctypes.CDLL(str(so)).start_of
    for K in range(16, 529, 16):
        GI = 128
        while K % GI:
            GI //= 2
        for NT in range(32, 257, 32):                              # the wide form's items
            if GI >= 128 or NT % (2 * GI) or NT >= K + 2 * GI:
                continue
            GG, groups, stored = NT // 2 // GI, K // GI, []
            for g0 in range(0, -(-K // NT) * 2 * GG, GG):
                at = start_of(g0, GG, groups)
                assert 0 <= at and at + GG <= groups, (K, NT, g0)
                early = (g0 - at) * GI
                stored += [g0 * GI + c - early for c in range(GG * GI) if c >= early]
            assert stored == list(range(K)), (K, NT)
        for NT in range(16, min(K, 128) + 1, 16):                  # the split form's tiles
            if (GI % NT if NT < GI else NT % GI):
                continue
            stored = []
            for k in range(0, K, NT):
                at = start_of(k, NT, K)
                assert 0 <= at and at + NT <= K and at % min(GI, NT) == 0, (K, NT, k)
                stored += range(k, at + NT)
            assert stored == list(range(K)), (K, NT)


def test_plan_cache_round_trip_and_rejects_garbage():
    c = npas.PlanCache()
    blob = B.BpBlob(None, B.BpDesc(512, 512, 3, 3, 16, 16, B.BF16, B.BF16, 3))
    k1 = c.conv_key((64, 28, 28, 512), blob, 1, 1, False, False, False)
    lb = B.BbBlob(None, B.BbDesc(2048, 512, 64, 64, B.BF16, B.BF16, 16))
    k2 = c.linear_key(3136, lb, True, True, False)
    assert k1 != c.conv_key((64, 28, 28, 512), B.BpBlob(None, B.BpDesc(512, 512, 3, 3, 16, 16, B.BF16, B.BF16, 1)), 1, 1,
                            False, False, False)                       # the mask statistic is part of the key
    c.put(k1, 7, 256 | (1 << 16), 155.25)
    c.put(k2, 6, 128, 11.5)
    c.put(c.two_key(k2, k2), 2, 0, 20.0)
    text = c.to_json()
    d = npas.PlanCache.from_json(text)
    assert d.get(k1) == (7, 256 | (1 << 16)) and d.get(k2) == (6, 128) and d.get("conv:other") is None and d.get(d.two_key(k2, k2)) == (2, 0)
    assert d.to_json() == text
    for bad in ('{"version": 2, "plans": {}}', '{"plans": []}', '{"version": 1, "plans": {"k": [1, 2]}}'):
        with pytest.raises(ValueError):
            npas.PlanCache.from_json(bad)
