"""The sweep planner (host logic, no GPU): every element of every tensor is covered by exactly one work item,
whatever the shapes, ranks, storage types and alignment, for the single-seed and the multi-seed plan, with and
without the tcgen05 path.  Checked by brute-force counting on small random models and by interval arithmetic on
the full-size configurations."""
import ctypes

import numpy as np
import pytest

from paper_2601_12917_b200 import synth, zgr


class PlanItem(ctypes.Structure):
    _fields_ = [("path", ctypes.c_int32), ("kpad", ctypes.c_int32), ("tensor", ctypes.c_int32), ("ncols", ctypes.c_int32),
                ("row0_or_e0", ctypes.c_int64), ("nrows_or_count", ctypes.c_int64), ("col0", ctypes.c_int64)]


def plan(shapes, ranks, dtypes, bits=16, sm_count=148, tcgen05=1, multi=0, alpha=0.5, misalign=()):
    L = zgr.lib()
    L.zgr_debug_plan.restype = ctypes.c_int
    n = len(shapes)
    arr = (zgr.ZgrTensor * n)()
    for l, ((m, c), r, dt) in enumerate(zip(shapes, ranks, dtypes)):
        base = 0x100000 * (l + 1) + (2 if l in misalign and dt != zgr.F32 else (4 if l in misalign else 0))
        arr[l] = zgr.ZgrTensor(base, m, c, dt, r, 0x40000000 if r else None)     # addresses are never dereferenced
    cfg = zgr.ZgrConfig(alpha, 1e-3, zgr.SCALE_UNIT, bits)
    count = ctypes.c_int64()
    rc = L.zgr_debug_plan(arr, n, ctypes.byref(cfg), sm_count, tcgen05, multi, None, ctypes.c_int64(0), ctypes.byref(count))
    assert rc == zgr.OK
    items = (PlanItem * count.value)()
    rc = L.zgr_debug_plan(arr, n, ctypes.byref(cfg), sm_count, tcgen05, multi, items, ctypes.c_int64(count.value), ctypes.byref(count))
    assert rc == zgr.OK and count.value == len(items)
    return list(items)


def kernels(shapes, ranks, dtypes, bits=16, sm_count=148, multi=0, misalign=()):
    """Name of the kernel that serves each tensor (zgr_debug_plan_kernels)."""
    n = len(shapes)
    arr = (zgr.ZgrTensor * n)()
    for l, ((m, c), r, dt) in enumerate(zip(shapes, ranks, dtypes)):
        arr[l] = zgr.ZgrTensor(0x100000 * (l + 1) + (4 if l in misalign else 0), m, c, dt, r, 0x40000000 if r else None)
    cfg = zgr.ZgrConfig(0.5, 1e-3, zgr.SCALE_UNIT, bits)
    out = (ctypes.c_int32 * n)()
    assert zgr.lib().zgr_debug_plan_kernels(arr, n, ctypes.byref(cfg), ctypes.c_int32(sm_count), ctypes.c_int32(1), ctypes.c_int32(multi), out) == zgr.OK
    return [zgr.KERNEL_NAMES[k] for k in out]


def check_exact_cover(items, shapes):
    per_tensor = {}
    for it in items:
        per_tensor.setdefault(it.tensor, []).append(it)
    assert sorted(per_tensor) == list(range(len(shapes)))          # every tensor is served
    for l, (m, c) in enumerate(shapes):
        its = per_tensor[l]
        paths = {it.path for it in its}
        assert len(paths) == 1, f"tensor {l} is split over kernel families {paths}"
        if paths == {0}:                                           # flat chunks of elements
            iv = sorted((it.row0_or_e0, it.nrows_or_count) for it in its)
            pos = 0
            for e0, cnt in iv:
                assert e0 == pos and cnt > 0 and e0 % 8 == 0
                pos += cnt
            assert pos == m * c
        else:                                                      # strips of columns x ranges of rows
            strips = {}
            for it in its:
                strips.setdefault((it.col0, it.ncols), []).append((it.row0_or_e0, it.nrows_or_count))
            pos = 0
            for (c0, nc) in sorted(strips):
                assert c0 == pos and nc > 0
                pos += nc
                r = 0
                for r0, nr in sorted(strips[(c0, nc)]):
                    assert r0 == r and nr > 0
                    r += nr
                assert r == m
            assert pos == c


def brute_force_counts(items, shapes):
    counts = [np.zeros(m * c, dtype=np.int32) for m, c in shapes]
    for it in items:
        m, c = shapes[it.tensor]
        if it.path == 0:
            counts[it.tensor][it.row0_or_e0: it.row0_or_e0 + it.nrows_or_count] += 1
        else:
            view = counts[it.tensor].reshape(m, c)
            view[it.row0_or_e0: it.row0_or_e0 + it.nrows_or_count, it.col0: it.col0 + it.ncols] += 1
    return counts


@pytest.mark.parametrize("multi", [0, 1])
@pytest.mark.parametrize("tcgen05", [0, 1])
@pytest.mark.parametrize("trial", range(6))
def test_random_models_are_covered_exactly_once(trial, tcgen05, multi):
    rng = np.random.default_rng(100 + trial)
    n = int(rng.integers(3, 9))
    shapes, ranks, dtypes = [], [], []
    for _ in range(n):
        if rng.random() < 0.3:
            shapes.append((1, int(rng.integers(1, 5000)))); ranks.append(0)
        else:
            m = int(rng.integers(1, 700))
            c = int(rng.integers(1, 160)) * (8 if rng.random() < 0.7 else 1)
            shapes.append((m, c)); ranks.append(int(rng.choice([0, 1, 3, 4, 8, 12, 16, 20, 32, 40, 64])))
        dtypes.append(int(rng.choice([zgr.F32, zgr.F16, zgr.BF16])))
    misalign = {int(rng.integers(0, n))} if rng.random() < 0.5 else set()
    items = plan(shapes, ranks, dtypes, bits=int(rng.choice([16, 32])), sm_count=int(rng.choice([1, 4, 148])), tcgen05=tcgen05, multi=multi,
                 misalign=misalign)
    check_exact_cover(items, shapes)
    for cnt in brute_force_counts(items, shapes):
        assert cnt.min() == 1 and cnt.max() == 1
    if multi:
        assert all(it.path != 2 for it in items)                   # the legacy tensor-core kernel serves one seed per sweep only
    if not tcgen05:
        assert all(it.path != 4 for it in items)


@pytest.mark.parametrize("name", ["tiny", "roberta_large", "opt_1p3b", "llama_7b", "llama_13b"])
def test_full_size_configurations(name):
    wl = synth.workload(name)
    shapes = [(t.rows, t.cols) for t in wl.tensors]
    ranks = [t.rank for t in wl.tensors]
    dt = {"f32": zgr.F32, "f16": zgr.F16, "bf16": zgr.BF16}[wl.dtype]
    items = plan(shapes, ranks, [dt] * len(shapes))
    check_exact_cover(items, shapes)
    covered = sum(it.nrows_or_count if it.path == 0 else it.nrows_or_count * it.ncols for it in items)
    assert covered == wl.params
    expected_path = {"f32": 1, "f16": 4, "bf16": 4}[wl.dtype]
    assert {it.path for it in items if ranks[it.tensor] > 0} == {expected_path}
    assert {it.path for it in items if ranks[it.tensor] == 0} == {0}
    # enough items to balance 148 persistent CTAs: the tail of a fixed round-robin stays below 3 % (the tcgen05 kernel
    # assigns its items that way; the CUDA-core contraction kernel hands them out by a counter and needs less)
    guided = [it for it in items if it.path != 0]
    per_cta = np.zeros(148)
    for i, it in enumerate(guided):
        per_cta[i % 148] += it.nrows_or_count * it.ncols
    if name != "tiny":
        assert per_cta.max() / per_cta.mean() < 1.03


# The tile kernel's large sets, whose item heights come from a replay of the hand-out: ragged rows in 16 bits, fp32 above rank 8, and
# rank 8 on either side of the sizes between which fp32 sets take it; shares of small sets beside them.
@pytest.mark.parametrize("sm_count", [148, 132, 1])
@pytest.mark.parametrize("shapes,ranks,dtype,path", [
    ([(1234, 4937), (4937, 1234), (1, 1234)] * 12, [16, 16, 0] * 12, zgr.BF16, 3), ([(6000, 5001)], [33], zgr.F16, 3),
    ([(4096, 1024), (1024, 4096), (50265, 1024)] * 3, [32] * 9, zgr.F32, 3), ([(2000, 5128)] * 3, [64, 24, 9], zgr.F32, 3),
    ([(1024, 2040)], [8], zgr.F32, 1), ([(1024, 2056)], [8], zgr.F32, 1), ([(8192, 4096)] * 3, [8] * 3, zgr.F32, 1), ([(8192, 8192)] * 4, [8] * 4, zgr.F32, 1),
    ([(300, 2051)] * 7, [16] * 7, zgr.BF16, 3)])
def test_large_sets_of_the_tile_kernel(shapes, ranks, dtype, path, sm_count):
    for multi in (0, 1):
        items = plan(shapes, ranks, [dtype] * len(shapes), sm_count=sm_count, multi=multi)
        check_exact_cover(items, shapes)
        assert {it.path for it in items if ranks[it.tensor] > 0} == {path}


# Both kernels with three-part operands carry the path of what they stand in for; what tells them apart.
@pytest.mark.parametrize("shapes,ranks,dtype,misalign,expected", [
    ([(1300, 2051), (40, 15), (1, 9)], [16, 8, 0], zgr.BF16, (), ["staged", "tile", "iso"]), ([(300, 2051)], [16], zgr.F16, (), ["tile"]),
    ([(1300, 2051), (500, 2051)], [16, 16], zgr.F16, (1,), ["staged", "tile"]), ([(4000, 5001), (2000, 5128)], [24, 24], zgr.F32, (), ["tile", "staged"]),
    ([(1300, 2056)], [8], zgr.BF16, (), ["staged"]), ([(500, 2056)], [8], zgr.BF16, (), ["fma"]), ([(1300, 2056)], [9], zgr.BF16, (), ["umma"]),
    ([(8192, 10240)], [4], zgr.F32, (), ["fma"])])
def test_kernel_of_each_tensor(shapes, ranks, dtype, misalign, expected):
    assert kernels(shapes, ranks, [dtype] * len(shapes), misalign=misalign) == expected
    assert zgr.lib().zgr_debug_plan_kernels(None, 0, None, ctypes.c_int32(148), ctypes.c_int32(1), ctypes.c_int32(0), None) == zgr.EINVAL


# The lines between the two, which depend on the whole set: small fp32 sets, tiles that are not full, short items from the counter, ragged
# rows whose spans of 256 cost too many tiles.
@pytest.mark.parametrize("d,layers,rank,dtype,expected", [
    (512, 2, 16, zgr.F32, "tile"), (768, 1, 16, zgr.F32, "staged"), (512, 1, 20, zgr.F32, "staged"), (192, 40, 16, zgr.F32, "tile"), (192, 40, 64, zgr.F32, "staged"),
    (320, 20, 4, zgr.F32, "staged"), (136, 40, 8, zgr.BF16, "tile"), (192, 40, 8, zgr.F16, "tile"), (320, 10, 8, zgr.BF16, "staged"), (320, 40, 8, zgr.BF16, "tile"), (256, 40, 8, zgr.BF16, "tile"),
    (256, 10, 8, zgr.BF16, "staged"), (384, 20, 8, zgr.BF16, "staged"), (125, 40, 16, zgr.BF16, "tile"), (261, 20, 16, zgr.BF16, "staged"), (141, 40, 16, zgr.F16, "staged")])
def test_lines_between_staged_and_tile_kernel(d, layers, rank, dtype, expected):
    shapes = [(d, d), (4 * d, d), (d, d), (d, 4 * d), (d, d), (d, d)] * layers
    assert set(kernels(shapes, [rank] * len(shapes), [dtype] * len(shapes))) == {expected}


def test_short_strips_that_are_not_full():
    for cols, expected in ((1424, "tile"), (1408, "staged")):
        assert set(kernels([(337, cols)] * 40, [4] * 40, [zgr.F32] * 40)) == {expected}


# Ragged sets whose spans cost a tile of the busiest SM: many seeds have the tile kernel, one the staged one.
@pytest.mark.parametrize("shapes,multi_kernel", [([(6917, 131)] * 4, "tile"), ([(1234, 1234)] * 4 + [(4937, 1234), (1234, 4937)], "tile"),
                                                  ([(1534, 1534)] * 4 + [(6137, 1534), (1534, 6137)], "staged")])
def test_kernel_of_many_seeds(shapes, multi_kernel):
    n = len(shapes)
    assert set(kernels(shapes, [16] * n, [zgr.BF16] * n)) == {"staged"}
    assert set(kernels(shapes, [16] * n, [zgr.BF16] * n, multi=1)) == {multi_kernel}
    check_exact_cover(plan(shapes, [16] * n, [zgr.BF16] * n, multi=1), shapes)


# Ragged sets between 12 and 24 tiles per SM: from the counter with one seed, in shares with many, unless their strips are short.
@pytest.mark.parametrize("d,ffn,layers,shares", [(1411, 5643, 2, True), (999, 3999, 3, True), (441, 1765, 12, False), (2051, 8203, 2, False)])
def test_shares_of_many_seeds(d, ffn, layers, shares):
    shapes = ([(d, d)] * 4 + [(ffn, d), (d, ffn)]) * layers
    one, many = (plan(shapes, [16] * len(shapes), [zgr.BF16] * len(shapes), multi=m) for m in (0, 1))
    check_exact_cover(many, shapes)
    assert ([(it.tensor, it.row0_or_e0, it.col0) for it in one] != [(it.tensor, it.row0_or_e0, it.col0) for it in many]) == shares
    tiles = sum(-(-m // 256) * 2 * -(-n // 128) for m, n in shapes)
    if shares:
        assert max(-(-it.nrows_or_count // 128) for it in many) <= -(-tiles // 148) and len(many) < len(one)


# Ragged 16-bit sets that are dealt out in shares: a share begins and ends in the middle of a span of 256 rows where that makes the
# largest one smaller, down to one tile above the mean (which is a whole number of tiles).  Tiles of 128 rows, two to a span.
@pytest.mark.parametrize("d,ffn,rank", [(1234, 4937, 16), (871, 3491, 32), (701, 2803, 64), (1534, 6137, 16), (501, 2003, 8)])
def test_shares_of_ragged_sets_are_even(d, ffn, rank):
    shapes = [(d, d)] * 4 + [(ffn, d), (d, ffn)]
    tiles = sum(-(-m // 256) * 2 * -(-n // 128) for m, n in shapes)
    assert tiles < 12 * 148 and sum(m * n for m, n in shapes) > 5 << 19
    for multi in (0, 1):
        items = plan(shapes, [rank] * 6, [zgr.BF16] * 6, multi=multi)
        check_exact_cover(items, shapes)
        assert max(-(-it.nrows_or_count // 128) for it in items) <= -(-tiles // 148)


# Last spans of every kind: one to eight rows (residues 4-7 without rows up to four), and around a block and a span.
HALVES = [(256 * (i % 3) + r, 263 + 16 * i) for i, r in enumerate([1, 3, 4, 5, 7, 8, 9, 127, 128, 132, 133, 252, 255, 256])] + [(2500, 1029)]


@pytest.mark.parametrize("sm_count", [148, 100])
def test_halves_of_last_spans_are_covered(sm_count):
    items = plan(HALVES, [min(16, m) for m, _ in HALVES], [zgr.F16] * len(HALVES), sm_count=sm_count)
    check_exact_cover(items, HALVES)
    for cnt in brute_force_counts(items, HALVES):
        assert cnt.min() == 1 and cnt.max() == 1
    assert any(it.row0_or_e0 % 256 for it in items)


def test_alpha_one_plans_everything_as_isotropic_and_errors_are_reported():
    items = plan([(64, 256), (1, 100)], [8, 0], [zgr.BF16, zgr.BF16], alpha=1.0)
    assert {it.path for it in items} == {0}
    L = zgr.lib()
    cnt = ctypes.c_int64()
    cfg = zgr.ZgrConfig(0.5, 1e-3, zgr.SCALE_UNIT, 16)
    arr = (zgr.ZgrTensor * 1)(zgr.ZgrTensor(0x1000, 4, 4, zgr.F32, 0, None))
    assert L.zgr_debug_plan(arr, 1, ctypes.byref(cfg), 0, 1, 0, None, ctypes.c_int64(0), ctypes.byref(cnt)) == zgr.EINVAL   # sm_count
    assert L.zgr_debug_plan(arr, 1, ctypes.byref(cfg), 148, 1, 0, None, ctypes.c_int64(0), None) == zgr.EINVAL
    bad = (zgr.ZgrTensor * 1)(zgr.ZgrTensor(0x1000, 4, 4, 7, 0, None))
    assert L.zgr_debug_plan(bad, 1, ctypes.byref(cfg), 148, 1, 0, None, ctypes.c_int64(0), ctypes.byref(cnt)) == zgr.EINVAL
