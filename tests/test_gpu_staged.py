"""The sweep whose weights are staged by TMA and whose operands have three parts, at the sizes where it can go wrong (needs a B200):
rows that are no multiple of eight elements long around octets, strips and spans of 256 rows, residues without rows, several tensors
of different row lengths in one launch.  Every call against the oracle, with the tolerances of helpers.py.  A set takes this kernel from
2.6 M weights on (fp32 up to rank 16: 6.8 M), hence the large first tensors."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_12917_b200 import zgr

from helpers import Pair
from test_plan import HALVES, kernels, plan

pytestmark = pytest.mark.gpu

LARGE = (1300, 2051)
# rows: fewer than eight residues, around a quarter's 32 lanes and a span; columns: two octets, one strip and one less or more, ends of rows
# that begin or end a strip
RAGGED = [(5, 17), (1, 143), (255, 19), (256, 127), (257, 129), (264, 135), (31, 263), (300, 385), (7, 2049)]


@pytest.mark.parametrize("dtype,bits", [("bf16", 16), ("f16", 32)])
@pytest.mark.parametrize("rank", [1, 16, 20, 64])
def test_ragged_rows(rank, dtype, bits):
    shapes = [LARGE] + RAGGED + [(1, 37)]
    ranks = [min(rank, m) for m, _ in shapes[:-1]] + [0]
    kinds = [{"f16": zgr.F16, "bf16": zgr.BF16}[dtype]] * len(shapes)
    assert all(it.row0_or_e0 % 256 == 0 for it in plan(shapes, ranks, kinds, bits=bits) if it.path == 3)      # whole spans
    p = Pair(shapes, ranks, dtype, bits=bits, seed=rank)
    p.lib.profile(True)
    reports = p.step(seed=17, lp=2.4, lm=1.7, lr=1e-4)
    assert {k["kernel"] for k in p.lib.profile_read()} == {"staged", "iso"}
    assert all(rep["moved"] > 0.3 for call in reports[:2] for rep in call)
    assert p.lib.device_status() == 0


# Rows shorter than two octets, and weights that do not begin on a 16-byte boundary, stay with the tile kernel beside it; the smaller fp32 set does
# altogether.
@pytest.mark.parametrize("dtype,cols", [("bf16", 2056), ("f32", 2056), ("f32", 5304)])
def test_whole_octets_beside_other_rows(dtype, cols):
    p = Pair([(1300, cols), (40, 15), (130, 64), (129, 72), (1, 136), (257, 200), (385, 129), (1, 9)], [16 if dtype == "f32" else 8, 3, 8, 4, 1, 8, 12, 0], dtype, bits=32, seed=4)
    p.step(seed=3, lp=1.8, lm=2.3, lr=1e-4)
    assert p.lib.device_status() == 0


@pytest.mark.parametrize("dtype,cols", [("bf16", 2051), ("f32", 2056), ("f32", 5304)])
@pytest.mark.parametrize("rank", [12, 40])
def test_norms_codes_and_several_seeds(rank, dtype, cols):
    shapes, ranks = [(1300, cols), (150, 203 if dtype == "bf16" else 200), (1, 25)], [rank, 20, 0]
    p = Pair(shapes, ranks, dtype, bits=16, seed=8, stats=True, alpha=0.4)
    q, sc, ze = oracle.dtc_quantise_int4(oracle.coeffs(9, 0, 16, ranks[1], shapes[1][1]))
    p.set_dtc(1, q, sc, ze, bits=4)
    p.step(seed=31, lp=2.2, lm=1.9, lr=1e-4)
    got = p.lib.get_stats(31)
    for l in range(3):
        np.testing.assert_allclose(got[l], oracle.stats_tensor(p.oracle_tensor(l), 31, l, 16, p.a, p.b), rtol=2e-5, atol=1e-9)
    p.lib.enable_stats(False)
    seeds, lp, lm = [41, 42, 43], [2.1, 1.6, 2.4], [1.9, 2.0, 1.8]
    coeffs = [oracle.update_coefficient(0.0, a, b, p.eps, 1e-4) for a, b in zip(lp, lm)]
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "three seeds")


# Shares that begin and end in the middle of a span, in last spans of every kind: one seed with norms and without, several seeds.
@pytest.mark.parametrize("rank,bits", [(16, 16), (64, 32)])
def test_shares_in_halves_of_spans(rank, bits):
    ranks = [min(rank, m) for m, _ in HALVES]
    assert any(it.row0_or_e0 % 256 for it in plan(HALVES, ranks, [zgr.BF16] * len(HALVES), bits=bits))
    p = Pair(HALVES, ranks, "bf16", bits=bits, seed=rank, stats=True)
    p.step(seed=21, lp=2.2, lm=1.9, lr=1e-4)
    got = p.lib.get_stats(21)
    for l in range(len(HALVES)):
        np.testing.assert_allclose(got[l], oracle.stats_tensor(p.oracle_tensor(l), 21, l, bits, p.a, p.b), rtol=2e-5, atol=1e-9)
    p.lib.enable_stats(False)
    p.call_and_check(22, 1e-3, lambda: p.lib.perturb(22, 1e-3), "perturb")
    p.call_and_check(22, -1e-3, lambda: p.lib.restore_update(22, 2.0, 2.0, 0.0), "restore")
    coeffs = [oracle.update_coefficient(0.0, 2.1, 1.9, p.eps, 1e-4), oracle.update_coefficient(0.0, 1.6, 2.0, p.eps, 1e-4)]
    p.call_and_check_multi([41, 42], coeffs, lambda: p.lib.restore_update_multi([41, 42], [2.1, 1.6], [1.9, 2.0], 1e-4), "two seeds")
    assert p.lib.device_status() == 0


# Items from the counter where the accumulated norms, one strip at a time (rank above 32) and several seeds go with them.
def test_norms_and_several_seeds_from_the_counter():
    shapes, ranks = [(4000, 5001), (2000, 5001), (1, 77)], [64, 40, 0]
    assert kernels(shapes, ranks, [zgr.BF16] * 3) == ["staged", "staged", "iso"]
    assert sum(it.path == 3 for it in plan(shapes, ranks, [zgr.BF16] * 3)) > torch.cuda.get_device_properties(0).multi_processor_count
    p = Pair(shapes, ranks, "bf16", bits=16, seed=9, stats=True)
    p.call_and_check(3, 1e-3, lambda: p.lib.perturb(3, 1e-3), "perturb")
    got = p.lib.get_stats(3)
    for l in range(3):
        np.testing.assert_allclose(got[l], oracle.stats_tensor(p.oracle_tensor(l), 3, l, 16, p.a, p.b), rtol=2e-5, atol=1e-9)
    p.call_and_check(3, -1e-3, lambda: p.lib.restore_update(3, 2.0, 2.0, 0.0), "restore")
    coeffs = [oracle.update_coefficient(0.0, 2.1, 1.9, p.eps, 1e-4), oracle.update_coefficient(0.0, 1.6, 2.0, p.eps, 1e-4)]
    p.call_and_check_multi([41, 42], coeffs, lambda: p.lib.restore_update_multi([41, 42], [2.1, 1.6], [1.9, 2.0], 1e-4), "two seeds")
    assert p.lib.device_status() == 0


# Ragged sets whose spans cost a tile of the busiest SM (four tiles against three): one seed on the staged kernel, several on the tile kernel,
# which reads the copies of U kept by residue in the order of the rows.  A new subspace reaches both.
@pytest.mark.parametrize("rank,dtype,bits", [(16, "f16", 16), (20, "bf16", 32), (64, "bf16", 16)])
def test_several_seeds_on_the_tile_kernel(rank, dtype, bits):
    shapes, ranks = [(6917, 131)] * 4 + [(1, 9)], [rank, rank, rank, 9, 0]
    p = Pair(shapes, ranks, dtype, bits=bits, seed=rank)
    p.lib.profile(True)
    p.step(seed=3, lp=1.8, lm=2.3, lr=1e-4)
    assert {k["kernel"] for k in p.lib.profile_read()} == {"staged", "iso"}
    seeds, lp, lm = [41, 42, 43, 44], [2.1, 1.6, 2.4, 1.7], [1.9, 2.0, 1.8, 2.2]
    coeffs = [oracle.update_coefficient(0.0, a, b, p.eps, 1e-4) for a, b in zip(lp, lm)]
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "four seeds")
    assert {k["kernel"] for k in p.lib.profile_read()} == {"tile", "iso"}
    p.U[1].copy_(p.U[1].flip(0))
    p.lib.update_subspace(1)
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "four seeds, new subspace")
    p.step(seed=4, lp=1.8, lm=2.3, lr=1e-4)
    assert p.lib.device_status() == 0


# Sets between 12 and 24 tiles per SM: items from the counter for one seed, another plan in shares for several, in turn.
def test_several_seeds_in_shares_of_their_own():
    shapes, ranks = [(25600, 131)] * 5 + [(1, 9)], [16, 16, 9, 16, 16, 0]
    dtypes = [zgr.BF16] * 6
    assert len(plan(shapes, ranks, dtypes)) != len(plan(shapes, ranks, dtypes, multi=1)) and kernels(shapes, ranks, dtypes, multi=1)[0] == "staged"
    p = Pair(shapes, ranks, "bf16", bits=16, seed=7)
    coeffs = [oracle.update_coefficient(0.0, 2.1, 1.9, p.eps, 1e-4), oracle.update_coefficient(0.0, 1.6, 2.0, p.eps, 1e-4)]
    for seed in (3, 4):
        p.step(seed=seed, lp=1.8, lm=2.3, lr=1e-4)
        p.call_and_check_multi([41, 42], coeffs, lambda: p.lib.restore_update_multi([41, 42], [2.1, 1.6], [1.9, 2.0], 1e-4), "two seeds")
    assert p.lib.device_status() == 0


# A delivered and a constructed subspace reach the copies of U that are kept by residue.
def test_new_subspaces_of_ragged_tensors():
    p = Pair([LARGE, (300, 385), (1, 9)], [16, 16, 0], "bf16", bits=16, seed=6)
    for l in (0, 1):
        p.U[l].copy_(p.U[l].flip(0))
    p.lib.update_subspace(0)
    p.lib.build_subspace(1, (p.U[1].flip(1) * 3.0).contiguous())
    p.step(seed=5, lp=2.0, lm=1.6, lr=1e-4)
    p.lib.update_subspaces([0, 1], [p.U[0], p.U[1]])
    p.step(seed=6, lp=2.0, lm=1.6, lr=1e-4)


# The same tensor alone (tile kernel) and beside a larger one (staged kernel), the sizes chosen so that the mixing scalars are the same: equal
# bits, whole octets and ends of rows alike.  On zero weights, whose result keeps the step's own 11 bits, so that one rounding of
# the fp32 step more or less shows (in about a dozen of the 112 000 elements at the ends).
@pytest.mark.parametrize("bits", [16, 32])
def test_ends_of_rows_as_in_the_tile_kernel(bits):
    rows, cols, rank = 16000, 61, 16                                       # d / K = rows / rank = 1000 in both sets
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    U = torch.linalg.qr(torch.randn(rows, rank, generator=gen, device="cuda"))[0].contiguous()
    V = torch.linalg.qr(torch.randn(1000, 1, generator=gen, device="cuda"))[0].contiguous()
    results = []
    for beside in (False, True):
        w, big = (torch.zeros(m, n, device="cuda", dtype=torch.float16) for m, n in ((rows, cols), (1000, 2051)))
        z = zgr.Zgr([w, big] if beside else [w], [U, V] if beside else [U], 0.5, 1e-3, zgr.SCALE_UNIT, bits)
        z.perturb(9, 1.0)
        one = w.clone()
        w.zero_()
        z.sweep_multi([10, 11], [0.75, -1.0])
        results.append((np.float32(z.scalars()), one, w))
    assert (results[0][0] == results[1][0]).all()
    assert torch.equal(results[0][1], results[1][1]) and torch.equal(results[0][2], results[1][2])
