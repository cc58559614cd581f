"""The kernels that are chosen by size, type and row length, at the sizes where they can go wrong (needs a B200):
edges of tiles and octets in the tile kernel (the staged kernel, which takes larger sets, has a file of its own), low ranks on the tensor-core kernels, more items than blocks, bases on
either side of the cluster and grid launches.  Every call against the oracle, with the tolerances of helpers.py."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_12917_b200 import synth, zgr

from helpers import Pair
from test_plan import kernels, plan

pytestmark = pytest.mark.gpu


# Octets straddle row ends when the row length is no multiple of eight: lengths below, at and above one octet, one strip of
# 128 columns and its overlap of 16, row counts around a warp's 32 and a tile's 128 rows, every contraction width.
@pytest.mark.parametrize("dtype,bits", [("f32", 32), ("f32", 16), ("bf16", 16), ("f16", 32)])
@pytest.mark.parametrize("rows,cols,rank", [(5, 3, 2), (33, 7, 16), (128, 9, 4), (31, 127, 17), (129, 129, 9), (127, 137, 33), (257, 150, 64), (300, 1285, 16),
                                            (64, 263, 1)])
def test_rows_that_are_no_multiple_of_eight(rows, cols, rank, dtype, bits):
    p = Pair([(rows, cols), (1, 37)], [rank, 0], dtype, bits=bits, seed=rows + cols)
    p.lib.profile(True)
    reports = p.step(seed=17, lp=2.4, lm=1.7, lr=1e-4)
    assert {k["path"] for k in p.lib.profile_read()} == {"generic", "iso"}
    assert all(rep["moved"] > 0.3 for call in reports[:2] for rep in call)
    assert p.lib.device_status() == 0


# fp32 with rank above 8 in whole octets: one short strip, exact tiles, ragged last rows and strip; several tensors, so that
# a block works on items of different tensors and widths.
@pytest.mark.parametrize("bits", [16, 32])
@pytest.mark.parametrize("shapes,ranks", [([(40, 8), (1, 9)], [9, 0]), ([(128, 128), (1, 9)], [16, 0]), ([(130, 264), (385, 136), (1, 9)], [32, 24, 0]),
                                          ([(200, 520), (96, 72), (1, 9)], [64, 40, 0])])
def test_fp32_above_rank_8(shapes, ranks, bits):
    p = Pair(shapes, ranks, "f32", bits=bits, seed=5)
    p.step(seed=3, lp=1.8, lm=2.3, lr=1e-4)
    assert p.lib.device_status() == 0


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_tile_kernel_norms_codes_and_several_seeds(dtype):
    shapes, ranks = [(150, 203), (70, 136), (1, 25)], [20, 12, 0]
    p = Pair(shapes, ranks, dtype, bits=16, seed=8, stats=True, alpha=0.4)
    G = oracle.coeffs(9, 0, 16, 20, 203)
    q, sc, ze = oracle.dtc_quantise_int4(G)
    p.set_dtc(0, q, sc, ze, bits=4)
    p.step(seed=31, lp=2.2, lm=1.9, lr=1e-4)
    got = p.lib.get_stats(31)
    for l in range(3):
        np.testing.assert_allclose(got[l], oracle.stats_tensor(p.oracle_tensor(l), 31, l, 16, p.a, p.b), rtol=2e-5, atol=1e-9)
    p.lib.enable_stats(False)
    seeds, lp, lm = [41, 42, 43], [2.1, 1.6, 2.4], [1.9, 2.0, 1.8]
    coeffs = [oracle.update_coefficient(0.0, a, b, p.eps, 1e-4) for a, b in zip(lp, lm)]
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "three seeds")


# Codes for rows of whole octets, which the strip reads eight at a time, all rows of the tensor coded or the first seven; one and two seeds.
@pytest.mark.parametrize("code_bits", [8, 4])
@pytest.mark.parametrize("n_rows", [None, 7])
def test_tile_kernel_codes_in_whole_octets(code_bits, n_rows):
    p = Pair([(150, 264), (1, 25)], [12, 0], "f32", bits=16, seed=8)
    if code_bits == 8:
        p.set_dtc(0, *synth.dtc_payload(12, 264, seed=3), bits=8, n_rows=n_rows)
    else:
        p.set_dtc(0, *oracle.dtc_quantise_int4(oracle.coeffs(9, 0, 16, 12, 264)), bits=4, n_rows=n_rows)
    p.step(seed=31, lp=2.2, lm=1.9, lr=1e-4)
    seeds, lp, lm = [41, 42], [2.1, 1.6], [1.9, 2.0]
    coeffs = [oracle.update_coefficient(0.0, a, b, p.eps, 1e-4) for a, b in zip(lp, lm)]
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "two seeds")


# Sets with more items than SMs: the staged and the tile kernel draw on their item counters (below about 29 M weights each block has a share of its
# own), in items of the two heights that the planner chose, and put the counter back to zero: five sweeps of one context in a row.
@pytest.mark.parametrize("dtype,shapes,ranks,kernel", [("bf16", [(4000, 5001), (2000, 5001), (1, 77)], [16, 16, 0], "staged"),
                                                        ("f32", [(4000, 5128), (2000, 5128), (1, 77)], [24, 24, 0], "staged"),
                                                        ("f32", [(4000, 5001), (2000, 5001), (1, 77)], [24, 24, 0], "tile")])
def test_tile_items_from_the_counter(dtype, shapes, ranks, kernel):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert kernels(shapes, ranks, [{"f32": zgr.F32, "bf16": zgr.BF16}[dtype]] * 3, sm_count=sms) == [kernel, kernel, "iso"]
    items = [it for it in plan(shapes, ranks, [{"f32": zgr.F32, "bf16": zgr.BF16}[dtype]] * 3, sm_count=sms) if it.path == 3]
    assert len(items) > sms and (32 + 16) * 40 >= 12 * sms        # more items than blocks, and enough tiles for the counter
    assert len({(it.nrows_or_count + 127) // 128 for it in items}) > 1
    p = Pair(shapes, ranks, dtype, bits=16, seed=9)
    p.step(seed=3, lp=2.3, lm=1.7, lr=1e-4)
    p.call_and_check(4, 1e-3, lambda: p.lib.perturb(4, 1e-3), "perturb")
    p.call_and_check(4, -1e-3, lambda: p.lib.restore_update(4, 2.0, 2.0, 0.0), "restore")
    assert p.lib.device_status() == 0


# Low ranks: sets of 2^21 weights and more leave the CUDA-core kernel for the tile kernel (larger ones for the staged one), which is reported under the same path with its
# contraction width (narrow and ragged last strips of the CUDA-core kernel are in the parity tests).
@pytest.mark.parametrize("dtype,path", [("bf16", "fma"), ("f16", "fma"), ("f32", "fma")])
@pytest.mark.parametrize("rank", [1, 4, 8])
def test_low_rank_sets_of_some_size(dtype, path, rank):
    p = Pair([(1030, 2056), (1, 40), (140, 72)], [rank, 0, rank], dtype, bits=16, seed=2)
    p.lib.profile(True)
    p.step(seed=6, lp=2.0, lm=1.7, lr=1e-4)
    read = p.lib.profile_read()
    assert {k["path"]: k["kpad"] for k in read} == {path: 16, "iso": 0}
    assert {k["kernel"] for k in read} == {"tile", "iso"}
    assert p.lib.device_status() == 0


# A subspace that is not normalised: entries up to 2^12 in size, which two fp16 parts cannot hold at any rows' scale.  On either side of
# 2^21 weights the same model gives the same z; the tolerances are those of helpers.check_sweep for a z that is `size` times larger.
@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("rows", [500, 1030])
def test_low_rank_subspace_of_any_size(rows, dtype):
    size = 2.0 ** 15
    p = Pair([(rows, 2056), (1, 40)], [8, 0], dtype, bits=16, seed=2)
    p.U[0] *= size
    p.lib.update_subspace(0)
    p.z_unit, p.sigma_z = (lambda: size), (lambda l: float(np.sqrt(p.a ** 2 + (p.b * size) ** 2 * 8 / rows)) if l == 0 else p.a)
    assert float(p.U[0].abs().max()) > 2.0 ** 11
    p.call_and_check(3, 1e-3 / size, lambda: p.lib.perturb(3, 1e-3 / size), "perturb")
    p.call_and_check(3, -1e-3 / size, lambda: p.lib.restore_update(3, 2.0, 2.0, 0.0), "restore")


# Strips of the CUDA-core kernel of at most 32, 64 and 128 columns: 8, 4 and 2 rows per warp.
@pytest.mark.parametrize("cols", [8, 32, 40, 64, 72, 128, 136, 392])
def test_narrow_strips(cols):
    p = Pair([(77, cols), (9, cols), (1, 8)], [8, 3, 0], "f32", bits=32, seed=cols)
    p.step(seed=12, lp=2.0, lm=1.6, lr=1e-4)


# z of a 16-bit tensor without a subspace (the hook sweeps an fp32 image with the hardware-approximation transform).
@pytest.mark.parametrize("bits", [16, 32])
def test_z_of_a_16_bit_tensor_without_a_subspace(bits):
    p = Pair([(70, 264), (1, 5001)], [9, 0], "bf16", bits=bits, seed=6)
    z = oracle.z_tensor(p.oracle_tensor(1), 77, 1, bits, p.a, p.b).ravel()
    assert np.abs(p.lib.debug_z(77, 1).double().cpu().numpy().ravel() - z).max() <= 1e-5


# 1-D tensors in the launch of the CUDA-core kernel (small sets): aligned, ragged and unaligned ones, one and several seeds.
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_one_dimensional_tensors_ride_along(dtype):
    p = Pair([(96, 256), (1, 1), (1, 9), (1, 5003), (40, 72), (1, 4096)], [4, 0, 0, 0, 8, 0], dtype, bits=16, seed=3)
    launches = p.lib.launch_count()
    p.step(seed=5, lp=2.1, lm=1.7, lr=1e-4)
    assert p.lib.launch_count() - launches == 6              # three sweeps, one kernel per contraction width
    seeds, lp, lm = [41, 42], [2.1, 1.6], [1.9, 2.0]
    coeffs = [oracle.update_coefficient(0.0, a, b, p.eps, 1e-4) for a, b in zip(lp, lm)]
    p.call_and_check_multi(seeds, coeffs, lambda: p.lib.restore_update_multi(seeds, lp, lm, 1e-4), "two seeds")


# More items than resident blocks: the item counter is used and put back to zero (three sweeps of one context in a row).
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_isotropic_sweeps_with_more_items_than_blocks(dtype):
    p = Pair([(1201, 2569), (3, 5)], [0, 0], dtype, bits=16, seed=4, alpha=1.0)
    p.step(seed=8, lp=2.3, lm=1.6, lr=1e-4)
    p.step(seed=9, lp=1.9, lm=2.2, lr=1e-4)


# 4096 entries per block of a cluster, then one block per SM; ranks that are padded; a short last block.  The last two
# exceed the shared memory of the whole chip and take the three-kernel path.
@pytest.mark.parametrize("rows,r", [(1, 1), (16, 16), (2048, 16), (2049, 16), (1025, 17), (513, 33), (9000, 64), (20001, 5), (60000, 64), (230000, 2)])
def test_basis_on_either_side_of_the_launch_shapes(rows, r):
    w = torch.zeros(rows, 8, device="cuda", dtype=torch.float32)
    z = zgr.Zgr([w], [torch.zeros(rows, r, device="cuda")], 0.5, 1e-3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows)
    A = torch.randn(rows, r, generator=gen, device="cuda") * torch.logspace(0, -3, r, device="cuda")
    for _ in range(2):                                     # the barrier counter is back at zero for the second call
        z.build_subspace(0, A.contiguous())
    U = z._keep[1][0].double()
    assert (U.T @ U - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max() <= 1e-6
    Q, R = torch.linalg.qr(A.double())
    Q = Q * torch.sign(torch.diagonal(R))
    assert (U - Q).abs().max() <= 1e-5
    if r > 1:                                              # dependent columns are refused whatever the launch, and nothing is written
        B = A.clone()
        B[:, r - 1] = B[:, 0]
        with pytest.raises(zgr.ZgrError) as e:
            z.build_subspace(0, B.contiguous())
        assert e.value.code == zgr.EINVAL
        assert torch.equal(z._keep[1][0].double(), U)


# Nearly parallel directions are independent down to an angle of 4.5e-8, whatever the launch: the basis of directions 6e-8 apart, one fp32
# rounding, is delivered as right as any (bounds as above), and an exact copy is refused.
@pytest.mark.parametrize("rows,r", [(2048, 2), (9000, 2), (20001, 33), (60000, 64), (230000, 2)])
def test_nearly_parallel_directions(rows, r):
    z = zgr.Zgr([torch.zeros(rows, 8, device="cuda")], [torch.zeros(rows, r, device="cuda")], 0.5, 1e-3)
    gen = torch.Generator(device="cuda")
    for seed in range(6):
        gen.manual_seed(seed)
        A = torch.randn(rows, r, generator=gen, device="cuda").double()
        A[:, r - 1] = A[:, 0] + 6e-8 * torch.randn(rows, generator=gen, device="cuda").double()
        A = A.float().contiguous()
        z.build_subspace(0, A)
        U = z._keep[1][0].double()
        assert (U.T @ U - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max() <= 1e-6
        Q, R = torch.linalg.qr(A.double())
        assert (U - Q * torch.sign(torch.diagonal(R))).abs().max() <= 1e-5
        A[:, r - 1] = A[:, 0]
        with pytest.raises(zgr.ZgrError) as e:
            z.build_subspace(0, A)
        assert e.value.code == zgr.EINVAL


# Accuracy of the fp32 transform against 64 bits: 3 M normals of an fp32 tensor without a subspace.  The one-pair form is off by 7.2e-8 rms
# and 8.9e-7 at most; the two-pair form that the kernels use may not be further off (it was, 9.3e-8 and 1.1e-6, with the
# lean of the hardware logarithm and square root left in).
@pytest.mark.parametrize("bits", [16, 32])
def test_normals_of_fp32_tensors(bits):
    p = Pair([(2048, 1536)], [0], "f32", bits=bits, seed=1, alpha=1.0)
    err = p.lib.debug_z(5, 0).double().cpu().numpy().ravel() - oracle.z_tensor(p.oracle_tensor(0), 5, 0, bits, p.a, p.b).ravel()
    assert np.sqrt(np.mean(err ** 2)) <= 7.2e-8 and np.abs(err).max() <= 9e-7


# Accuracy of the tile kernel's contraction against 64 bits, alone (alpha = 0) and on coefficients with all 24 bits (codes minus an odd zero
# point, formed here as the kernel forms them): not behind a chain of fp32 multiply-adds, whose error is given first (one fp32
# rounding is 2.5e-8, the truncation of the tensor cores alone 4.6e-8 to 7.7e-8).
@pytest.mark.parametrize("cols", [1536, 1537])
@pytest.mark.parametrize("rank,chain", [(2, 3.4e-8), (4, 4.0e-8), (8, 5.0e-8), (16, 7.6e-8), (32, 1.0e-7), (64, 1.5e-7)])
def test_contraction_of_fp32_tensors(rank, chain, cols):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rank)
    w = torch.zeros(2048, cols, device="cuda")
    U = torch.linalg.qr(torch.randn(2048, rank, generator=gen, device="cuda"))[0].contiguous()
    q = torch.randint(-127, 128, (rank, cols), generator=gen, device="cuda").to(torch.int8)
    scale, zero = (torch.rand(rank, generator=gen, device="cuda") + 0.5) / 64, 2 * torch.rand(rank, generator=gen, device="cuda") - 1
    z = zgr.Zgr([w], [U], 0.0, 1e-3, zgr.SCALE_PAPER, 16)
    z.set_coeffs_dtc(0, q, scale, zero)
    z.perturb(1, 1e-3)                                     # (also brings the codes into the device's table)
    z.restore_update(1, 2.0, 2.0, 0.0)
    b = torch.tensor(z.scalars()[1], dtype=torch.float64, device="cuda").float()
    exact = U.double() @ ((scale * b)[:, None] * (q.float() - zero[:, None])).double()
    err = z.debug_z(1, 0).double() - exact
    assert float(err.norm() / exact.norm()) <= chain
    assert abs(float((err * exact.sign()).sum() / exact.abs().sum())) <= 1e-8      # and no lean
