"""zgr_build_subspace takes a second Cholesky pass only where the first one's factor asks for it (needs a B200): directions on either side
of that line, in the cluster and the grid launch, give the basis of a QR factorisation in 64 bits to one rounding of fp32."""
import pytest
import torch

from paper_2601_12917_b200 import zgr

pytestmark = pytest.mark.gpu


# Condition numbers 1 to 1e6 (the line is at about 100 for these): an error of 1e-10 from one pass, or condition times 1e-16 from two, is far
# below the rounding of the result, half an ulp or 2^-24 of an entry; 1e-9 is left for the rest.
@pytest.mark.parametrize("cond", [1.0, 10.0, 50.0, 100.0, 200.0, 1e3, 1e6])
@pytest.mark.parametrize("rows,r", [(500, 3), (2048, 16), (9000, 16), (1500, 33), (7000, 64)])
def test_one_pass_or_two(rows, r, cond):
    z = zgr.Zgr([torch.zeros(rows, 8, device="cuda")], [torch.zeros(rows, r, device="cuda")], 0.5, 1e-3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(rows + r)
    left = torch.linalg.qr(torch.randn(rows, r, generator=gen, device="cuda", dtype=torch.float64))[0]
    right = torch.linalg.qr(torch.randn(r, r, generator=gen, device="cuda", dtype=torch.float64))[0]
    spread = torch.logspace(0, -torch.log10(torch.tensor(cond)).item(), r, device="cuda", dtype=torch.float64)
    A = ((left * spread) @ right).float().contiguous()
    z.build_subspace(0, A)
    U = z._keep[1][0].double()
    Q, R = torch.linalg.qr(A.double())
    Q = Q * torch.sign(torch.diagonal(R))
    assert ((U - Q).abs() <= 2.0 ** -24 * Q.abs() + 1e-9).all()
    assert (U.T @ U - torch.eye(r, device="cuda", dtype=torch.float64)).abs().max() <= 1.2e-7
