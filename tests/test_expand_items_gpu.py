"""Plain expansion where a CTA runs several row tiles: from the second one on, other
warps prepare the coefficients, in a second buffer, while the first is still read."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,k", [(39000, 256, 9), (128 * 305 + 1, 128, 64), (60001, 264, 65),
                                   (128 * 456, 384, 128)])
def test_many_row_tiles(sn, T, d, k):
    gen = torch.Generator().manual_seed(T + k)
    U = torch.linalg.qr(torch.randn(d, k, generator=gen, dtype=torch.float64))[0]
    basis = sn.Basis(U.float().contiguous().cuda())
    C = torch.randn(T, k, generator=gen).bfloat16().cuda()
    got = torch.empty(T, d, device="cuda", dtype=torch.bfloat16)
    sn.sn_decompress_bwd(basis, C, out=got)
    sn.sn_check_errors(basis)
    Ub = U.float().bfloat16().double().cuda()       # the tensor cores read U in bf16
    want = C.double() @ Ub.T
    # exact products summed in fp32 (k steps, 2^-23 each at most), one rounding to bf16
    bound = want.abs() * 2.0 ** -8 + (C.double().abs() @ Ub.abs().T) * k * 2.0 ** -23
    assert ((got.double() - want).abs() <= bound).all()
    basis.destroy()
