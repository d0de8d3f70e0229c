"""The subspace update at the edges of its kernels' tiles, against the fp64 oracle.

The step runs a CTA per 64 rows of U with 4 x 4 register tiles of the k x k products,
shared by groups of threads for small k; past one CTA per SM (152 x 64 rows) a CTA
owns several blocks of rows.  The accumulation transposes Cg 64 tokens at a time.
Bars: those of the update's other tests (1e-4 relative for the step, U^T U = I to
1e-5, 1e-2 for M, 1e-3 for the residual).
"""
import numpy as np
import pytest
import torch

from gpu_util import dev, widen
from paper_2506_01260_gb300 import workloads as W
from test_grassmann_gpu import basis_and_grads, grassmann_oracle, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,k", [(16, 1), (64, 4), (72, 5), (128, 33), (200, 64), (264, 65),
                                 (1000, 89), (520, 128), (12008, 8), (9800, 41)])
def test_step_shapes(sn, d, k):
    g = grassmann_oracle()
    rng = np.random.default_rng(d + k)
    U32 = W.orthonormal_basis(d, k, rng).astype(np.float32)
    # any M has a tangent part; a step of about a tenth of the basis
    M32 = (U32 @ rng.standard_normal((k, k)) + rng.standard_normal((d, k)) / np.sqrt(d)).astype(np.float32)
    eta = 0.1 / (2.0 * np.linalg.norm(M32.astype(np.float64), 2) / 3)
    basis = sn.Basis(dev(U32))
    U1 = sn.sn_grassmann_step(basis, dev(M32), 3, eta)
    U2 = sn.sn_grassmann_step(basis, dev(M32), 3, eta)
    sn.sn_check_errors(basis)
    assert torch.equal(U1, U2)                       # no order of arrival in the sums
    got = U1.cpu().numpy().astype(np.float64)
    ref = g.step(U32.astype(np.float64), M32.astype(np.float64), 3, eta)
    assert rel(got, ref) <= 1e-4
    assert np.max(np.abs(got.T @ got - np.eye(k))) <= 1e-5
    basis.destroy()


@pytest.mark.parametrize("d,k,T", [(128, 7, 1), (256, 33, 63), (264, 64, 65), (512, 127, 129),
                                   (136, 2, 40000)])
def test_accumulate_shapes(sn, d, k, T):
    g = grassmann_oracle()
    U32, (Gb,) = basis_and_grads(sn, d, k, T, 1, seed=T + k)
    basis = sn.Basis(dev(U32))
    G = dev(Gb)
    Cg = sn.sn_compress_bwd(basis, G)
    M = torch.zeros(d, k, dtype=torch.float32, device="cuda")
    acc = torch.zeros(1, dtype=torch.float64, device="cuda")
    sn.sn_grassmann_accumulate(basis, G, Cg, M)
    sn.sn_grassmann_residual(basis, G, Cg, acc)
    sn.sn_check_errors(basis)
    G64, U64 = widen(Gb), U32.astype(np.float64)
    assert rel(M.cpu().numpy().astype(np.float64), g.accumulate(np.zeros((d, k)), G64, U64)) <= 1e-2
    assert abs(acc.item() - g.residual(G64, U64)) <= 1e-3 * np.sum(G64 * G64)
    basis.destroy()


@pytest.mark.parametrize("signs", [(1, 1, -1, -1), (1, -1, 1, -1)])
def test_step_sums_past_fp32(sn, signs):
    """Block sums of U^T M near fp32's largest number, two of either sign: on the way the sum
    passes what fp32 holds, and is 0 in the end.  The step moves U by about 24 times its
    norm; bars as above."""
    g = grassmann_oracle()
    d, eta = 256, 1e-38
    U32 = np.full((d, 1), 1 / 16, np.float32)
    M32 = np.repeat(np.float32(7.5e37) * np.array(signs, np.float32), 64).reshape(d, 1)
    basis = sn.Basis(dev(U32))
    got = sn.sn_grassmann_step(basis, dev(M32), 1, eta)
    sn.sn_check_errors(basis)
    got = got.cpu().numpy().astype(np.float64)
    # the step size reaches the kernel as 2 eta rounded to fp32
    ref = g.step(U32.astype(np.float64), M32.astype(np.float64), 1, float(np.float32(2 * np.float32(eta))) / 2)
    assert rel(got, ref) <= 1e-4
    assert abs((got.T @ got).item() - 1) <= 1e-5
    basis.destroy()


@pytest.mark.parametrize("d,k,T", [(128, 7, 1), (256, 33, 63), (264, 64, 65), (512, 127, 129),
                                   (136, 2, 20000)])
def test_accumulate_and_residual_of_what_the_kernels_read(sn, d, k, T):
    """G^T Cg and |G|^2 - |Cg|^2 in fp64 from the bf16 G and Cg themselves.  M: products exact in
    fp32, an addition for every 16 tokens and split, each off by at most an ulp of a sum no
    larger than the last.  The residual: runs of 128 squares in fp32, off by about
    sqrt(128) / 2 * 2^-24 = 3.4e-7 of themselves at random, the rest in fp64.  Both bars lie below
    what one lost token, or one lost 16-byte piece of G, makes."""
    U32, (Gb,) = basis_and_grads(sn, d, k, T, 1, seed=T + k)
    basis = sn.Basis(dev(U32))
    G = dev(Gb)
    Cg = sn.sn_compress_bwd(basis, G)
    M0 = torch.full((d, k), 0.5, device="cuda")
    M, acc = M0.clone(), torch.full((1,), 3.0, dtype=torch.float64, device="cuda")
    sn.sn_grassmann_accumulate(basis, G, Cg, M)
    sn.sn_grassmann_residual(basis, G, Cg, acc)
    sn.sn_check_errors(basis)
    G64, C64 = G.double(), Cg.double()
    want, sq = M0.double() + G64.T @ C64, G64.square().sum().item()
    m_bar, r_bar = (T / 16 + 16) * 2.0 ** -23 * want.norm().item(), 1e-6 * (sq + C64.square().sum().item())
    assert (M.double() - want).norm().item() <= m_bar
    assert abs(acc.item() - 3.0 - (sq - C64.square().sum().item())) <= r_bar
    lost = min((G64[t].norm() * C64[t].norm()).item() for t in (0, T // 2, T - 1))
    assert m_bar < lost and r_bar < G64[-1, -8:].square().sum().item()
    basis.destroy()
