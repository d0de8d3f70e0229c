"""GPU parity of the row-constant AdamW step (Sec. 5) against the fp64 oracle in
oracle/adamw.py.  Bar: 1e-5 relative Frobenius error on W, M and V after three
steps (fp32 arithmetic; bf16 gradients are handed to the oracle as the exact
values the GPU saw), and a weight in S stays in S to 1e-5 relative."""
import importlib.util
import os

import numpy as np
import pytest
import torch

from gpu_util import widen
from paper_2506_01260_gb300 import workloads as W_

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
HP = dict(lr=3e-3, beta1=0.9, beta2=0.95, eps=1e-8, lam=1e-4)


def adamw_oracle():
    spec = importlib.util.spec_from_file_location("oracle_adamw",
                                                  os.path.join(HERE, "..", "oracle", "adamw.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("gdt", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols", [(512, 1000), (4096, 300), (7, 3), (130, 1002)])
def test_three_steps_match_oracle(sn, gdt, rows, cols):
    a = adamw_oracle()
    rng = np.random.default_rng(rows + cols)
    W0 = rng.standard_normal((rows, cols)).astype(np.float32)
    W = torch.tensor(W0, device="cuda")
    M = torch.zeros_like(W)
    V = torch.zeros_like(W)
    W64, M64, V64 = W0.astype(np.float64), np.zeros((rows, cols)), np.zeros((rows, cols))
    for t in (1, 2, 3):
        g64 = rng.standard_normal((rows, cols)) * rng.uniform(0.1, 3.0, (1, cols))
        if gdt == "bf16":
            gb = W_.to_bf16(g64)
            g = torch.from_numpy(gb.view(np.int16)).view(torch.bfloat16).cuda()
            gx = widen(gb)
        else:
            g = torch.tensor(g64.astype(np.float32), device="cuda")
            gx = g64.astype(np.float32).astype(np.float64)
        sn.sn_adamw_rowconst(W, g, M, V, t, HP["lr"], HP["beta1"], HP["beta2"], HP["eps"],
                             HP["lam"])
        W64, M64, V64 = a.step(W64, gx, M64, V64, t, HP["lr"], HP["beta1"], HP["beta2"],
                               HP["eps"], HP["lam"])
    torch.cuda.synchronize()
    assert rel(W.cpu().numpy().astype(np.float64), W64) <= 1e-5
    assert rel(M.cpu().numpy().astype(np.float64), M64) <= 1e-5
    assert rel(V.cpu().numpy().astype(np.float64), V64) <= 1e-5


def test_weight_in_subspace_stays_there(sn):
    rng = np.random.default_rng(11)
    d, k, n = 1024, 20, 700
    U = W_.orthonormal_basis(d, k, rng)
    W = torch.tensor((U @ rng.standard_normal((k, n))).astype(np.float32), device="cuda")
    M = torch.zeros_like(W)
    V = torch.zeros_like(W)
    Ut = torch.tensor(U, device="cuda")
    for t in range(1, 6):
        g = torch.tensor((U @ rng.standard_normal((k, n))).astype(np.float32), device="cuda")
        sn.sn_adamw_rowconst(W, g, M, V, t, 1e-2, 0.9, 0.99, 1e-8, 1e-3)
    Wd = W.double()
    out = Wd - Ut @ (Ut.t() @ Wd)
    assert float(out.norm() / Wd.norm()) <= 1e-5


def test_adamw_argument_errors(sn):
    W = torch.zeros(64, 32, device="cuda")
    M = torch.zeros_like(W)
    V = torch.zeros_like(W)
    g = torch.zeros_like(W)
    with pytest.raises(sn.SNError) as e:
        sn.sn_adamw_rowconst(W, g, M, V, 0, 1e-3)             # steps count from 1
    assert e.value.status == sn.SN_ERR_INVALID_ARG
    with pytest.raises(sn.SNError) as e:
        sn.sn_adamw_rowconst(W, g, M, M, 1, 1e-3)             # V overlapping M
    assert e.value.status == sn.SN_ERR_INVALID_ARG
    with pytest.raises(sn.SNError) as e:
        sn.sn_adamw_rowconst(W, g, M, V, 1, 1e-3, workspace=torch.empty(4, device="cuda"))
    assert e.value.status == sn.SN_ERR_INVALID_ARG


@pytest.mark.parametrize("rows,cols", [(16 * 65535 + 37, 4), (16 * 65535 + 5, 1), (17, 1028), (9, 1024)])
def test_row_blocks(sn, rows, cols):
    """More runs of 16 and 8 rows than a grid's y extent holds, and a few rows: one step
    against the definition in fp64.  M and V carry one rounding; W's rate comes from
    fp32 column sums, whose error of about 1e-6 moves W by that part of a 1e-3 step."""
    g = torch.Generator(device="cuda").manual_seed(rows)
    W, M, grad = (torch.randn(rows, cols, generator=g, device="cuda") for _ in range(3))
    V = torch.rand(rows, cols, generator=g, device="cuda")
    M64 = 0.9 * M.double() + 0.1 * grad.double()
    V64 = 0.95 * V.double() + 0.05 * grad.double() ** 2
    rate = (V64.mean(0) / (1 - 0.95 ** 2)).sqrt() + 1e-8
    W64 = W.double() - 1e-3 * (M64 / (1 - 0.9 ** 2)) / rate - 1e-4 * W.double()
    sn.sn_adamw_rowconst(W, grad, M, V, 2, 1e-3, 0.9, 0.95, 1e-8, 1e-4)
    for got, want in ((W, W64), (M, M64), (V, V64)):
        assert float((got.double() - want).norm() / want.norm()) <= 1e-6


@pytest.mark.parametrize("cols", [4, 3])
def test_column_sums_take_one_addition_per_64_rows(sn, cols):
    """Equal gradients down a column make every partial sum equal, so the sum's rounding does
    not depend on the order of arrival.  n additions of equal terms to a running sum S err
    by at most half an ulp of it each, n / 2 * 2^-24 of the final sum; 64 rows meet before
    a column takes an addition.  With beta = 0, eps = 0, lr = 1 and W = 0 the step is
    -g / sqrt(mean g^2) = -1, with half the sum's relative error."""
    rows = 1 << 20
    g = torch.tensor([1.922119140625, 1.453369140625, 1.312744140625, 1.218994140625][:cols])
    grad = g.cuda().expand(rows, cols).contiguous()
    W, M, V = (torch.zeros(rows, cols, device="cuda") for _ in range(3))
    sn.sn_adamw_rowconst(W, grad, M, V, 1, 1.0, 0.0, 0.0, 0.0, 0.0)
    bound = 0.5 * (rows / 64 / 2 + 64) * 2.0 ** -24 + 8 * 2.0 ** -24
    assert float((W.double() + 1).abs().max()) <= bound


@pytest.mark.parametrize("gdt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,cols", [(5000, 1), (4097, 2), (5, 3), (4096 + 1, 4), (2050, 5), (777, 8),
                                       (1030, 12), (511, 33), (131, 63), (65, 65), (300, 252), (129, 260)])
def test_narrow_weights(sn, gdt, rows, cols):
    """Blocks with fewer lanes along the columns, at both sides of their row runs' ends: the
    step against the definition in fp64, bars as in test_row_blocks."""
    g = torch.Generator(device="cuda").manual_seed(rows)
    W, M, grad = (torch.randn(rows, cols, generator=g, device="cuda") for _ in range(3))
    V = torch.rand(rows, cols, generator=g, device="cuda")
    grad = grad.to(gdt)
    M64 = 0.9 * M.double() + 0.1 * grad.double()
    V64 = 0.95 * V.double() + 0.05 * grad.double() ** 2
    rate = (V64.mean(0) / (1 - 0.95 ** 2)).sqrt() + 1e-8
    W64 = W.double() - 1e-3 * (M64 / (1 - 0.9 ** 2)) / rate - 1e-4 * W.double()
    sn.sn_adamw_rowconst(W, grad, M, V, 2, 1e-3, 0.9, 0.95, 1e-8, 1e-4)
    for got, want in ((W, W64), (M, M64), (V, V64)):
        assert float((got.double() - want).norm() / want.norm()) <= 1e-6


@pytest.mark.parametrize("cols", [4, 1])
def test_a_narrow_weight_costs_like_a_wide_one(sn, cols):
    """As many elements in a few columns: every thread of a block has rows to work on, so the
    step takes less than ten times as long as the same number of elements in 1024 columns
    (a block with one busy thread in 256 takes thirty times as long)."""
    def fastest(rows, cols):
        W, grad, M, V = (torch.rand(rows, cols, device="cuda") for _ in range(4))
        ws = torch.empty(4 * cols, dtype=torch.uint8, device="cuda")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        times = []
        for _ in range(6):
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(4):
                sn.sn_adamw_rowconst(W, grad, M, V, 2, 1e-3, workspace=ws)
            ev[1].record()
            ev[1].synchronize()
            times.append(ev[0].elapsed_time(ev[1]))
        return min(times)
    assert fastest((1 << 22) // cols, cols) <= 10 * fastest(1 << 12, 1 << 10)
