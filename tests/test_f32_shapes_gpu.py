"""The fp32 kernels at the edges of their tiles, against the fp64 oracle.

The compress covers k with 4, 8, ..., 24, 32, 48, 64, 96 or 128 columns, 32 tokens
a CTA and 32 columns of d a chunk, shared out over warps and clusters of up to
8 CTAs; the expansion takes 16 rows a warp and 128 columns a CTA; the projection
128 columns a warp and 8 rows a step.  Bar: the fp32 parity bar (1e-5 relative
Frobenius error, 1e-4 on every row).  fp32 sums of d = 16 .. 1032 products differ
from the exact ones by about sqrt(d) 2^-24 of their size, 2e-6 at most, so the bar
is a missing or doubled product's, not the arithmetic's.
"""
import numpy as np
import pytest
import torch

from gpu_util import assert_parity, dev, guarded, guards_intact, host
from paper_2506_01260_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (T, seq_len, d, k, vocab): every compress width, one and many CTAs per cluster, d that
# ends inside a chunk, T around the 32- and 128-row tiles
SHAPES = [(1, 4, 16, 1, 5), (31, 8, 40, 4, 9), (32, 32, 64, 5, 50), (33, 10, 200, 8, 50),
          (127, 64, 264, 12, 50), (128, 128, 1032, 16, 200), (129, 50, 512, 17, 200),
          (65, 20, 512, 20, 200), (257, 256, 520, 21, 200), (40, 20, 512, 24, 99),
          (100, 30, 512, 25, 99), (70, 20, 512, 32, 99), (64, 64, 264, 33, 99),
          (95, 20, 512, 48, 99), (130, 20, 512, 49, 99), (50, 20, 264, 64, 99),
          (61, 20, 512, 65, 99), (97, 20, 512, 82, 99), (99, 20, 512, 97, 99),
          (5000, 700, 136, 20, 999)]


@pytest.mark.parametrize("T,n,d,k,vocab", SHAPES)
def test_f32_boundary_shapes(sn, oracle, T, n, d, k, vocab):
    wl = W.Workload("f32", 1, n, d, k, vocab, 500 + T + d + k, off_scale=1e-2, grad=True)
    inp = W.generate(wl, T=T, dtype="f32")
    basis = sn.Basis(dev(inp["U"]))
    X, tok, pe, ids, G = (dev(inp[n_]) for n_ in ("X", "tok_emb", "pos_emb", "ids", "G"))
    bufs = [guarded((T, w), X.dtype) for w in (k, d, k, d)]
    C, Xr, Cg, Gr = (b[1] for b in bufs)
    sn.sn_compress_fwd(basis, X, ids, tok, n, pos_emb=pe, out=C)
    sn.sn_decompress_fwd(basis, C, ids, tok, n, pos_emb=pe, out=Xr)
    sn.sn_compress_bwd(basis, G, out=Cg)
    sn.sn_decompress_bwd(basis, Cg, out=Gr)
    sn.sn_check_errors(basis)
    assert all(guards_intact(b[0]) for b in bufs)
    U = inp["U"]
    emb = (inp["ids"], inp["tok_emb"], U, n)
    assert_parity(host(C), oracle.compress_fwd(inp["X"], *emb, pos_emb=inp["pos_emb"])[1], "f32")
    assert_parity(host(Xr), oracle.decompress_fwd(host(C), *emb, pos_emb=inp["pos_emb"])[1], "f32")
    assert_parity(host(Cg), oracle.compress_bwd(inp["G"], U)[1], "f32")
    assert_parity(host(Gr), oracle.decompress_bwd(host(Cg), U)[1], "f32")
    basis.destroy()


@pytest.mark.parametrize("d,k,cols,pad", [(16, 1, 1, 0), (40, 5, 3, 8), (200, 20, 127, 0),
                                          (520, 24, 130, 4), (264, 32, 513, 0), (72, 41, 260, 0),
                                          (520, 64, 126, 8), (136, 82, 257, 0), (1032, 128, 131, 0)])
def test_f32_projection_shapes(sn, oracle, d, k, cols, pad):
    rng = np.random.default_rng(d + k + cols)
    U = W.orthonormal_basis(d, k, rng).astype(np.float32)
    ld = (cols + 3) // 4 * 4 + pad
    Wh = (0.02 * rng.standard_normal((d, ld))).astype(np.float32)
    basis = sn.Basis(dev(U))
    full, out = guarded((d, ld), dev(Wh).dtype)
    out[:] = 7.0
    sn.sn_project_weight(basis, dev(Wh)[:, :cols], out=out[:, :cols])
    sn.sn_check_errors(basis)
    assert guards_intact(full) and bool((out[:, cols:] == 7.0).all())
    _, W64, _ = oracle.project_weight(np.ascontiguousarray(Wh[:, :cols]), U)
    assert_parity(host(out[:, :cols]), W64, "f32")
    basis.destroy()


@pytest.mark.parametrize("d,k", [(16, 1), (264, 5), (520, 20), (1000, 41), (136, 64), (2056, 127), (512, 128)])
@pytest.mark.parametrize("with_pos", [False, True])
def test_few_rows_give_the_tiles_bits(sn, d, k, with_pos):
    """Reconstruction of 4903 rows takes the tile kernel, of a few of them the one for few rows:
    one chain of sums over j in both, so the same bits; ids out of range included."""
    T, vocab, n = 4903, 50, 64
    g = torch.Generator().manual_seed(d + k)
    U = torch.linalg.qr(torch.randn(d, k, generator=g, dtype=torch.float64))[0].float().contiguous().cuda()
    C, tok, pe = (torch.randn(r, w, generator=g).cuda() for r, w in ((T, k), (vocab, d), (n, d)))
    ids = torch.randint(vocab, (T,), generator=g).int()
    pos = torch.randint(n, (T,), generator=g).int()
    ids[5], ids[4096], pos[9] = vocab, -1, n
    ids, pos = ids.cuda(), pos.cuda()
    basis = sn.Basis(U)

    def both(t0, t1):
        fwd = sn.sn_decompress_fwd(basis, C[t0:t1].clone(), ids[t0:t1].clone(), tok, n,
                                   pos_emb=pe if with_pos else None,
                                   pos=pos[t0:t1].clone() if with_pos else None)
        return fwd, sn.sn_decompress_bwd(basis, C[t0:t1].clone())
    whole = both(0, T)
    for t0, rows in ((0, 1), (3, 7), (0, 8), (4090, 9), (100, 16), (1000, 130), (4803, 100)):
        for w, f in zip(whole, both(t0, t0 + rows)):
            assert torch.equal(f, w[t0:t0 + rows])
    assert not whole[0][5].any() and not whole[0][4096].any() and bool(whole[0][6].any())
    with pytest.raises(sn.SNError):
        sn.sn_check_errors(basis)
    basis.destroy()


def test_few_rows_at_a_wide_basis_start_at_once(sn):
    """65 rows at k = 128 read sixteen times the coefficients of k = 8 but take less than twice as
    long (three times, where every CTA first copies 128 columns of U^T)."""
    T, d = 65, 1000
    tok = torch.randn(50, d, device="cuda")
    ids = torch.randint(50, (T,), device="cuda", dtype=torch.int32)

    def fastest(k):
        U = torch.linalg.qr(torch.randn(d, k, dtype=torch.float64))[0].float().contiguous().cuda()
        basis, C, out = sn.Basis(U), torch.randn(T, k, device="cuda"), torch.empty(T, d, device="cuda")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(20):
                sn.sn_decompress_fwd(basis, C, ids, tok, T, out=out)
            ev[1].record()
            ev[1].synchronize()
            times.append(ev[0].elapsed_time(ev[1]))
        basis.destroy()
        return min(times)
    assert fastest(128) <= 2 * fastest(8)
