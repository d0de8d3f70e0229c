"""The calls outside the boundary step captured into CUDA graphs, and two steps at once.

The Grassmann step is a cooperative launch behind a zeroed pair of barrier words, the fp32
calls launch clusters, AdamW three dependent kernels, the comparators dependent kernels:
each is captured alone, replayed twice on poisoned outputs, and gives the eager call's bits
each time.  (Shapes at which no result depends on the order of arrival: up to 64 rows for
AdamW, whose columns then take one atomic; the residual is one fp64 atomic per block, held
to 1e-12.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu


def basis(sn, d, k, seed=0):
    g = torch.Generator().manual_seed(seed)
    U = torch.linalg.qr(torch.randn(d, k, generator=g, dtype=torch.float64))[0]
    return sn.Basis(U.float().contiguous().cuda())


def rand(*shape, seed=1, dtype=torch.float32):
    return torch.randn(*shape, generator=torch.Generator().manual_seed(seed)).to(dtype).cuda()


def space(n):
    return torch.empty(max(256, n), dtype=torch.uint8, device="cuda")


def grassmann(sn, dtype):
    T, d, k = 3000, 1000, 41
    b, G, Cg = basis(sn, d, k), rand(T, d, dtype=torch.bfloat16), rand(T, k, seed=2, dtype=torch.bfloat16)
    a, s = sn.sn_grassmann_workspace(b, T)
    wa, ws = space(a), space(s)
    out = {"M": torch.empty(d, k, device="cuda"), "acc": torch.empty(1, dtype=torch.float64, device="cuda"),
           "U": torch.empty(d, k, device="cuda")}

    def run():
        out["M"].zero_()
        out["acc"].zero_()
        sn.sn_grassmann_accumulate(b, G, Cg, out["M"], workspace=wa)
        sn.sn_grassmann_residual(b, G, Cg, out["acc"])
        sn.sn_grassmann_step(b, out["M"], 1, 1e-5, out=out["U"], workspace=ws)
    return b, run, out


def fp32(sn, dtype):
    T, d, k, cols = 100, 2048, 20, 264
    b, X, Wt = basis(sn, d, k), rand(T, d), rand(d, cols, seed=2)
    tok, ids = rand(50, d, seed=3), torch.randint(50, (T,)).int().cuda()
    ws = space(sn.sn_project_weight_workspace(b, torch.float32, cols))
    out = {n: torch.empty(T, k, device="cuda") for n in ("C", "Cg")}
    out.update(X=torch.empty(T, d, device="cuda"), G=torch.empty(T, d, device="cuda"), W=torch.empty_like(Wt))

    def run():
        sn.sn_compress_fwd(b, X, ids, tok, T, out=out["C"])
        sn.sn_decompress_fwd(b, out["C"], ids, tok, T, out=out["X"])
        sn.sn_compress_bwd(b, X, out=out["Cg"])
        sn.sn_decompress_bwd(b, out["Cg"], out=out["G"])
        sn.sn_project_weight(b, Wt, out=out["W"], workspace=ws)
    return b, run, out


def adamw(sn, dtype):
    rows, cols = 64, 1000
    start = [rand(rows, cols, seed=i) for i in range(2)] + [rand(rows, cols, seed=2).square()]
    grad, ws = rand(rows, cols, seed=3, dtype=dtype), space(4 * cols)
    out = {n: torch.empty(rows, cols, device="cuda") for n in "WMV"}

    def run():
        for t, s in zip(out.values(), start):
            t.copy_(s)
        sn.sn_adamw_rowconst(out["W"], grad, out["M"], out["V"], 3, 1e-3, workspace=ws)
    return None, run, out


def lossy(sn, dtype):
    X, out = rand(200, 1000, dtype=torch.bfloat16), {}

    def run():
        out["v"], out["c"] = sn.sn_topk_compress(X, 20)
        out["Xk"] = sn.sn_topk_restore(out["v"], out["c"], 1000)
        out["b"], out["s"] = sn.sn_sign_compress(X)
        out["Xs"] = sn.sn_sign_restore(out["b"], out["s"], 1000)
        for f in ("int8", "e4m3"):
            out["q" + f], out["qs" + f] = sn.sn_quant_compress(X, f)
            out["Xq" + f] = sn.sn_quant_restore(out["q" + f], out["qs" + f], f)
    return None, run, out


def raw(t):
    return t.view(torch.uint8) if t.element_size() == 1 else t.contiguous().view(torch.uint8)


@pytest.mark.parametrize("make,dtype", [(grassmann, None), (fp32, None), (adamw, torch.float32),
                                        (adamw, torch.bfloat16), (lossy, None)])
def test_captured_calls_replay_eager_bits(sn, make, dtype):
    b, run, out = make(sn, dtype)
    run()
    torch.cuda.synchronize()
    want = {n: t.clone() for n, t in out.items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for _ in range(2):
        for t in out.values():
            raw(t).fill_(0xA5)
        graph.replay()
        torch.cuda.synchronize()
        for n, t in out.items():
            if n == "acc":
                assert abs(t.item() / want[n].item() - 1) <= 1e-12
            else:
                assert torch.equal(raw(t), raw(want[n])), n
    if b is not None:
        sn.sn_check_errors(b)
        b.destroy()


@pytest.mark.parametrize("d,k", [(1024, 20), (8192, 82)])
def test_two_steps_on_two_streams(sn, d, k):
    """Two cooperative grids, together more CTAs than SMs at the larger size, each with its
    basis, workspace and output: neither waits for the other in vain, and both give the
    bits of a step alone."""
    U = torch.linalg.qr(torch.randn(d, k, generator=torch.Generator().manual_seed(3), dtype=torch.float64))[0]
    U, M = U.float().contiguous().cuda(), rand(d, k, seed=4)
    bases = [sn.Basis(U) for _ in range(2)]
    want = sn.sn_grassmann_step(bases[0], M, 1, 1e-3)
    ws = [space(sn.sn_grassmann_workspace(b, 1)[1]) for b in bases]
    outs = [[torch.empty_like(U) for _ in range(8)] for _ in bases]
    streams = [torch.cuda.Stream() for _ in bases]
    torch.cuda.synchronize()
    for i in range(8):
        for b, w, o, s in zip(bases, ws, outs, streams):
            sn.sn_grassmann_step(b, M, 1, 1e-3, out=o[i], workspace=w, stream=s)
    torch.cuda.synchronize()
    for b, o in zip(bases, outs):
        sn.sn_check_errors(b)
        assert all(torch.equal(x, want) for x in o)
        b.destroy()
