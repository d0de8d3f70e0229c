"""The calls whose speed counts: what a training program asks of this library, as cases that can
be timed one by one.

A case is one pass through the public entry points of `paper_2506_01260_gb300.sn` the way a
program calls them: the tables, the basis handle, the workspaces and the output buffers are
made once (`prepare`), the calls are made for every batch (`run`).  `work` counts the bytes and
operations a pass cannot do without, `exact` gives its results in 64 bits from plain torch, and
`draw` makes further cases of the same ranges.
"""
import math

import torch

from paper_2506_01260_gb300 import sn

QFORMATS = ("int8", "e4m3")
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
ADAMW = dict(lr=1e-4, beta1=0.9, beta2=0.95, eps=1e-8, lam=1e-5)


def listed():
    return [
        # One pipeline boundary, both directions (compress and reconstruct the activations, compress
        # and recover their gradients).  The smallest model of the tests: latency and launches.
        _boundary("boundary_tiny_bf16", 2, 128, 256, 8, 1024),
        # The same for a micro-batch of a 1B-class model.
        _boundary("boundary_1b_bf16", 8, 1024, 2048, 20, 32000),
        # A micro-batch of an 8B-class model (uniform ids: every gathered row is a new one).
        _boundary("boundary_8b_bf16", 4, 4096, 4096, 41, 128256),
        # The large stream: 65536 tokens, d = 8192, Zipf ids as in text.
        _boundary("boundary_stream_bf16", 16, 4096, 8192, 82, 128256, ids="zipf", noise=0.05),
        # Documents packed into one row of tokens, positions restarting at each (so they come as
        # an array), and sizes that fill no tile: T, d and k are all ragged.
        _boundary("boundary_packed_bf16", 1, 4173, 2056, 33, 32000, pos="packed", ctx=1024,
                  ids="zipf"),
        # The fp32 path at the 1B class: runs that must not round the wire to 16 bits.
        _boundary("boundary_1b_f32", 8, 1024, 2048, 20, 32000, dtype="f32"),
        # Projection of the residual-writing weights onto S, every iteration: attention output
        # and MLP output of an 8B-class layer; the 1B class in fp32.
        _project("project_8b_bf16", 4096, 41, 4096, 14336),
        _project("project_1b_f32", 2048, 20, 2048, 8192, dtype="f32"),
        # The forward compress from tables that were projected once per basis.
        _boundary("projected_8b_bf16", 4, 4096, 4096, 41, 128256, kind="projected"),
        # The subspace update at the end of a window: the last accumulation and its residual,
        # then the step on the Grassmann manifold.
        {"name": "subspace_8b", "kind": "subspace", "T": 16384, "d": 4096, "k": 41},
        # The row-constant AdamW step on the MLP output weight of an 8B-class layer.
        {"name": "adamw_8b", "kind": "adamw", "rows": 4096, "cols": 14336, "grad": "bf16"},
        # The lossy comparators at the codec's wire size (top-k of k / 2) and their other rates.
        {"name": "lossy_8b", "kind": "lossy", "T": 16384, "d": 4096, "kk": 20},
    ]


def _boundary(name, batch, n, d, k, vocab, dtype="bf16", ids="uniform", pos="implicit", ctx=0,
              noise=0.0, kind="boundary"):
    """`n` tokens a sequence; `ctx`: rows of the positional table where positions are packed."""
    return {"name": name, "kind": kind, "batch": batch, "n": n, "d": d, "k": k, "vocab": vocab,
            "dtype": dtype, "ids": ids, "pos": pos, "ctx": ctx or n, "noise": noise}


def _project(name, d, k, cols, cols2, dtype="bf16", pad=0):
    """Two weights [d, cols] and [d, cols2]; `pad`: unused columns at the end of their rows."""
    return {"name": name, "kind": "project", "d": d, "k": k, "cols": cols, "cols2": cols2,
            "dtype": dtype, "pad": pad}


# ---- more cases of the same ranges ---------------------------------------------------

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A model width: mostly a multiple of 128, sometimes only of 8."""
    d = _log(rng, lo, hi)
    step = 128 if rng.random() < 0.6 and d >= 256 else 8
    return max(lo, d // step * step)


def _rank(rng, d):
    return max(1, min(128, d, int(round(d * rng.uniform(0.005, 0.02)))))


def draw(rng):
    kind = rng.choice(["boundary", "boundary", "boundary", "boundary_f32", "project", "project_f32",
                       "projected", "subspace", "adamw", "lossy"])
    if kind in ("boundary", "boundary_f32", "projected"):
        f32 = kind == "boundary_f32"
        d = _width(rng, 256, 4096 if f32 else 8192)
        most = (1 << 24) if f32 else (1 << 29)              # elements of X
        T = _log(rng, 64, min(65536, most // d))
        pos = rng.choice(["implicit", "implicit", "packed", "none"])
        n = T
        if pos == "implicit":                                 # whole sequences, of any length
            n = rng.choice([128, 512, 1024, 2048, 4096, rng.randrange(50, 3000)])
            n = min(n, T)
        batch = max(1, T // n)
        c = _boundary("", batch, n, d, _rank(rng, d), rng.choice([1024, 32000, 50257, 128256]),
                      dtype="f32" if f32 else "bf16", ids=rng.choice(["uniform", "zipf"]), pos=pos,
                      ctx=rng.choice([256, 1024, 4096]) if pos == "packed" else 0,
                      noise=rng.choice([0.0, 0.05]), kind="projected" if kind == "projected" else "boundary")
    elif kind in ("project", "project_f32"):
        f32 = kind == "project_f32"
        d = _width(rng, 256, 2048 if f32 else 8192)
        cols = _log(rng, 64, min(16384, (1 << 23 if f32 else 1 << 26) // d))
        cols2 = _log(rng, 64, min(16384, (1 << 23 if f32 else 1 << 26) // d))
        if rng.random() < 0.6:
            cols, cols2 = (max(64, c // 64 * 64) for c in (cols, cols2))
        c = _project("", d, _rank(rng, d), cols, cols2, dtype="f32" if f32 else "bf16",
                     pad=rng.choice([0, 0, 24]))
    elif kind == "subspace":
        d = _width(rng, 256, 8192)
        c = {"kind": kind, "T": _log(rng, 256, min(65536, (1 << 28) // d)), "d": d,
             "k": _rank(rng, d)}
    elif kind == "adamw":
        rows = _log(rng, 256, 8192)
        cols = _log(rng, 256, 14336)
        c = {"kind": kind, "rows": rows, "cols": cols if rng.random() < 0.3 else cols // 8 * 8,
             "grad": rng.choice(["bf16", "f32"])}
    else:
        d = _width(rng, 256, 8192)
        c = {"kind": kind, "T": _log(rng, 64, min(65536, (1 << 27) // d)), "d": d,
             "kk": max(1, _rank(rng, d) // 2)}
    c.pop("name", None)
    return c


# ---- inputs --------------------------------------------------------------------------------

def _basis(d, k, g):
    """U [d, k] fp32: the orthonormal factor of a Gaussian matrix (diag(R) > 0)."""
    q = _qr(torch.randn(d, k, generator=g, device="cuda", dtype=torch.float64))
    return q.float().contiguous()


def _qr(a):
    """The orthonormal factor of `a` with diag(R) > 0, factored on the host."""
    q, r = torch.linalg.qr(a.cpu())
    s = torch.sign(torch.diagonal(r))
    return (q * torch.where(s == 0, torch.ones_like(s), s)).cuda()


def _ids(case, T, g):
    vocab = case["vocab"]
    if case["ids"] == "uniform":
        return torch.randint(vocab, (T,), generator=g, device="cuda", dtype=torch.int32)
    p = torch.arange(1, vocab + 1, device="cuda", dtype=torch.float64) ** -1.1
    ranks = torch.multinomial(p, T, replacement=True, generator=g)
    return torch.randperm(vocab, generator=g, device="cuda")[ranks].int()


def _packed_positions(T, ctx, seed):
    """Positions of documents of random lengths (at most `ctx`) packed one after another."""
    g = torch.Generator().manual_seed(seed)
    parts, left = [], T
    while left > 0:
        n = min(left, int(torch.randint(max(1, ctx // 16), ctx + 1, (1,), generator=g)))
        parts.append(torch.arange(n, dtype=torch.int32))
        left -= n
    return torch.cat(parts).cuda()


def _boundary_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    T, d, k, dt = case["batch"] * case["n"], case["d"], case["k"], DTYPES[case["dtype"]]
    s = {"U": _basis(d, k, g), "seq_len": case["ctx"]}
    s["tok"] = torch.randn(case["vocab"], d, generator=g, device="cuda", dtype=dt).mul_(0.02)
    s["pe"] = None
    if case["pos"] != "none":
        s["pe"] = torch.randn(case["ctx"], d, generator=g, device="cuda", dtype=dt).mul_(0.02)
    s["ids"] = _ids(case, T, g)
    s["pos"] = _packed_positions(T, case["ctx"], seed) if case["pos"] == "packed" else None
    # X: embeddings, a part in the subspace and a little (or `noise` of the energy) outside it
    s["X"] = torch.empty(T, d, device="cuda", dtype=dt)
    off = math.sqrt(case["noise"] / (1 - case["noise"]) * k / d) if case["noise"] else 1e-3
    for t0 in range(0, T, 8192):
        t1 = min(T, t0 + 8192)
        x = torch.randn(t1 - t0, k, generator=g, device="cuda") @ s["U"].T
        x += off * torch.randn(t1 - t0, d, generator=g, device="cuda")
        x += _embeddings(s, t0, t1, torch.float32)
        s["X"][t0:t1] = x.to(dt)
    if case["kind"] == "boundary":
        s["G"] = torch.randn(T, d, generator=g, device="cuda", dtype=dt)
        s["C_in"] = torch.randn(T, k, generator=g, device="cuda", dtype=dt)    # from the wire
        s["Cg_in"] = torch.randn(T, k, generator=g, device="cuda", dtype=dt)
    return s


def _embeddings(s, t0, t1, dt):
    e = s["tok"][s["ids"][t0:t1].long()].to(dt)
    if s["pe"] is not None:
        if s["pos"] is not None:
            p = s["pos"][t0:t1].long()
        else:
            p = torch.arange(t0, t1, device="cuda") % s["seq_len"]
        e = e + s["pe"][p].to(dt)
    return e


def _project_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    d, dt = case["d"], DTYPES[case["dtype"]]
    s = {"U": _basis(d, case["k"], g)}
    for name in ("cols", "cols2"):
        ld = (case[name] + 7) // 8 * 8 + case["pad"]
        w = torch.randn(d, ld, generator=g, device="cuda", dtype=dt).mul_(0.02)
        s[name] = w[:, :case[name]]
    return s


def _subspace_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    T, d, k = case["T"], case["d"], case["k"]
    s = {"U": _basis(d, k, g)}
    s["G"] = torch.randn(T, d, generator=g, device="cuda", dtype=torch.bfloat16)
    s["Cg"] = (s["G"].float() @ s["U"]).bfloat16()
    s["eta"] = 0.05 / T                                     # a step of a few hundredths
    return s


def _adamw_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["rows"], case["cols"])
    s = {"W": torch.randn(*shape, generator=g, device="cuda").mul_(0.02),
         "M": torch.randn(*shape, generator=g, device="cuda").mul_(1e-3),
         "V": torch.randn(*shape, generator=g, device="cuda").mul_(1e-3).square_()}
    s["grad"] = torch.randn(*shape, generator=g, device="cuda").mul_(1e-3).to(DTYPES[case["grad"]])
    return s


def _lossy_inputs(case, seed):
    """A batch as the boundary sees it: unit variance, a few channels much larger."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(case["T"], case["d"], generator=g, device="cuda")
    big = torch.rand(case["d"], generator=g, device="cuda") < 0.01
    return {"X": torch.where(big, 4 * x, x).bfloat16()}


_INPUTS = {"boundary": _boundary_inputs, "projected": _boundary_inputs, "project": _project_inputs,
           "subspace": _subspace_inputs, "adamw": _adamw_inputs, "lossy": _lossy_inputs}


def prepare(case, seed):
    kind = case["kind"]
    s = _INPUTS[kind](case, seed)
    s["kind"] = kind
    if "U" in s:
        s["basis"] = sn.Basis(s["U"])
    if kind == "boundary":
        s["C"], s["Cg"] = torch.empty_like(s["C_in"]), torch.empty_like(s["Cg_in"])
        s["X_out"], s["G_out"] = torch.empty_like(s["X"]), torch.empty_like(s["G"])
    elif kind == "projected":
        s["TU"], s["PU"] = sn.sn_project_tables(s["basis"], s["tok"], pos_emb=s["pe"])
        s["C"] = torch.empty(s["X"].shape[0], case["k"], device="cuda", dtype=s["X"].dtype)
    elif kind == "project":
        for name in ("cols", "cols2"):
            w = s[name]
            s[name + "_out"] = torch.empty(w.shape[0], w.stride(0), device="cuda",
                                           dtype=w.dtype)[:, :w.shape[1]]
            n = sn.sn_project_weight_workspace(s["basis"], w.dtype, w.shape[1])
            s[name + "_ws"] = torch.empty(max(16, n), device="cuda", dtype=torch.uint8)
    elif kind == "subspace":
        a, b = sn.sn_grassmann_workspace(s["basis"], case["T"])
        s["ws"] = torch.empty(max(256, a, b), device="cuda", dtype=torch.uint8)
        s["M"] = torch.zeros(case["d"], case["k"], device="cuda")
        s["acc"] = torch.zeros(1, device="cuda", dtype=torch.float64)
        s["U_new"] = torch.empty_like(s["M"])
    elif kind == "adamw":
        s["ws"] = torch.empty(case["cols"], device="cuda")
    elif kind == "lossy":
        s["d"], s["kk"] = case["d"], case["kk"]
    return s


# ---- one pass --------------------------------------------------------------------------------

def run(s):
    return _RUN[s["kind"]](s)


def _run_boundary(s):
    b, n, pe, pos = s["basis"], s["seq_len"], s["pe"], s["pos"]
    C = sn.sn_compress_fwd(b, s["X"], s["ids"], s["tok"], n, pos_emb=pe, pos=pos, out=s["C"])
    X = sn.sn_decompress_fwd(b, s["C_in"], s["ids"], s["tok"], n, pos_emb=pe, pos=pos,
                             out=s["X_out"])
    Cg = sn.sn_compress_bwd(b, s["G"], out=s["Cg"])
    G = sn.sn_decompress_bwd(b, s["Cg_in"], out=s["G_out"])
    return {"C": C, "X": X, "Cg": Cg, "G": G}


def _run_projected(s):
    return {"C": sn.sn_compress_fwd_projected(s["basis"], s["X"], s["ids"], s["TU"], s["seq_len"],
                                              PU=s["PU"], pos=s["pos"], out=s["C"])}


def _run_project(s):
    return {name: sn.sn_project_weight(s["basis"], s[name], out=s[name + "_out"],
                                       workspace=s[name + "_ws"])
            for name in ("cols", "cols2")}


def _run_subspace(s):
    b, G, Cg = s["basis"], s["G"], s["Cg"]
    M, acc = s["M"].zero_(), s["acc"].zero_()
    sn.sn_grassmann_accumulate(b, G, Cg, M, workspace=s["ws"])
    sn.sn_grassmann_residual(b, G, Cg, acc)
    U = sn.sn_grassmann_step(b, M, 1, s["eta"], out=s["U_new"], workspace=s["ws"])
    return {"M": M, "acc": acc, "U": U}


def _run_adamw(s):
    sn.sn_adamw_rowconst(s["W"], s["grad"], s["M"], s["V"], 100, workspace=s["ws"], **ADAMW)
    return {"W": s["W"], "M": s["M"], "V": s["V"]}


def _run_lossy(s):
    X, d = s["X"], s["d"]
    vals, cols = sn.sn_topk_compress(X, s["kk"])
    out = {"vals": vals, "cols": cols, "topk": sn.sn_topk_restore(vals, cols, d)}
    bits, scale = sn.sn_sign_compress(X)
    out.update(bits=bits, scale=scale, sign=sn.sn_sign_restore(bits, scale, d))
    for f in QFORMATS:
        codes, scale = sn.sn_quant_compress(X, f)
        out[f] = {"codes": codes, "scale": scale, "X": sn.sn_quant_restore(codes, scale, f)}
    return out


_RUN = {"boundary": _run_boundary, "projected": _run_projected, "project": _run_project,
        "subspace": _run_subspace, "adamw": _run_adamw, "lossy": _run_lossy}


# ---- what a pass cannot do without -----------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("boundary", "projected"):
        T, d, k = case["batch"] * case["n"], case["d"], case["k"]
        es = 2 if case["dtype"] == "bf16" else 4
        u = _expected_unique(case, T)                       # rows of the token table read
        n = 0 if case["pos"] == "none" else min(case["ctx"], T)
        if kind == "projected":
            return {"bytes": es * T * (d + k) + 4 * (u + n + d) * k + 4 * T, "flops": 2 * T * d * k}
        one = es * T * (d + k) + 4 * d * k
        fwd = one + es * (u + n) * d + 4 * T * (2 if case["pos"] == "packed" else 1)
        return {"bytes": 2 * fwd + 2 * one, "flops": 8 * T * d * k}
    if kind == "project":
        d, k, cols = case["d"], case["k"], case["cols"] + case["cols2"]
        es = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": 2 * es * d * cols + 2 * 4 * d * k, "flops": 4 * d * k * cols}
    if kind == "subspace":
        T, d, k = case["T"], case["d"], case["k"]
        return {"bytes": 2 * T * (d + k) + 4 * 3 * d * k, "flops": 2 * T * d * k + 12 * d * k * k}
    if kind == "adamw":
        n = case["rows"] * case["cols"]
        return {"bytes": n * (24 + (2 if case["grad"] == "bf16" else 4)), "flops": 14 * n}
    T, d, kk = case["T"], case["d"], case["kk"]
    x = 2 * T * d
    topk = 2 * x + 2 * 4 * T * kk
    sign = 2 * x + 2 * (4 * T * ((d + 31) // 32) + 4 * T)
    quant = 2 * x + 2 * (T * d + 4 * T)
    return {"bytes": topk + sign + 2 * quant, "flops": 16 * T * d}


def _expected_unique(case, T):
    vocab = case["vocab"]
    if case["ids"] == "uniform":
        return int(vocab * (1 - (1 - 1 / vocab) ** T))
    w = [(r + 1) ** -1.1 for r in range(vocab)]
    z = sum(w)
    return int(sum(1 - (1 - x / z) ** T for x in w))


# ---- the results in 64 bits --------------------------------------------------------------------

def exact(case, seed):
    s = _INPUTS[case["kind"]](case, seed)
    return _EXACT[case["kind"]](case, s)


def _exact_compress(s, X, U, embeddings):
    C = torch.empty(X.shape[0], U.shape[1], device="cuda", dtype=torch.float64)
    for t0 in range(0, X.shape[0], 8192):
        t1 = min(X.shape[0], t0 + 8192)
        r = X[t0:t1].double()
        if embeddings:
            r -= _embeddings(s, t0, t1, torch.float64)
        C[t0:t1] = r @ U
    return C


def _exact_boundary(case, s):
    U = s["U"].double()
    C = _exact_compress(s, s["X"], U, True)
    if case["kind"] == "projected":
        return {"C": C}
    X = s["C_in"].double() @ U.T
    for t0 in range(0, X.shape[0], 8192):
        t1 = min(X.shape[0], t0 + 8192)
        X[t0:t1] += _embeddings(s, t0, t1, torch.float64)
    return {"C": C, "X": X, "Cg": _exact_compress(s, s["G"], U, False),
            "G": s["Cg_in"].double() @ U.T}


def _exact_project(case, s):
    U = s["U"].double()
    return {name: U @ (U.T @ s[name].double()) for name in ("cols", "cols2")}


def _exact_subspace(case, s):
    U, G, Cg = s["U"].double(), s["G"], s["Cg"].double()
    M = torch.zeros(U.shape, device="cuda", dtype=torch.float64)
    sq = torch.zeros((), device="cuda", dtype=torch.float64)
    for t0 in range(0, G.shape[0], 8192):
        g = G[t0:t0 + 8192].double()
        M += g.T @ Cg[t0:t0 + 8192]
        sq += g.square().sum()
    grad = -2 * M
    return {"M": M, "acc": (sq - Cg.square().sum()).reshape(1),
            "U": _qr(U - s["eta"] * (grad - U @ (U.T @ grad)))}


def _exact_adamw(case, s):
    h, t = ADAMW, 100
    g = s["grad"].double()
    M = h["beta1"] * s["M"].double() + (1 - h["beta1"]) * g
    V = h["beta2"] * s["V"].double() + (1 - h["beta2"]) * g * g
    rate = (V.mean(0) / (1 - h["beta2"] ** t)).sqrt() + h["eps"]
    W = s["W"].double()
    W = W - h["lr"] * (M / (1 - h["beta1"] ** t)) / rate - h["lam"] * W
    return {"W": W, "M": M, "V": V}


def _exact_lossy(case, s):
    x = s["X"].double()
    mag = x.abs()
    cols = torch.sort(mag, dim=1, descending=True, stable=True)[1][:, :case["kk"]]
    cols = torch.sort(cols, dim=1)[0]
    vals = x.gather(1, cols)
    mean = mag.mean(1)
    out = {"vals": vals, "cols": None, "topk": torch.zeros_like(x).scatter_(1, cols, vals),
           "bits": None, "scale": mean,
           "sign": torch.where(x < 0, -mean[:, None], mean[:, None])}
    for f, qmax in zip(QFORMATS, (127.0, 448.0)):
        # the restored values hang on the codes, which are decided in fp32
        out[f] = {"codes": None, "scale": mag.amax(1) / qmax, "X": None}
    return out


_EXACT = {"boundary": _exact_boundary, "projected": _exact_boundary, "project": _exact_project,
          "subspace": _exact_subspace, "adamw": _exact_adamw, "lossy": _exact_lossy}
