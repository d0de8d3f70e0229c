"""Calls on a stream whose context has only a part of the GPU's SMs (a green context).

The Grassmann step's CTAs wait for one another, so its grid may be no larger than the SMs
that the stream's context has; with fewer a CTA owns several blocks of rows.  Bars as for
the step on the whole GPU.  The fp32 calls share a reduction among the CTAs of a cluster,
which such a context may have no place for: there they run without clusters.  Their bars:
d fp32 products summed in any order, d * 2^-24 of the sum of magnitudes."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_util import dev
from paper_2506_01260_gb300 import workloads as W
from test_grassmann_gpu import grassmann_oracle, rel

pytestmark = pytest.mark.gpu

SM_RESOURCE, DEFAULT_STREAM, NON_BLOCKING, IGNORE_COSCHEDULING = 1, 1, 1, 1


class Resource(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92),
                ("sm_count", ctypes.c_uint), ("rest", ctypes.c_ubyte * 44)]


class GreenContext:
    """`sms` SMs of the current device, and a stream of their own."""

    def __init__(self, sms, flags):
        torch.cuda.current_stream().synchronize()          # the primary context exists
        self.cu = ctypes.CDLL("libcuda.so.1")
        whole, part, n = Resource(), Resource(), ctypes.c_uint(1)
        desc, self.ctx, self.stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        self("cuDeviceGetDevResource", 0, ctypes.byref(whole), SM_RESOURCE)
        self("cuDevSmResourceSplitByCount", ctypes.byref(part), ctypes.byref(n), ctypes.byref(whole),
             None, flags, sms)
        self("cuDevResourceGenerateDesc", ctypes.byref(desc), ctypes.byref(part), 1)
        self("cuGreenCtxCreate", ctypes.byref(self.ctx), desc, 0, DEFAULT_STREAM)
        self("cuGreenCtxStreamCreate", ctypes.byref(self.stream), self.ctx, NON_BLOCKING, 0)
        self.sms, self.all = part.sm_count, whole.sm_count

    def __call__(self, name, *args):
        status = getattr(self.cu, name)(*args)
        assert status == 0, "%s returned %d" % (name, status)

    def synchronize(self):
        self("cuStreamSynchronize", self.stream)

    def destroy(self):
        self("cuStreamDestroy_v2", self.stream)
        self("cuGreenCtxDestroy", self.ctx)


@pytest.fixture(params=[(16, 0), (2, IGNORE_COSCHEDULING)], ids=["16 SMs", "any 2 SMs"])
def green(sn, request):
    g = GreenContext(*request.param)
    yield g
    g.destroy()


@pytest.mark.parametrize("d,k", [(2048, 20), (4104, 89)])
def test_step_on_part_of_the_sms(sn, green, d, k):
    assert green.sms < min(green.all, d // 64)             # fewer SMs than blocks of 64 rows
    o = grassmann_oracle()
    rng = np.random.default_rng(d + k)
    U32 = W.orthonormal_basis(d, k, rng).astype(np.float32)
    M32 = rng.standard_normal((d, k)).astype(np.float32)
    eta = 0.1 / (2.0 * np.linalg.norm(M32.astype(np.float64), 2))
    basis = sn.Basis(dev(U32))
    M, out = dev(M32), torch.empty(d, k, device="cuda")
    ws = torch.empty(sn.sn_grassmann_workspace(basis, 1)[1], dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    sn.sn_grassmann_step(basis, M, 1, eta, out=out, workspace=ws, stream=green.stream.value)
    green.synchronize()
    sn.sn_check_errors(basis)
    got = out.cpu().numpy().astype(np.float64)
    assert rel(got, o.step(U32.astype(np.float64), M32.astype(np.float64), 1, eta)) <= 1e-4
    assert np.max(np.abs(got.T @ got - np.eye(k))) <= 1e-5
    basis.destroy()


def test_fp32_reductions_on_part_of_the_sms(sn, green):
    T, d, k, cols = 40, 2048, 20, 200                      # a few tiles: clusters on the whole GPU
    g = torch.Generator().manual_seed(5)
    U = torch.linalg.qr(torch.randn(d, k, generator=g, dtype=torch.float64))[0].float().contiguous().cuda()
    X, Wt = torch.randn(T, d, generator=g).cuda(), torch.randn(d, cols, generator=g).cuda()
    tok, ids = torch.randn(50, d, generator=g).cuda(), torch.randint(50, (T,), generator=g).int().cuda()
    basis = sn.Basis(U)
    Cf, Cb, Wo = torch.empty(T, k, device="cuda"), torch.empty(T, k, device="cuda"), torch.empty_like(Wt)
    ws = torch.empty(sn.sn_project_weight_workspace(basis, torch.float32, cols), dtype=torch.uint8,
                     device="cuda")
    torch.cuda.synchronize()
    s = green.stream.value
    sn.sn_compress_fwd(basis, X, ids, tok, T, out=Cf, stream=s)
    sn.sn_compress_bwd(basis, X, out=Cb, stream=s)
    sn.sn_project_weight(basis, Wt, out=Wo, workspace=ws, stream=s)
    green.synchronize()
    sn.sn_check_errors(basis)
    U64, W64, R64 = U.double(), Wt.double(), X.double() - tok[ids.long()].double()
    A = U64.abs().T @ W64.abs()
    for got, want, size in ((Cb, X.double() @ U64, X.double().abs() @ U64.abs()),
                            (Cf, R64 @ U64, (R64.abs() + X.double().abs()) @ U64.abs()),
                            (Wo, U64 @ (U64.T @ W64), 2 * U64.abs() @ A)):
        assert ((got.double() - want).abs() <= d * 2.0 ** -24 * size).all()
    basis.destroy()
