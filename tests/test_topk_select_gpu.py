"""Top-k selection where its two searches start or end early: rows of one key, keys that
differ only in their last bits, all zero, one large entry, more candidates than lanes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rows(kind, T, d, rng):
    sign = rng.integers(0, 2, (T, d)).astype(np.uint16) << 15
    if kind == "one key":
        key = np.full((T, d), 0x3F80)
    elif kind == "last bits":
        key = 0x3F80 + rng.integers(0, 4, (T, d))
    elif kind == "zero":
        key = np.zeros((T, d))
    elif kind == "spike":
        key = np.zeros((T, d))
        key[np.arange(T), rng.integers(0, d, T)] = 0x7F7F
    else:                                       # every exponent
        key = rng.integers(0, 0x7F80, (T, d))
    return sign | key.astype(np.uint16)


@pytest.mark.parametrize("d,kk", [(8, 1), (64, 33), (512, 24), (520, 70), (4096, 20), (4096, 96),
                                  (1024, 200)])
@pytest.mark.parametrize("kind", ["one key", "last bits", "zero", "spike", "all"])
def test_kept_entries(sn, kind, d, kk):
    kk = min(kk, d)
    x = rows(kind, 67, d, np.random.default_rng(d + kk))
    key = (x & 0x7FFF).astype(np.int64)
    order = np.argsort(-key, axis=1, kind="stable")[:, :kk]     # largest first, lowest column of equals
    want = np.sort(order, axis=1)
    vals, cols = sn.sn_topk_compress(torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16), kk)
    assert np.array_equal(cols.cpu().view(torch.int16).numpy().view(np.uint16).astype(np.int64), want)
    assert np.array_equal(vals.view(torch.int16).cpu().numpy().view(np.uint16),
                          np.take_along_axis(x, want, axis=1))
