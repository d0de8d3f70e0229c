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


@pytest.mark.parametrize("kk", [20, 41, 60, 90])
@pytest.mark.parametrize("m", [63, 64, 65, 96, 128, 129, 255, 256, 257])
def test_counts_of_candidates(sn, m, kk):
    """m entries whose keys differ in their last two bits, one in each of the first m chunks, and
    zeros: all m are candidates, few enough for one register a lane or as many as there are."""
    m, d = max(m, kk), 4096
    rng = np.random.default_rng(m + kk)
    x = np.zeros((33, d), np.uint16)
    x[:, 8 * np.arange(m) + rng.integers(0, 8, m)] = 0x4000 + rng.integers(0, 4, (33, m))
    order = np.argsort(-x.astype(np.int64), axis=1, kind="stable")[:, :kk]
    want = np.sort(order, axis=1)
    vals, cols = sn.sn_topk_compress(torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16), kk)
    assert np.array_equal(cols.cpu().view(torch.int16).numpy().view(np.uint16).astype(np.int64), want)
    assert np.array_equal(vals.view(torch.int16).cpu().numpy().view(np.uint16),
                          np.take_along_axis(x, want, axis=1))


def test_more_than_64_candidates_cost_little(sn):
    """kk = 64 of 1024 leaves about 100 candidates a row, kk = 41 about 60: the search over the
    larger number takes less than 1.3 times as long (1.43 with a vote per 32 of them)."""
    X = torch.randn(30000, 1024, generator=torch.Generator(device="cuda").manual_seed(1),
                    device="cuda").bfloat16()

    def fastest(kk):
        v, c = sn.sn_topk_compress(X, kk)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(20):
                sn.sn_topk_compress(X, kk, values=v, cols=c)
            ev[1].record()
            ev[1].synchronize()
            times.append(ev[0].elapsed_time(ev[1]))
        return min(times)
    assert fastest(64) <= 1.3 * fastest(41)
