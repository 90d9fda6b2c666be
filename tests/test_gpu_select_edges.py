"""Candidate selection at the edges of its window sizes (register-held and memory passes) and on keys that tie, crowd
or spread: the kept set is exactly the K smallest keys, equal ones in index order, as a stable sort of the unary
table's bits gives it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _descriptors(rng, n, F, kind):
    if kind == "equal":                     # one value for every key
        return np.ones((n, F), np.float32)
    f = rng.normal(size=(n, F)).astype(np.float32)
    if kind == "ties":                      # a few values, each many times
        return f[rng.integers(0, 5, n)]
    if kind == "crowded":                   # most keys within a few bits of each other, a few far away
        f = np.ones((n, F), np.float32) + np.float32(2.0 ** -20) * rng.integers(0, 3, (n, F)).astype(np.float32)
        f[rng.random(n) < 0.05] *= 1e3
        return f
    if kind == "wide":                      # keys over the whole exponent range, zeros among them
        f = np.zeros((n, F), np.float32)
        f[:, 0] = (2.0 ** rng.integers(-60, 60, n)) * (rng.random(n) < 0.9)
        return f
    return f


@pytest.mark.parametrize("kind", ["normal", "equal", "ties", "crowded", "wide"])
@pytest.mark.parametrize("K", [64, 37, 5])
def test_kept_set_is_the_stable_order(kind, K):
    torch = pytest.importorskip("torch")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    rng = np.random.default_rng(K)
    sizes = [K, K + 1, 63, 64, 65, 66, 127, 128, 129, 255, 256, 257, 400, 639, 640, 641, 1500]
    t = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    for dense in (False, True):             # the call's typical window decides which kernel runs
        if dense:
            t = np.concatenate([t, np.repeat(len(sizes), 9000).astype(np.int32)])
        S, F = len(t), 7
        fs = _descriptors(rng, S, F, kind)
        fm = np.zeros((3, F), np.float32) if kind != "normal" else rng.normal(size=(3, F)).astype(np.float32)
        model = hgm.Model(rng.random((3, 2), np.float32), np.zeros(3, np.int32), fm)
        scene = hgm.Scene(rng.random((S, 2), np.float32), t, fs)
        p = hgm.default_params(K=K, window=0)
        first, n = hgm.offsets(model, scene, p)
        U = torch.empty((3, S), device="cuda")
        hgm.unary(model, scene, 0.6, U)
        key = U.cpu().numpy()
        idx = torch.empty((n, 3, K), dtype=torch.int32, device="cuda")
        cnt = torch.empty((n, 3), dtype=torch.int32, device="cuda")
        hgm.candidates(model, scene, p, first, n, idx, cnt)
        idx, cnt = idx.cpu().numpy(), cnt.cpu().numpy()
        for o in range(n):
            lo, hi = np.searchsorted(t, [first + o, first + o + 1])
            for i in range(3):
                want = np.sort(lo + np.argsort(key[i, lo:hi], kind="stable")[:K])
                assert cnt[o, i] == len(want)
                assert np.array_equal(idx[o, i, :len(want)], want), (o, i)
                assert (idx[o, i, len(want):] == -1).all()
