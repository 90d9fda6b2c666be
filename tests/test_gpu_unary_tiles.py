"""The FP32 unary table at the edges of its two tile shapes and of its component stages: bit-identical to the
fixed-order sum it is defined as (d = a - b, s = fma(d, d, s), IEEE square root, times lambda1), computed here in
FP64 with one rounding per operation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _table(a, b, lam):
    """FP32 results of each step: a product of two FP32 values and a sum are exact enough in FP64 to round once
    (24 + 24 bits of product, aligned sums beyond 53 bits only where the addend is negligible)."""
    s = np.zeros((a.shape[0], b.shape[0]), np.float32)
    for k in range(a.shape[1]):
        d = a[:, None, k] - b[None, :, k]
        s = (d.astype(np.float64) * d + s).astype(np.float32)
    return np.float32(lam) * np.sqrt(s)


@pytest.mark.parametrize("M,S,F", [(3, 1, 1), (16, 32, 4), (17, 33, 31), (15, 31, 32), (5, 600, 33), (40, 300, 162),
                                   (33, 129, 200), (64, 20001, 162), (65, 40000, 37), (32, 38912, 64)])
def test_unary_tile_edges(M, S, F):
    torch = pytest.importorskip("torch")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    rng = np.random.default_rng(M * S + F)
    fm, fs = (rng.normal(size=(n, F)).astype(np.float32) for n in (M, S))
    tm, ts = (np.sort(rng.integers(0, 9, n)).astype(np.int32) for n in (M, S))
    model = hgm.Model(rng.random((M, 2), np.float32), tm, fm)
    scene = hgm.Scene(rng.random((S, 2), np.float32), ts, fs)
    out = torch.full((M, S), -1.0, device="cuda")
    hgm.unary(model, scene, 0.6, out)
    got = out.cpu().numpy()
    cols = np.unique(np.concatenate([np.arange(min(S, 300)), np.arange(max(0, S - 300), S), rng.integers(0, S, 200)]))
    want = _table(fm, fs[cols], 0.6)
    # double rounding of the FP64 emulation can move a step by one unit in the last place in rare cases
    assert np.max(np.abs(got[:, cols] - want)) <= 2 * np.max(np.spacing(want))
    assert np.mean(got[:, cols] == want) >= 0.999
    assert (got >= 0).all()
