"""The BF16 unary table at the edges of its tiles and runs of model tiles (grids of one tile up to several turns of the
chip), and beyond the staged width: against the same expansion of BF16-rounded rows in FP64."""
import numpy as np
import pytest

from oracle.mlp import bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,S,F", [(3, 1, 1), (31, 33, 15), (127, 128, 16), (128, 129, 162), (129, 257, 176),
                                   (700, 3000, 162), (1500, 6001, 40), (300, 40000, 64), (40, 500, 256), (40, 500, 300)])
def test_bf16_tile_edges(M, S, F):
    torch = pytest.importorskip("torch")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    rng = np.random.default_rng(M + S + F)
    fm, fs = (rng.normal(size=(n, F)).astype(np.float32) for n in (M, S))
    model = hgm.Model(rng.random((M, 2), np.float32), np.sort(rng.integers(0, 9, M)).astype(np.int32), fm)
    scene = hgm.Scene(rng.random((S, 2), np.float32), np.sort(rng.integers(0, 9, S)).astype(np.int32), fs)
    out = torch.full((M, S), -1.0, device="cuda")
    hgm.unary_bf16(model, scene, 0.6, out)
    got = out.cpu().numpy()
    a, b = bf16(fm), bf16(fs)
    na, nb = (a * a).sum(1)[:, None], (b * b).sum(1)[None]
    d2 = np.maximum(na + nb - 2.0 * a @ b.T, 0.0)
    # FP32 norms and products: each of the three terms is off by at most F 2^-24 of its magnitude, twice that here
    err2 = 2.0 * F * 2.0 ** -24 * (na + nb + 2.0 * np.abs(a) @ np.abs(b).T) + 1e-30
    lo, hi = 0.6 * np.sqrt(np.maximum(d2 - err2, 0.0)), 0.6 * np.sqrt(d2 + err2)
    assert (got >= lo * (1 - 1e-6)).all() and (got <= hi * (1 + 1e-6)).all()
