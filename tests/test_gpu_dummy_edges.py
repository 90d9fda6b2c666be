"""The dummy-assignment recursion at the edges of its tables: caps around both table sizes and off the 4-cell tiles,
crowded and empty windows, every closeness limit, a dummy that is free, cheap and dear (beyond FP32's range too),
coincident points, a model whose tables would not fit a full grid. Against
the FP64 oracle on every offset (energies 1e-5 relative, assignments equal or of the same FP64 energy)."""
import numpy as np
import pytest

from gpu_util import check_offset
from paper_1505_00581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,lam,crowd,T,window,M,wd", [
    (3, 4.0, 0.0, 10, 1, 5, 4.0), (17, 6.0, 0.0, 10, 2, 9, 8.0), (31, 9.0, 0.2, 10, 3, 12, 3.0),
    (32, 20.0, 0.0, 4, 2, 8, 20.0), (33, 8.0, 0.1, 10, 2, 10, 5.0), (47, 20.0, 0.3, 10, 3, 7, 2.0),
    (63, 30.0, 0.0, 0, 1, 6, 12.0), (64, 4.0, 0.5, 10, 3, 11, 8.0), (64, 30.0, 0.0, 2, 3, 9, 6.0),
    (64, 0.3, 0.0, 10, 2, 20, 8.0), (61, 25.0, 0.1, 10, 2, 3, 0.0)])
def test_dummy_list_edges(K, lam, crowd, T, window, M, wd):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    import oracle
    oracle.build()
    rng = np.random.default_rng(2000 * K + M)
    mod = synth.make_model(rng, M, F=16, frame=(60.0, 40.0), t_span=10, T=max(T, 6))
    sc = synth.make_scene(rng, 24, (60.0, 40.0), ("poisson", lam), mod.centres, [mod], [(0, 2)])
    t, xy = sc.t.copy(), sc.xy.copy()
    t[rng.random(len(t)) < crowd] = 12
    xy[rng.random(len(t)) < 0.1] = (5.0, 5.0)            # several points at one position
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(xy, t, sc.f, 24)
    first, e, a = hgm.match(m, s, hgm.default_params(K=K, window=window, T=T, dummy_cost=wd))
    orc = oracle.Oracle(mod.xy, mod.t, mod.f, xy, t, sc.f, 24, K=K, window=window, T=T, lambda1=0.6, lambda2=0.2,
                        lambda3=5.0, dummy_cost=wd)
    assert np.isfinite(e).all()
    for k in range(len(e)):
        ok, _, why = check_offset(orc, first + k, e[k], a[k])
        assert ok, (first + k, why)


@pytest.mark.parametrize("K", [24, 64])
@pytest.mark.parametrize("wd", [2e38, 1e38, 3e37, 1e37])
def test_a_dummy_whose_sums_overflow_is_never_taken(K, wd):
    """lambda1 W^d, or the sums of it along a chain, beyond FP32's largest value: eps costs +inf there, and every
    offset that has a chain of real points keeps its plain optimum (of any W^d above, since one eps costs more)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    import oracle
    oracle.build()
    rng = np.random.default_rng(0)
    mod = synth.make_model(rng, 9, F=16, frame=(60.0, 40.0), t_span=10)
    sc = synth.make_scene(rng, 30, (60.0, 40.0), ("poisson", 6.0), mod.centres, [mod], [(0, 2)])
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(sc.xy, sc.t, sc.f, 30)
    first, e, a = hgm.match(m, s, hgm.default_params(K=K, window=2, lambda1=2.0, dummy_cost=wd))
    orc = oracle.Oracle(mod.xy, mod.t, mod.f, sc.xy, sc.t, sc.f, 30, K=K, window=2, T=10, lambda1=2.0, lambda2=0.2,
                        lambda3=5.0)
    feasible = 0
    for k in range(len(e)):
        if np.isfinite(orc.match(first + k)[0]):
            ok, _, why = check_offset(orc, first + k, e[k], a[k])
            assert ok, (first + k, why)
            feasible += 1
        elif 2.0 * wd > np.finfo(np.float32).max:
            assert np.isinf(e[k]) and np.all(a[k] == -1)
    assert feasible >= 10


def test_a_very_long_model_fits():
    """450,000 model points at K = 4: the argmin tables of a full grid would take 325 GB. One far scene point, so that
    every point takes eps: the energy is the sum of lambda1 W^d = 1/2, exact in FP32."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    M = 450_000
    m = hgm.Model(np.zeros((M, 2), np.float32), np.zeros(M, np.int32), np.zeros((M, 1), np.float32))
    s = hgm.Scene(np.zeros((1, 2), np.float32), np.zeros(1, np.int32), np.full((1, 1), 8.0, np.float32), 1)
    p = hgm.default_params(K=4, window=0, lambda1=0.5, dummy_cost=1.0, offset_lo=0, offset_hi=0)
    hgm.set_workspace_budget(64 << 20)
    try:
        _, e, a = hgm.match(m, s, p)
    finally:
        hgm.set_workspace_budget(0)
    assert e[0] == 0.5 * M and np.all(a == -2)
