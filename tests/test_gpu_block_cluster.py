"""The whole-block problem in its shared-memory form at the edges of its split: one CTA per pair with the argmin
tables in shared memory or not, several CTAs per pair (many cells, or few pairs), uneven frames, no closeness
limit. Against the FP64 oracle, with the bounds of the other whole-block tests (energies 1e-5 relative)."""
import numpy as np
import pytest

from paper_1505_00581_gb300 import synth
from test_gpu_block import LAM, _check, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _uneven(rng, mods, n_frames, lam, crowd):
    """A scene whose frames are mostly sparse, some empty, and one crowded: no split falls evenly."""
    pool = np.concatenate([m.centres for m in mods])
    sc = synth.make_scene(rng, n_frames, (60.0, 40.0), ("poisson", lam), pool, mods, [(0, n_frames // 3)])
    t = sc.t.copy()
    t[rng.random(len(t)) < crowd] = n_frames // 2
    return synth.Scene(sc.xy, t, sc.f, None, n_frames, [])


# frames, points per frame, share of points moved to one frame, T, models: about 200 cells (256 threads) up to
# 20,000 (more than one CTA holds, eight CTAs share a pair), pairs enough to leave one CTA each or few
@pytest.mark.parametrize("n_frames,lam,crowd,T,n_models,M", [
    (12, 1.0, 0.0, 10, 2, 5), (40, 1.2, 0.0, 10, 3, 12), (60, 4.0, 0.1, 10, 1, 9), (90, 6.0, 0.1, 10, 1, 6),
    (200, 3.0, 0.05, 10, 2, 20), (30, 3.0, 0.1, 0, 1, 6), (400, 2.0, 0.0, 25, 1, 8), (50, 2.0, 0.0, 1, 2, 3),
    (300, 5.5, 0.02, 10, 3, 7)])
def test_block_split_edges(env, n_frames, lam, crowd, T, n_models, M):  # noqa: F811
    torch, hgm, oracle = env
    rng = np.random.default_rng(77 + n_frames)
    mods = [synth.make_model(rng, M + k, F=16, frame=(60.0, 40.0), t_span=8) for k in range(n_models)]
    scs = [_uneven(rng, mods, n_frames, lam, crowd), _uneven(rng, mods, max(5, n_frames // 3), lam, 0.0)]
    _check(hgm, oracle, mods, scs, T=T)


def test_block_many_pairs_equal_single_calls(env):  # noqa: F811
    """More pairs than SMs (one CTA each), and every pair alone (several CTAs): the same bits."""
    torch, hgm, oracle = env
    rng = np.random.default_rng(5)
    mods = [synth.make_model(rng, 10, F=16, frame=(60.0, 40.0), t_span=9) for _ in range(100)]
    scs = [_uneven(rng, mods[:3], 150, 2.5, 0.03), _uneven(rng, mods[:3], 60, 1.5, 0.0)]
    M = [hgm.Model(m.xy, m.t, m.f) for m in mods]
    S = [hgm.Scene(s.xy, s.t, s.f, s.n_frames) for s in scs]
    p = hgm.default_params(K=8, window=1, T=10)
    e, a = hgm.match_block(M, S, p)
    for m in (0, 57, 99):
        e1, a1 = hgm.match_block([M[m]], [S[0]], p)
        assert e1[0] == e[2 * m]
        assert np.array_equal(a1, a[20 * m:20 * m + 10])


@pytest.mark.parametrize("T", [0, 4500])
def test_block_long_time_differences_take_the_general_form(env, T):  # noqa: F811
    """Bands that span 4,096 frames or more do not fit a cell's record and take the kernel on global tables."""
    torch, hgm, oracle = env
    rng = np.random.default_rng(9)
    mods = [synth.make_model(rng, M, F=16, frame=(60.0, 40.0), t_span=8) for M in (4, 7)]
    _check(hgm, oracle, mods, [_uneven(rng, mods, 5000, 0.012, 0.05), _uneven(rng, mods, 4700, 0.006, 0.0)], T=T)
