"""The recursion kernel at the edges of its lists: caps around the two table sizes and off the 4-cell tiles, lists
shorter than the cap and of very different lengths, crowded frames (many points of equal time), every closeness
limit, points shared between lists, numbers of units for every form of the launch. Against the FP64 oracle on every offset
(tests/gpu_util.check_offset: energies 1e-5 relative, assignments equal or of the same FP64 energy)."""
import numpy as np
import pytest

from gpu_util import check_offset
from paper_1505_00581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    hgm.load()
    import oracle
    oracle.build()
    return torch, hgm, oracle


def _scene(rng, mod, n_frames, lam, crowd):
    sc = synth.make_scene(rng, n_frames, (60.0, 40.0), ("poisson", lam), mod.centres, [mod], [(0, 2)])
    t = sc.t.copy()
    t[rng.random(len(t)) < crowd] = n_frames // 2
    return synth.Scene(sc.xy, t, sc.f, None, n_frames, [])


@pytest.mark.parametrize("K,lam,crowd,T,window,M", [
    (17, 6.0, 0.0, 10, 2, 9), (31, 9.0, 0.2, 10, 3, 12), (32, 20.0, 0.0, 4, 2, 8), (33, 8.0, 0.1, 10, 2, 10),
    (47, 20.0, 0.3, 10, 3, 7), (63, 30.0, 0.0, 0, 1, 6), (64, 4.0, 0.5, 10, 3, 11), (64, 30.0, 0.0, 2, 3, 9),
    (64, 1.0, 0.0, 10, 3, 20), (61, 25.0, 0.1, 10, 2, 3)])
def test_list_edges(env, K, lam, crowd, T, window, M):
    torch, hgm, oracle = env
    rng = np.random.default_rng(1000 * K + M)
    mod = synth.make_model(rng, M, F=16, frame=(60.0, 40.0), t_span=10, T=max(T, 6))
    sc = _scene(rng, mod, 26, lam, crowd)
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(sc.xy, sc.t, sc.f, sc.n_frames)
    p = hgm.default_params(K=K, window=window, T=T)
    first, e, a = hgm.match(m, s, p)
    orc = oracle.Oracle(mod.xy, mod.t, mod.f, sc.xy, sc.t, sc.f, sc.n_frames, K=K, window=window, T=T,
                        lambda1=0.6, lambda2=0.2, lambda3=5.0)
    for k in range(len(e)):
        ok, _, why = check_offset(orc, first + k, e[k], a[k])
        assert ok, (first + k, why)
    # the same pair several times over: enough units for each form of the launch (a cluster per unit, a unit per SM,
    # the variants; with short lists four warps per unit, then two), whose bits must be those of the one pair
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for units in (sms // 2, 9 * sms):
        n = -(-units // len(e))
        eb = np.empty(n * e.size, np.float32)
        ab = np.empty(n * a.size, np.int32)
        hgm.match_batch([m] * n, [s], p, eb, ab)
        assert np.array_equal(eb.reshape(n, -1), np.broadcast_to(e, (n, e.size)))
        assert np.array_equal(ab.reshape(n, -1), np.broadcast_to(a.reshape(-1), (n, a.size)))


@pytest.mark.parametrize("K", [32, 64])
def test_few_and_many_units_give_the_same_bits(env, K):
    """One offset, some and thousands of units in a call (the launch shapes differ, results must not)."""
    torch, hgm, oracle = env
    rng = np.random.default_rng(K)
    mod = synth.make_model(rng, 14, F=16, frame=(60.0, 40.0), t_span=10)
    sc = _scene(rng, mod, 700, 12.0, 0.01)
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(sc.xy, sc.t, sc.f, sc.n_frames)
    first, e, a = hgm.match(m, s, hgm.default_params(K=K, window=3))
    for lo, n in ((first, 1), (first + 300, 31), (first + 400, 32), (first + 100, 40), (first + 200, 160), (first + 5, 400)):
        p = hgm.default_params(K=K, window=3, offset_lo=lo, offset_hi=lo + n - 1)
        f1, e1, a1 = hgm.match(m, s, p)
        assert f1 == lo and len(e1) == n
        assert np.array_equal(e1, e[lo - first:lo - first + n]) and np.array_equal(a1, a[lo - first:lo - first + n])


@pytest.mark.parametrize("K", [32, 64])
@pytest.mark.parametrize("n", [1, 20, 100, 300])
def test_fallback_of_few_and_many_units(env, K, n):
    """A keep of one leaves a chain of this crowded scene without a feasible assignment almost everywhere: the
    fallback's launches for few, some and many units give the exact path's bits on every unit they solve."""
    torch, hgm, oracle = env
    rng = np.random.default_rng(K)
    mod = synth.make_model(rng, 14, F=16, frame=(60.0, 40.0), t_span=10)
    sc = _scene(rng, mod, 700, 12.0, 0.01)
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(sc.xy, sc.t, sc.f, sc.n_frames)
    first, _ = hgm.offsets(m, s, hgm.default_params(K=K, window=3))
    lo = first + 150
    _, e, a = hgm.match(m, s, hgm.default_params(K=K, window=3, offset_lo=lo, offset_hi=lo + n - 1))
    hgm.prune_counters(True)
    prop = hgm.Proposal(16, seed=5)
    p = hgm.default_params(K=K, window=3, prune=prop, keep=1, offset_lo=lo, offset_hi=lo + n - 1)
    _, e1, a1 = hgm.match(m, s, p)
    solved = e1 == e
    assert solved.mean() > 0.9 and np.array_equal(a1[solved], a[solved])
    assert np.all(e1[~solved] > e[~solved])


def test_autotune_times_the_variants_on_a_small_sample(env):
    """One unit takes a cluster of four CTAs in a call, a variant's single CTA in the tuner: about twice as long
    for the 126 steps here. Tuning that ran the call's own form would show the same time."""
    torch, hgm, oracle = env
    rng = np.random.default_rng(4)
    mod = synth.make_model(rng, 128, F=16, frame=(60.0, 40.0), t_span=30)
    m = hgm.Model(mod.xy, mod.t, mod.f)
    sc = _scene(rng, mod, 60, 12.0, 0.0)
    s = hgm.Scene(sc.xy, sc.t, sc.f, sc.n_frames)
    p = hgm.default_params(K=64, window=3, offset_lo=5, offset_hi=5)

    def ms_per_launch(fn):
        hgm.profile_reset()
        hgm.profile_enable(True)
        fn()
        hgm.profile_enable(False)
        ms, n = hgm.profile_read()["recurse"]
        return ms / n

    hgm.set_recurse_variant(0)
    hgm.match(m, s, p)
    call = min(ms_per_launch(lambda: hgm.match(m, s, p)) for _ in range(5))
    tuned = ms_per_launch(lambda: hgm.autotune([m], [s], p, use_cache=False))
    assert tuned > 1.4 * call, (tuned, call)
    # nothing to choose: the choice stays, the three times are one measurement
    hgm.set_recurse_variant(2)
    for kw in (dict(K=16), dict(K=64, dummy_cost=4.0)):
        best, ms = hgm.autotune([m], [s], hgm.default_params(window=3, offset_lo=5, offset_hi=5, **kw), use_cache=False)
        assert best == 2 and len(set(ms.values())) == 1
    hgm.set_recurse_variant(0)


@pytest.mark.parametrize("K,lam,crowd,T,window,M", [
    (1, 3.0, 0.0, 10, 1, 5), (5, 6.0, 0.2, 10, 2, 9), (8, 20.0, 0.0, 4, 2, 8), (9, 8.0, 0.1, 10, 2, 10),
    (13, 20.0, 0.3, 0, 2, 7), (16, 30.0, 0.0, 10, 1, 3), (16, 1.0, 0.2, 10, 3, 20), (15, 12.0, 0.0, 2, 3, 9)])
def test_short_list_edges(env, K, lam, crowd, T, window, M):
    """The short-list kernel (caps up to 8 and up to 16) as above; the caps the large kernel takes next give the same
    optimum where no list is cut by either (tested through the oracle)."""
    test_list_edges(env, K, lam, crowd, T, window, M)


@pytest.mark.parametrize("K", [8, 16])
def test_short_lists_few_and_many_units(env, K):
    test_few_and_many_units_give_the_same_bits(env, K)
    torch, hgm, oracle = env
    rng = np.random.default_rng(K)
    mod = synth.make_model(rng, 12, F=16, frame=(60.0, 40.0), t_span=10)
    sc = _scene(rng, mod, 2500, 6.0, 0.0)       # more units than the four-warp form takes
    m, s = hgm.Model(mod.xy, mod.t, mod.f), hgm.Scene(sc.xy, sc.t, sc.f, sc.n_frames)
    first, e, a = hgm.match(m, s, hgm.default_params(K=K, window=3))
    p = hgm.default_params(K=K, window=3, offset_lo=first + 1000, offset_hi=first + 1099)
    f1, e1, a1 = hgm.match(m, s, p)
    assert np.array_equal(e1, e[1000:1100]) and np.array_equal(a1, a[1000:1100])
