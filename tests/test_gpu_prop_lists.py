"""The proposal's scoring and keep kernels at the edges of their tiles and lists: list lengths that share a
128-row tile 128, 32, 8 or 2 at a time, models whose last tile is partly empty, and keeps from one candidate
to all but one, with distinct and with equal scores."""
import itertools

import numpy as np
import pytest

from gpu_util import handles
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


def _pair(seed, M, frames=40, density=30.0):
    rng = np.random.default_rng(seed)
    mod = synth.make_model(rng, M, t_span=max(8, 2 * M))
    sc = synth.make_scene(rng, frames, (320.0, 240.0), ("poisson", density), mod.centres, [mod], [(0, 5)])
    return mod, sc


def _scores(torch, hgm, m, s, prop, K, M):
    p = hgm.default_params(K=K, window=3)
    first, n = hgm.offsets(m, s, p)
    idx = torch.empty((n, M, K), dtype=torch.int32, device="cuda")
    cnt = torch.empty((n, M), dtype=torch.int32, device="cuda")
    hgm.candidates(m, s, p, first, n, idx, cnt)
    sco = torch.full((n, M, K), 7.0, dtype=torch.float32, device="cuda")
    hgm.prop_scores(prop, m, s, p, first, n, sco)
    torch.cuda.synchronize()
    return idx.cpu().numpy(), cnt.cpu().numpy(), sco.cpu().numpy()


@pytest.mark.parametrize("M", [3, 9, 33])
@pytest.mark.parametrize("K", [1, 3, 13, 48])
def test_a_candidates_score_does_not_depend_on_the_lists_length(env, K, M):
    """A logit is a function of (offset, model point, scene point): every candidate of a short list is in the
    K = 64 list of the same window too and has the same bits there, whatever tile and row it falls on. Empty
    slots score -inf."""
    torch, hgm, _ = env
    mod, sc = _pair(7 + M, M, frames=20 + 4 * M)
    m, s = handles(hgm, mod, sc, torch)
    prop = hgm.Proposal(162, seed=5)
    ia, ca, sa = _scores(torch, hgm, m, s, prop, 64, M)
    ib, cb, sb = _scores(torch, hgm, m, s, prop, K, M)
    assert ia.shape[0] == ib.shape[0]
    checked = 0
    for k, i in itertools.product(range(ia.shape[0]), range(M)):
        full = {int(j): sa[k, i, q] for q, j in enumerate(ia[k, i, :ca[k, i]])}
        for q in range(K):
            if q < cb[k, i]:
                assert sb[k, i, q] == full[int(ib[k, i, q])], (k, i, q)
                checked += 1
            else:
                assert sb[k, i, q] == -np.inf
    assert checked > 0


@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("K,keep", [(64, 1), (64, 10), (40, 16), (20, 19)])
def test_kept_candidates_are_the_highest_scores(env, K, keep, equal):
    """On a 3-point model the pruned optimum equals the brute-force minimum of Eq. 9 over the `keep` highest
    logits of each list (ties: lower slot). All-zero weights make every score equal. The tolerance is the
    FP32 recursion's against the FP64 oracle on three terms, as for the exact path: 1e-5 relative."""
    torch, hgm, oracle = env
    mod, sc = _pair(31, 3, density=20.0)
    wl = synth.Workload("tiny", [mod], [sc], K=K, window=3)
    m, s = handles(hgm, mod, sc, torch)
    prop = hgm.Proposal(162, seed=5)
    if equal:
        w, _ = prop.get()
        prop.set(np.zeros_like(w))
    idx, cnt, sco = _scores(torch, hgm, m, s, prop, K, 3)
    p = hgm.default_params(K=K, window=3, prune=prop, keep=keep)
    first, n = hgm.offsets(m, s, p)
    e = torch.empty(n, dtype=torch.float32, device="cuda")
    a = torch.empty((n, 3), dtype=torch.int32, device="cuda")
    hgm.match(m, s, p, e, a)
    e = e.cpu().numpy()
    mperm, sperm = m.order(), s.order()
    orc = oracle.Oracle.from_workload(wl)
    checked = 0
    for k in range(0, n, 9):
        lists = []
        for i in range(3):
            c = int(cnt[k, i])
            top = sorted(range(c), key=lambda j: (-float(sco[k, i, j]), j))[:keep]
            lists.append([int(sperm[idx[k, i, j]]) for j in sorted(top)])
        best, z = np.inf, np.empty(3, np.int64)
        for combo in itertools.product(*lists):
            z[mperm] = combo
            best = min(best, orc.energy(z))
        if not np.isfinite(best):
            best = orc.match(first + k)[0]   # the fallback to the full lists
        if np.isfinite(best):
            assert abs(float(e[k]) - best) <= 1e-5 * max(1.0, best), (k, e[k], best)
            checked += 1
        else:
            assert not np.isfinite(e[k])
    assert checked > 0
