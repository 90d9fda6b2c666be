"""The proposal network's training pass (one kernel, 128 batch rows per tile) at the edges of its tiles and
chunks, against the BF16-operand reference of oracle/mlp.py."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1505_00581_gb300 import build, hgm
    build.build()
    hgm.load()
    return torch, hgm


def _case(hgm, F, B, seed):
    prop = hgm.Proposal(F, seed=seed)
    d = prop.unflatten(prop.get()[0].astype(np.float64))
    rng = np.random.default_rng(seed)
    for k in ("b1", "b2"):
        d[k] = (0.1 * rng.normal(size=128)).astype(np.float32).astype(np.float64)
    prop.set(np.concatenate([d[k].reshape(-1) for k in ("W1", "b1", "W2", "b2", "w3", "b3")]).astype(np.float32))
    X = rng.normal(size=(B, 2 * F + 3)).astype(np.float32)
    y = (rng.random(B) < 0.25).astype(np.float32)
    return prop, d, X, y


def _flips(p, x, y):
    """Per gradient element, the magnitude of the terms whose ReLU derivative rounding may flip. z2 moves by at
    most 2^-7 |W2 h1| for an h1 on the neighbouring BF16 value (two of the largest taken), z1 by the FP32
    accumulation of its n products, n 2^-24 sum |W1 x|."""
    c = mlp.forward_bf16(p, x)
    B = x.shape[0]
    dz3 = (1.0 / (1.0 + np.exp(-c["z3"])) - y) / B
    o = np.abs(np.outer(dz3, p["w3"]))
    big = np.stack([np.max(np.abs(p["W2"]) * np.abs(h)[None], axis=1) for h in c["h1"]])
    e2 = o * (np.abs(c["z2"]) <= 2.0 ** -6 * big)
    amb1 = np.abs(c["z1"]) <= x.shape[1] * 2.0 ** -24 * (np.abs(x) @ np.abs(p["W1"]).T)
    e1 = (e2 @ np.abs(p["W2"])) * (c["z1"] > 0) + ((o * (c["z2"] > 0) + e2) @ np.abs(p["W2"])) * amb1
    return {"W1": e1.T @ np.abs(x), "b1": e1.sum(axis=0), "W2": e2.T @ np.abs(c["h1"]), "b2": e2.sum(axis=0),
            "w3": 0.0, "b3": 0.0}


# F: one, two, three (resident) and four or more (staged again for the backward pass) chunks of 128 components,
# component counts that are and are not multiples of 16 or of the padded row; B: one row, the tile's edges,
# several tiles, and more tiles than SMs (a CTA adds to its own share)
@pytest.mark.parametrize("F,B", [(1, 1), (16, 127), (62, 128), (63, 129), (100, 300), (162, 513), (190, 65),
                                 (191, 200), (300, 130), (8, 20000), (200, 20000)])
def test_gradients_at_tile_and_chunk_edges(env, F, B):
    """Bounds as in test_gpu_prop.test_gradients_match_fp64: every element within 2^-6 of its scale (an
    activation computed in FP32 may land on the neighbouring BF16 value), the median within 2^-12; FP32 sums of
    n <= 20,000 terms add at most n 2^-24 = 1.2e-3 of the scale, and sums over 128-row tiles far less. Where
    such a difference takes a unit across 0, its ReLU's derivative flips and the sample's whole term comes or
    goes: _flips adds those terms for the units that close to 0."""
    torch, hgm = env
    prop, ref, X, y = _case(hgm, F, B, 5 + F)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    loss, g = prop.gradients(Xd, yd)
    gd = prop.unflatten(g.astype(np.float64))
    loss_emu, g_emu, scale = mlp.backward_bf16(ref, X.astype(np.float64), y.astype(np.float64))
    flips = _flips(ref, X.astype(np.float64), y.astype(np.float64))
    assert abs(loss - loss_emu) <= 1e-5 * max(1.0, loss_emu)
    ratios = []
    for k in ("W1", "b1", "W2", "b2", "w3", "b3"):
        err, sc = np.abs(gd[k] - g_emu[k]), scale[k] + 1e-30
        assert np.all(err <= 2.0 ** -6 * sc + flips[k] + 1e-12), (k, float(np.max(err / sc)))
        ratios.append((err / sc).reshape(-1))
    assert np.median(np.concatenate(ratios)) <= 2.0 ** -12
    loss2, g2 = prop.gradients(Xd, yd)
    assert loss2 == loss and np.array_equal(g2, g)       # the sums have a fixed order
    out = torch.empty(B, device="cuda")
    prop.forward(Xd, out)
    z = mlp.forward_bf16(ref, X.astype(np.float64))["z3"]
    assert np.max(np.abs(out.cpu().numpy() - z)) <= 2e-3 * max(1.0, np.max(np.abs(z)))


def test_step_equals_gradients_and_adam(env):
    """train_step's weights = Adam on the gradients call's values (the same kernels), in FP32: a few roundings of
    the update's size lr."""
    torch, hgm = env
    prop, ref, X, y = _case(hgm, 50, 700, 3)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    w = prop.get()[0].astype(np.float64)
    m, v = np.zeros_like(w), np.zeros_like(w)
    for t in (1, 2, 3):
        w = prop.get()[0].astype(np.float64)
        _, g = prop.gradients(Xd, yd)
        g = g.astype(np.float64)
        prop.train_step(Xd, yd, 1e-3)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        want = w - 1e-3 * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
        # FP32: c2 = 1 - 0.999^t keeps 2^-24 / 0.001 = 6e-5 of relative error, the update half of that
        assert np.max(np.abs(prop.get()[0] - want)) <= 1e-3 * 1e-4 + 2.0 ** -23 * np.max(np.abs(w))


@pytest.mark.parametrize("at", [0, 7, -1])
def test_logits_may_lie_in_the_input(env, at):
    """313 tiles on 152 SMs: the first round's logits would land in rows that the later rounds still read."""
    torch, hgm = env
    B, F = 40000, 1
    prop = hgm.Proposal(F, seed=9)
    X = torch.from_numpy(np.random.default_rng(9).normal(size=(B, 2 * F + 3)).astype(np.float32)).cuda()
    want = torch.empty(B, device="cuda")
    prop.forward(X, want)
    flat = X.view(-1)
    out = flat[flat.numel() - B:] if at < 0 else flat[at:at + B]
    prop.forward(X, out)
    assert torch.equal(out, want)
