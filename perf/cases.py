"""Performance cases of the matching library: what a program that uses it has it do, through its public calls.

Seven kinds of work, each a dict of plain values:

* ``pair``: one model against one scene, every offset: `hgm.match`, `hgm.match_noalloc` (a loop that may not
  allocate) or a recorded plan's replay;
* ``batch``: several models against several scenes in one call (`hgm.match_batch`), in FP32 or with the BF16
  unary table, with or without learned pruning or the dummy assignment;
* ``chains``: models of several points per frame split into single-point chains (`hgm.match_chains_batch`);
* ``arrive``: scenes that arrive as host arrays: handles created, matched, results read back, in every pass;
* ``block``: whole scenes, every point a candidate (`hgm.match_block`);
* ``stream``: one block of a video in, every model's result out (`hgm.Stream`), host to host;
* ``train``: a run of optimiser steps of the proposal network from given weights (`hgm.Proposal`).

Inputs are synthetic, shaped like the repository's workloads: uniform positions, Poisson counts per frame,
cluster-structured descriptors, and jittered copies of models placed in the scenes. They are made on the GPU
from the seed alone. `exact` computes the same answers in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_1505_00581_gb300 import hgm

LAM1, LAM2, LAM3, T_CLOSE = 0.6, 0.2, 5.0, 10
SPAN = 30                       # frames a model of the batch kinds covers
HIDDEN = 128                    # width of the proposal network
TWO_PI = 2.0 * math.pi


# ---- the cases -----------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one short model against a two-second scene; latency and launches count
        dict(name="pair_short", kind="pair", entry="match", M=16, F=162, frames=60, density=10.0, K=32, window=2),
        # a real-time loop that may not allocate: one model, ten seconds of a sparse video
        dict(name="pair_noalloc", kind="pair", entry="noalloc", M=30, F=162, frames=300, density=30.0, K=64, window=3),
        # the ordinary batch: models of 16..64 points against scenes of 300 frames with 30 points per frame
        dict(name="batch_exact", kind="batch", n_models=10, M_lo=16, M_hi=64, F=162, n_scenes=2, frames=300,
             density=30.0, hop=0, K=64, window=3, precision=0, keep=0, dummy=-1.0),
        # crowded scenes, long models, windows of about 560 points; the scenes are blocks of longer videos
        dict(name="batch_dense", kind="batch", n_models=24, M_lo=16, M_hi=256, F=162, n_scenes=4, frames=75,
             density=80.0, hop=40, K=64, window=3, precision=0, keep=0, dummy=-1.0),
        # the same work with the learned pruning (16 of 64 candidates kept) and the BF16 unary table
        dict(name="pruned_dense", kind="batch", n_models=24, M_lo=16, M_hi=256, F=162, n_scenes=4, frames=75,
             density=80.0, hop=40, K=64, window=3, precision=1, keep=16, dummy=-1.0),
        # the BF16 unary table without pruning, descriptors padded to 176 components
        dict(name="batch_bf16", kind="batch", n_models=8, M_lo=32, M_hi=128, F=176, n_scenes=1, frames=400,
             density=60.0, hop=0, K=64, window=3, precision=1, keep=0, dummy=-1.0),
        # model points may stay unmatched (occlusion): the dummy assignment at the benchmark's cost
        dict(name="batch_dummy", kind="batch", n_models=10, M_lo=16, M_hi=64, F=162, n_scenes=1, frames=300,
             density=30.0, hop=0, K=64, window=3, precision=0, keep=0, dummy=8.0),
        # several points per model frame, matched as two chains
        dict(name="chains", kind="chains", n_models=10, M_lo=40, M_hi=80, F=162, n_scenes=1, frames=300,
             density=30.0, K=64, window=3, n_chains=2),
        # a new scene arrives in host memory: upload, sort, match against kept models, read back
        dict(name="scene_arrives", kind="arrive", n_models=4, M_lo=16, M_hi=64, F=162, n_scenes=1, frames=900,
             density=30.0, K=64, window=3),
        # the paper's own problem: 50 models of 30 points against a 723-frame scene of about 750 points
        dict(name="whole_scene", kind="block", n_models=50, M=30, F=162, frames=723, density=1.0),
        # the paper's real-time form: one 60-frame block, 50 models, host points in and host results out
        dict(name="stream_block", kind="stream", n_models=50, M=30, F=162, frames=60, density=1.0),
        # training the proposal network: optimiser steps on batches of candidate pairs
        dict(name="train", kind="train", B=4096, F=162, steps=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["pair", "pair", "batch", "batch", "batch", "batch", "chains", "arrive", "block", "block",
                       "stream", "train", "train"])
    F = rng.choice([162, 162, 176, 128, 100, 33, 75])
    if kind == "pair":
        return dict(kind=kind, entry=rng.choice(["match", "noalloc", "plan"]), M=int(_log(rng, 5, 128)), F=F,
                    frames=int(_log(rng, 45, 500)), density=round(_log(rng, 4.0, 60.0), 2), K=rng.randint(9, 64),
                    window=rng.randint(1, 4))
    if kind in ("batch", "arrive", "chains"):
        frames = int(_log(rng, 60, 700))
        density = round(_log(rng, 8.0, 85.0), 2)
        M_lo = rng.randint(40, 60) if kind == "chains" else rng.randint(12, 40)
        M_hi = rng.randint(M_lo, 200 if kind == "batch" else 80)
        # offsets x scenes x models x points of a model: bounded so that no form costs more than batch_dense
        most = 0.5 * 24 * 4 * 40 * 136
        room = most / ((frames - SPAN) * 0.5 * (M_lo + M_hi))
        n_models = max(1, min(16, int(_log(rng, 1.0, max(1.01, room)))))
        n_scenes = max(1, min(4, int(room / n_models)))
        while frames > 60 and n_models * n_scenes * (frames - SPAN) * 0.5 * (M_lo + M_hi) > most:
            frames -= 10
        case = dict(kind=kind, n_models=n_models, M_lo=M_lo, M_hi=M_hi, F=F, n_scenes=n_scenes, frames=frames,
                    density=density, K=rng.choice([64, 64, rng.randint(12, 63)]), window=rng.randint(1, 3))
        if kind == "batch":
            form = rng.choice(["exact", "bf16", "pruned", "pruned", "dummy"])
            case.update(hop=rng.choice([0, 0, 16]), precision=1 if form in ("bf16", "pruned") else 0,
                        keep=0 if form != "pruned" else min(case["K"] - 1, rng.randint(8, 20)),
                        dummy=round(rng.uniform(6.0, 14.0), 2) if form == "dummy" else -1.0)
        if kind == "chains":
            case["n_chains"] = rng.randint(1, 3)
        return case
    if kind == "block":
        return dict(kind=kind, n_models=int(_log(rng, 1, 60)), M=rng.randint(10, 40), F=F,
                    frames=int(_log(rng, 60, 800)), density=round(_log(rng, 0.5, 2.0), 2))
    if kind == "stream":
        return dict(kind=kind, n_models=int(_log(rng, 4, 60)), M=rng.randint(15, 30), F=F,
                    frames=rng.randint(40, 90), density=round(_log(rng, 0.6, 2.0), 2))
    return dict(kind="train", B=int(_log(rng, 64, 8192)), F=F, steps=rng.randint(1, 8))


# ---- inputs ----------------------------------------------------------------------------------------------------
def _size(case):
    """Sides of a frame: the sparse videos are 160 x 120, the crowded ones larger (the benchmark's shapes)."""
    if case["kind"] in ("block", "stream") or case["density"] < 15:
        return 160.0, 120.0
    return (320.0, 240.0) if case["density"] < 45 else (640.0, 480.0)


def _models(case, rng, gen, per_frame_one=False):
    """[(xy, t, f, centres)]: cluster-structured descriptors; frames sorted, consecutive triples within T."""
    n = case.get("n_models", 1)
    W, H = _size(case)
    out = []
    for k in range(n):
        if "M" in case:
            M = case["M"]
        else:   # sizes spread over the range, the same for every seed: the work does not depend on the seed
            M = int(round(case["M_lo"] + (case["M_hi"] - case["M_lo"]) * (k + 0.5) / n))
        if per_frame_one:
            t = np.arange(M)
        else:   # first and last frame fixed, so that the number of offsets does not depend on the seed
            last = min(SPAN, 2 * M) - 1
            while True:
                t = np.sort(np.concatenate([[0, last], rng.integers(0, last + 1, size=M - 2)]))
                if np.all(t[2:] - t[:-2] < T_CLOSE):
                    break
        centres = torch.randn((8, case["F"]), generator=gen, device="cuda")
        lab = torch.randint(0, 8, (M,), generator=gen, device="cuda")
        f = centres[lab] + 0.3 * torch.randn((M, case["F"]), generator=gen, device="cuda")
        xy = torch.rand((M, 2), generator=gen, device="cuda") * torch.tensor([W, H], device="cuda")
        out.append((xy, torch.from_numpy(t.astype(np.int32)).cuda(), f, centres))
    return out


def _scene(case, models, rng, gen):
    """(xy, t, f, frames): clutter in frame order, then jittered copies of models (so not time sorted)."""
    W, H = _size(case)
    nf = case["frames"]
    counts = rng.poisson(case["density"], size=nf)
    t = torch.from_numpy(np.repeat(np.arange(nf), counts).astype(np.int32)).cuda()
    pool = torch.cat([m[3] for m in models])
    n = int(t.shape[0])
    side = torch.tensor([W, H], device="cuda")
    xs = [torch.rand((n, 2), generator=gen, device="cuda") * side]
    ts = [t]
    pick = torch.randint(0, pool.shape[0], (n,), generator=gen, device="cuda")
    fs = [pool[pick] + 0.3 * torch.randn((n, case["F"]), generator=gen, device="cuda")]
    for _ in range(max(1, nf // 150)):
        xy, mt, f, _c = models[int(rng.integers(len(models)))]
        o = int(rng.integers(0, max(1, nf - SPAN)))
        jt = torch.randn(mt.shape, generator=gen, device="cuda").round().int()
        xs.append(xy + 2.0 * torch.randn(xy.shape, generator=gen, device="cuda"))
        ts.append((mt + o + jt).clamp(0, nf - 1))
        fs.append(f + 0.1 * torch.randn(f.shape, generator=gen, device="cuda"))
    return torch.cat(xs).contiguous(), torch.cat(ts).contiguous(), torch.cat(fs).contiguous(), nf


def _distance_net(F, gen):
    """Proposal weights that score a candidate by a sketch of its descriptor distance, its distance in the frame
    and its frame difference, as a trained network comes to do: hidden units are relu(+-g.(f - f')) for random
    directions g, the second layer mixes them, the output weighs them negatively."""
    d = 2 * F + 3
    W1 = torch.zeros((HIDDEN, d), device="cuda")
    g = torch.randn((62, F), generator=gen, device="cuda") / math.sqrt(F)
    W1[0:62, :F], W1[0:62, F:2 * F] = g, -g
    W1[62:124, :F], W1[62:124, F:2 * F] = -g, g
    for k, s in ((124, 0.5), (125, -0.5)):
        W1[k, 2 * F + 2] = s
    W1[126, 2 * F], W1[127, 2 * F + 1] = 0.05, 0.05
    W2 = torch.eye(HIDDEN, device="cuda") + 0.02 * torch.randn((HIDDEN, HIDDEN), generator=gen, device="cuda")
    w3 = -torch.full((HIDDEN,), 1.0 / 62, device="cuda")
    w3[124:126] = -0.3
    w3[126:128] = -0.02
    z = torch.zeros(HIDDEN, device="cuda")
    return torch.cat([W1.reshape(-1), z, W2.reshape(-1), z + 0.01, w3, z[:1] + 1.0]).cpu().numpy()


def _inputs(case, seed):
    """The arrays of a case: {"models", "scenes", "net"}; the same for `prepare` and `exact`."""
    rng = np.random.default_rng([seed, 20150500])
    gen = torch.Generator(device="cuda").manual_seed(seed * 1000003 + 17)
    if case["kind"] == "train":
        F, B, n = case["F"], case["B"], case["steps"]
        d = 2 * F + 3
        w = [math.sqrt(2.0 / d) * torch.randn((HIDDEN, d), generator=gen, device="cuda"), torch.zeros(HIDDEN, device="cuda"),
             math.sqrt(2.0 / HIDDEN) * torch.randn((HIDDEN, HIDDEN), generator=gen, device="cuda"),
             torch.zeros(HIDDEN, device="cuda"),
             math.sqrt(1.0 / HIDDEN) * torch.randn((HIDDEN,), generator=gen, device="cuda"),
             torch.zeros(1, device="cuda")]
        X, y = [], []
        for _ in range(n):   # candidate pairs: a model row, a clutter or matching row, position and frame differences
            cen = torch.randn((8, F), generator=gen, device="cuda")
            la = torch.randint(0, 8, (B,), generator=gen, device="cuda")
            pos = torch.rand((B,), generator=gen, device="cuda") < 1.0 / 16
            lb = torch.where(pos, la, torch.randint(0, 8, (B,), generator=gen, device="cuda"))
            fa = cen[la] + 0.3 * torch.randn((B, F), generator=gen, device="cuda")
            fb = torch.where(pos[:, None], fa, cen[lb]) + 0.2 * torch.randn((B, F), generator=gen, device="cuda")
            X.append(torch.cat([fa, fb, torch.randn((B, 3), generator=gen, device="cuda")], dim=1).contiguous())
            y.append(pos.float())
        return dict(weights=torch.cat([v.reshape(-1) for v in w]).cpu().numpy(), X=X, y=y)
    one = case["kind"] in ("block", "stream")
    models = _models(case, rng, gen, per_frame_one=one)
    scenes = [_scene(case, models, rng, gen) for _ in range(case.get("n_scenes", 1))]
    net = _distance_net(case["F"], gen) if case.get("keep", 0) else None
    return dict(models=models, scenes=scenes, net=net)


def _params(case, **over):
    p = dict(lambda1=LAM1, lambda2=LAM2, lambda3=LAM3, T=T_CLOSE)
    for k in ("K", "window", "precision"):
        if k in case:
            p[k] = case[k]
    if case.get("dummy", -1.0) >= 0:
        p["dummy_cost"] = case["dummy"]
    if case.get("hop", 0):
        p["offset_lo"], p["offset_hi"] = case["window"], case["window"] + case["hop"] - 1
    p.update(over)
    return hgm.default_params(**p)


# ---- a pass ------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    st = dict(case=case)
    if kind == "train":
        st.update(prop=hgm.Proposal(case["F"], weights=d["weights"]), weights=d["weights"], X=d["X"], y=d["y"],
                  loss=[torch.zeros(1, device="cuda") for _ in d["X"]])
        return st
    st["models"] = [hgm.Model(xy, t, f) for xy, t, f, _c in d["models"]]
    if kind in ("arrive", "stream"):   # the points are still in (pinned) host memory
        st["host"] = [tuple(v.cpu().pin_memory() for v in s[:3]) + (s[3],) for s in d["scenes"]]
        st["params"] = _params(case)
        if kind == "stream":
            st["stream"] = hgm.Stream(st["models"], st["params"], case["frames"],
                                      max_points=max(256, int(d["scenes"][0][1].shape[0])))
        return st
    st["scenes"] = [hgm.Scene(xy, t, f, nf) for xy, t, f, nf in d["scenes"]]
    st["prop"] = hgm.Proposal(case["F"], weights=d["net"]) if d["net"] is not None else None
    st["params"] = _params(case, **({"prune": st["prop"], "keep": case["keep"]} if st["prop"] is not None else {}))
    if kind == "block":
        ne, na = len(st["models"]) * len(st["scenes"]), sum(m.M for m in st["models"]) * len(st["scenes"])
    else:
        _first, es, as_ = hgm.batch_layout(st["models"], st["scenes"], st["params"])
        ne, na = int(es[-1]), int(as_[-1])
    st["energy"] = torch.empty(ne, dtype=torch.float32, device="cuda")
    st["assign"] = torch.empty(na, dtype=torch.int32, device="cuda")
    if case.get("entry") == "plan":
        st["plan"] = hgm.Plan(st["models"], st["scenes"], st["params"], st["energy"], st["assign"])
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "train":
        prop = st["prop"]
        prop.set(st["weights"])
        for X, y, loss in zip(st["X"], st["y"], st["loss"]):
            prop.train_step(X, y, 1e-3, loss)
        return {"loss": list(st["loss"]), "weights": prop.get()[0]}
    if kind == "stream":
        xy, t, f, _nf = st["host"][0]
        e, a = st["stream"].match(xy, t, f)
        return {"energy": e, "assign": a}
    if kind == "arrive":
        scenes = [hgm.Scene(xy, t, f, nf) for xy, t, f, nf in st["host"]]
        _first, es, as_ = hgm.batch_layout(st["models"], scenes, st["params"])
        e = np.empty(int(es[-1]), np.float32)
        a = np.empty(int(as_[-1]), np.int32)
        hgm.match_batch(st["models"], scenes, st["params"], e, a)
        for s in scenes:
            s.close()
        return {"energy": e, "assign": a}
    args = (st["energy"], st["assign"])
    if kind == "pair":
        m, s = st["models"][0], st["scenes"][0]
        if case["entry"] == "plan":
            st["plan"].run()
        elif case["entry"] == "noalloc":
            hgm.match_noalloc(m, s, st["params"], *args)
        else:
            hgm.match(m, s, st["params"], *args)
    elif kind == "block":
        hgm.match_block(st["models"], st["scenes"], st["params"], *args)
    elif kind == "chains":
        hgm.match_chains_batch(st["models"], st["scenes"], st["params"], case["n_chains"], *args)
    else:
        hgm.match_batch(st["models"], st["scenes"], st["params"], *args)
    return {"energy": st["energy"], "assign": st["assign"]}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def _model_sizes(case):
    n = case.get("n_models", 1)
    if "M" in case:
        return [case["M"]] * n
    return [int(round(case["M_lo"] + (case["M_hi"] - case["M_lo"]) * (k + 0.5) / n)) for k in range(n)]


def work(case):
    """Bytes: points, weights and results once each. Flops: the descriptor distance of every (model point,
    reachable scene point), and one 12-operation triple for every cell (z_{i-1}, z_{i-2}) of the recursion that
    can be feasible (each needs its minimum); the network's products where it runs."""
    F, kind = case["F"], case["kind"]
    if kind == "train":
        d, B, n = 2 * F + 3, case["B"], case["steps"]
        par = HIDDEN * (d + HIDDEN + 3) + 1
        products = 2 * B * HIDDEN * (d + HIDDEN + 1)
        return {"bytes": n * B * (d + 1) * 4 + 2 * par * 4, "flops": n * (2 * products + 2 * B * HIDDEN * (HIDDEN + 1))}
    sizes = _model_sizes(case)
    ns, nf = case.get("n_scenes", 1), case["frames"]
    S = case["density"] * nf
    point = 4.0 * (F + 3)
    rows = float(sum(sizes))
    if kind in ("block", "stream"):
        band = case["density"] * T_CLOSE
        return {"bytes": point * (S * ns + rows) + ns * (4 * len(sizes) + 4 * rows),
                "flops": ns * (3.0 * F * rows * S + 12.0 * (rows - 2 * len(sizes)) * S * band)}
    offs = case["hop"] if case.get("hop", 0) else max(1, nf - SPAN + 1)
    K = min(case["K"], case["density"] * (2 * case["window"] + 1))
    cells = 0.5 * K * K
    fl = ns * (3.0 * F * rows * S + 12.0 * offs * (rows - 2 * len(sizes)) * cells)
    if case.get("keep", 0):
        cells = 0.5 * case["keep"] ** 2
        fl = ns * (3.0 * F * rows * S + 12.0 * offs * (rows - 2 * len(sizes)) * cells +
                   2.0 * HIDDEN * HIDDEN * offs * rows * K + 2.0 * HIDDEN * F * (S + rows))
    return {"bytes": point * (S * ns + rows) + ns * offs * (4 * len(sizes) + 4 * rows), "flops": fl}


def tolerance(case):
    """About four times what was seen between the FP32 results and the same in 64 bits (matching), and between
    two orders of a batch's rows (training). Assignments: nearly equal chains may swap."""
    if case["kind"] == "train":
        return {"rel": 5e-5, "max": 0.03}    # max: Adam's first steps are +-lr, a gradient near 0 may flip its sign
    if case.get("keep", 0) or case.get("precision", 0):
        return {"rel": 1e-3, "max": 0.2, "differ": 0.01}     # which candidates are kept hangs on BF16 values
    return {"rel": 2e-6, "max": 2e-5, "differ": 2e-3}


# ---- the same in 64 bits ---------------------------------------------------------------------------------------------
def _wrap(x):
    return x - TWO_PI * torch.round(x / TWO_PI)


def _dir(p, q):
    d = q - p
    return torch.atan2(d[..., 1], d[..., 0])


def _angles(xy):
    """Signed model angles of every hyperedge (i, i-1, i-2): A1 at i-1, A2 at i."""
    i, j, k = xy[2:], xy[1:-1], xy[:-2]
    return _wrap(_dir(j, k) - _dir(j, i)), _wrap(_dir(i, k) - _dir(i, j))


def _sorted(points):
    xy, t, f = points[:3]
    order = torch.argsort(t.long(), stable=True)
    return xy[order].double(), t[order].long(), f[order].double()


def _lists(model, scene, U, offs, K, window):
    """Candidate lists of offsets `offs`: sorted scene indices [n, M, K] (ascending, -1 after the last)."""
    t, nf = scene["t"], scene["nf"]
    start = torch.searchsorted(t, torch.arange(nf + 1, device="cuda"))
    c = model["t"][None, :] + offs[:, None]
    f0, f1 = (c - window).clamp(min=0), (c + window).clamp(max=nf - 1)
    j0 = start[f0.clamp(max=nf)]
    cnt = torch.where(f0 <= f1, start[(f1 + 1).clamp(0, nf)] - j0, torch.zeros_like(j0))
    width = max(int(cnt.max()), K)
    w = torch.arange(width, device="cuda")
    j = j0[..., None] + w
    ok = w < cnt[..., None]
    key = torch.gather(U[None].expand(len(offs), -1, -1), 2, j.clamp(max=U.shape[1] - 1))
    key = torch.where(ok, key, torch.full_like(key, math.inf))
    val, pick = torch.topk(key, K, dim=-1, largest=False)
    idx = torch.where(torch.isfinite(val), torch.gather(j, 2, pick), torch.full_like(pick, 1 << 40))
    idx = torch.sort(idx, dim=-1).values
    return torch.where(idx < (1 << 40), idx, torch.full_like(idx, -1))


def _solve(model, scene, U, idx, ueps=None):
    """Minimal energies of the recursion over the lists idx [n, M, K]; ueps: cost of the dummy assignment."""
    n, M, K = idx.shape
    if ueps is not None:
        idx = torch.cat([idx, torch.full((n, M, 1), -2, device="cuda", dtype=idx.dtype)], dim=2)
        K += 1
    xy, t = scene["xy"], scene["t"]
    A1, A2 = model["ang"]
    inf = torch.tensor(math.inf, device="cuda", dtype=torch.float64)
    safe = idx.clamp(min=0)

    def lst(i):
        j = idx[:, i]
        u = torch.where(j >= 0, torch.gather(U[i][None].expand(n, -1), 1, safe[:, i]), inf)
        real = j >= 0
        if ueps is not None:
            u = torch.where(j == -2, torch.full_like(u, ueps), u)
        return dict(j=j, real=real, eps=j == -2, u=u, xy=xy[safe[:, i]], t=t[safe[:, i]])

    def pair_ok(p, q):   # p later in the chain than q: [n, p, q], true where the pair may stand in one triple
        ok = (p["t"][:, :, None] >= q["t"][:, None, :]) & (p["j"][:, :, None] != q["j"][:, None, :])
        ok &= p["t"][:, :, None] - q["t"][:, None, :] < T_CLOSE
        ok &= p["real"][:, :, None] & q["real"][:, None, :]
        return ok | p["eps"][:, :, None] & (q["real"] | q["eps"])[:, None, :] | p["real"][:, :, None] & q["eps"][:, None, :]

    alpha = torch.zeros((n, K, K), device="cuda", dtype=torch.float64)     # alpha_{i+1}(a, b)
    L = {i: lst(i) for i in (M - 1, M - 2) if i >= 0}
    for i in range(M - 1, 1, -1):
        L[i - 2] = lst(i - 2)
        a, b, c = L[i], L[i - 1], L[i - 2]
        mt = model["t"]
        dab = (mt[i] - mt[i - 1] - (a["t"][:, :, None] - b["t"][:, None, :])).abs().double()
        dbc = (mt[i - 1] - mt[i - 2] - (b["t"][:, :, None] - c["t"][:, None, :])).abs().double()
        if ueps is not None:
            dab = torch.where(a["real"][:, :, None] & b["real"][:, None, :], dab, 0.0 * dab)
            dbc = torch.where(b["real"][:, :, None] & c["real"][:, None, :], dbc, 0.0 * dbc)
        base = torch.where(pair_ok(a, b), a["u"][:, :, None] + LAM2 * dab + alpha, inf)        # [n, a, b]
        p1 = A1[i - 2] + _dir(b["xy"][:, None], a["xy"][:, :, None])                              # theta(b->a)
        p2 = A2[i - 2] + _dir(a["xy"][:, :, None], b["xy"][:, None])                              # theta(a->b)
        q1 = _dir(b["xy"][:, :, None], c["xy"][:, None])                                        # [n, b, c]
        r = _dir(a["xy"][:, :, None], c["xy"][:, None])                                         # [n, a, c]
        okac, okbc = pair_ok(a, c), pair_ok(b, c)
        new = torch.empty((n, K, K), device="cuda", dtype=torch.float64)
        step = max(1, int(6e7 / K ** 3))
        for k0 in range(0, n, step):
            s = slice(k0, min(n, k0 + step))
            g = _wrap(p1[s, :, :, None] - q1[s, None]).square_()
            g += _wrap(p2[s, :, :, None] - r[s, :, None, :]).square_()
            g = g.sqrt_().mul_(LAM2 * LAM3)
            if ueps is not None:
                real = a["real"][s, :, None, None] & b["real"][s, None, :, None] & c["real"][s, None, None, :]
                g = torch.where(real, g, 0.0 * g)
            g += torch.where(okac[s], 0.0, inf)[:, :, None, :]
            g += base[s, :, :, None]
            new[s] = g.amin(dim=1)
        alpha = torch.where(okbc, new + LAM2 * dbc, inf)
        del L[i]
    return (L[0]["u"][:, None, :] + L[1]["u"][:, :, None] + alpha).flatten(1).amin(dim=1)


def _network(net, F):
    w = torch.from_numpy(net).cuda().double()
    d, at, out = 2 * F + 3, 0, []
    for shape in ((HIDDEN, d), (HIDDEN,), (HIDDEN, HIDDEN), (HIDDEN,), (HIDDEN,), (1,)):
        k = int(np.prod(shape))
        out.append(w[at:at + k].reshape(shape))
        at += k
    return out


def _keep(case, net, model, scene, idx, offs):
    """The `keep` best-scored candidates of every list, in ascending scene index."""
    F = case["F"]
    W1, b1, W2, b2, w3, b3 = net
    P = model["f"] @ W1[:, :F].T + b1
    Q = scene["f"] @ W1[:, F:2 * F].T
    out = torch.empty(idx.shape[:2] + (case["keep"],), device="cuda", dtype=idx.dtype)
    for k in range(idx.shape[0]):
        j = idx[k].clamp(min=0)
        dxy = (scene["xy"][j] - model["xy"][:, None]) / 100.0
        dt = (scene["t"][j] - model["t"][:, None] - offs[k]).double() / max(case["window"], 1)
        h = P[:, None] + Q[j] + torch.cat([dxy, dt[..., None]], dim=-1) @ W1[:, 2 * F:].T
        z = torch.relu(torch.relu(h) @ W2.T + b2) @ w3 + b3
        z = torch.where(idx[k] >= 0, z, torch.full_like(z, -math.inf))
        pick = torch.sort(z, dim=-1, descending=True, stable=True).indices[:, :case["keep"]]
        got = torch.gather(idx[k], 1, pick)
        got = torch.sort(torch.where(got >= 0, got, torch.full_like(got, 1 << 40)), dim=-1).values
        out[k] = torch.where(got < (1 << 40), got, torch.full_like(got, -1))
    return out


def _pair_energies(case, model, scene, net, span=None):
    """Energies of one (model, scene) pair at every offset; span: (first, last) model frame that set the range."""
    lo, hi = span if span else (int(model["t"].min()), int(model["t"].max()))
    o0, o1 = -lo, scene["nf"] - 1 - hi
    if case.get("hop", 0):
        o0, o1 = max(o0, case["window"]), min(o1, case["window"] + case["hop"] - 1)
    if o1 < o0:
        return torch.zeros(0, device="cuda", dtype=torch.float64)
    U = LAM1 * torch.cdist(model["f"], scene["f"], compute_mode="donot_use_mm_for_euclid_dist")
    ueps = LAM1 * case["dummy"] if case.get("dummy", -1.0) >= 0 else None
    out = []
    width = case["density"] * (2 * case["window"] + 1) + 60
    chunk = max(1, int(4e7 / (model["t"].shape[0] * width)))
    for k0 in range(o0, o1 + 1, chunk):
        offs = torch.arange(k0, min(o1 + 1, k0 + chunk), device="cuda")
        idx = _lists(model, scene, U, offs, case["K"], case["window"])
        if net is None:
            out.append(_solve(model, scene, U, idx, ueps))
            continue
        e = _solve(model, scene, U, _keep(case, net, model, scene, idx, offs))
        bad = torch.nonzero(~torch.isfinite(e)).flatten()
        if len(bad):
            e[bad] = _solve(model, scene, U, idx[bad])
        out.append(e)
    return torch.cat(out)


def _block_energies(model, scene):
    """The whole-block problem of one pair: every scene point a candidate, as lists over the time band."""
    xy, t, nf = scene["xy"], scene["t"], scene["nf"]
    S, M = t.shape[0], model["t"].shape[0]
    start = torch.searchsorted(t, torch.arange(nf + 1, device="cuda"))
    clo, chi = start[(t - T_CLOSE + 1).clamp(min=0)], start[t + 1]          # c of b: [clo, chi)
    alo, ahi = start[t], start[(t + T_CLOSE).clamp(max=nf)]                 # a of b
    wc, wa = int((chi - clo).max()), int((ahi - alo).max())
    c = clo[:, None] + torch.arange(wc, device="cuda")                      # [S, wc]
    a = alo[:, None] + torch.arange(wa, device="cuda")                      # [S, wa]
    okc = (c < chi[:, None]) & (c != torch.arange(S, device="cuda")[:, None])
    oka = (a < ahi[:, None]) & (a != torch.arange(S, device="cuda")[:, None])
    c, a = c.clamp(max=S - 1), a.clamp(max=S - 1)
    A1, A2 = model["ang"]
    U = LAM1 * torch.cdist(model["f"], scene["f"], compute_mode="donot_use_mm_for_euclid_dist")
    inf = torch.tensor(math.inf, device="cuda", dtype=torch.float64)
    dba, dab = _dir(xy[:, None], xy[a]), _dir(xy[a], xy[:, None])           # [S, wa]
    dbc = _dir(xy[:, None], xy[c])                                          # [S, wc]
    dac = _dir(xy[a][:, :, None], xy[c][:, None])                           # [S, wa, wc]
    ok = (t[a][:, :, None] - t[c][:, None] < T_CLOSE) & (a[:, :, None] != c[:, None]) & oka[:, :, None] & okc[:, None]
    # where the cell (a, b) sits in a's band
    at = (torch.arange(S, device="cuda")[:, None] - clo[a]).clamp(0, wc - 1)
    alpha = torch.zeros((S, wc), device="cuda", dtype=torch.float64)
    for i in range(M - 1, 1, -1):
        mt = model["t"]
        base = U[i][a] + LAM2 * (mt[i] - mt[i - 1] - (t[a] - t[:, None])).abs().double() + alpha[a, at]
        g = _wrap(A1[i - 2] + dba[:, :, None] - dbc[:, None]).square() + _wrap(A2[i - 2] + dab[:, :, None] - dac).square()
        v = torch.where(ok, base[:, :, None] + LAM2 * LAM3 * g.sqrt(), inf).amin(dim=1)
        alpha = v + LAM2 * (mt[i - 1] - mt[i - 2] - (t[:, None] - t[c])).abs().double()
    e = torch.where(okc, U[0][c] + U[1][:, None] + alpha, inf)
    return e.amin().reshape(1)


def _train_exact(case, seed):
    d = _inputs(case, seed)
    w = [v.clone().requires_grad_() for v in _network(d["weights"], case["F"])]
    m, s = [torch.zeros_like(v) for v in w], [torch.zeros_like(v) for v in w]
    losses = []
    for k, (X, y) in enumerate(zip(d["X"], d["y"])):
        W1, b1, W2, b2, w3, b3 = w
        z = torch.relu(torch.relu(X.double() @ W1.T + b1) @ W2.T + b2) @ w3 + b3
        loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y.double())
        losses.append(loss.detach().reshape(1))
        grads = torch.autograd.grad(loss, w)
        c1, c2 = 1 - 0.9 ** (k + 1), 1 - 0.999 ** (k + 1)
        with torch.no_grad():
            for v, g, a, b in zip(w, grads, m, s):
                a.mul_(0.9).add_(g, alpha=0.1)
                b.mul_(0.999).addcmul_(g, g, value=0.001)
                v -= 1e-3 * (a / c1) / ((b / c2).sqrt() + 1e-8)
    return {"loss": losses, "weights": torch.cat([v.detach().reshape(-1) for v in w])}


def exact(case, seed):
    """Energies (the training losses and weights) in 64 bits; assignments have no such value. None where it
    would take long: long models at the full cap."""
    if case["kind"] == "train":
        return _train_exact(case, seed)
    sizes = _model_sizes(case)
    if case["kind"] not in ("block", "stream") and not case.get("keep", 0):
        offs = case["hop"] if case.get("hop", 0) else max(1, case["frames"] - SPAN + 1)
        K = min(case["K"], case["density"] * (2 * case["window"] + 1))
        if sum(sizes) * offs * case.get("n_scenes", 1) * K ** 3 > 2.5e11:
            return None
    d = _inputs(case, seed)
    models = []
    for m in d["models"]:
        xy, t, f = _sorted(m)
        models.append(dict(xy=xy, t=t, f=f, ang=_angles(xy)))
    scenes = []
    for s in d["scenes"]:
        xy, t, f = _sorted(s)
        scenes.append(dict(xy=xy, t=t, f=f, nf=s[3]))
    net = _network(d["net"], case["F"]) if d["net"] is not None else None
    out = []
    for m in models:
        for s in scenes:
            if case["kind"] in ("block", "stream"):
                out.append(_block_energies(m, s))
            elif case["kind"] == "chains":
                out.append(_chain_energies(case, m, s))
            else:
                out.append(_pair_energies(case, m, s, net))
    return {"energy": torch.cat(out), "assign": None}


def _chain_energies(case, model, scene):
    """The mean over the model's single-point chains: chain k has the k-th point of every frame that has one."""
    t = model["t"]
    same = t[:, None] == t[None]
    rank = torch.tril(same, -1).sum(dim=1)
    parts = []
    for k in range(case["n_chains"]):
        sel = rank == k
        if int(sel.sum()) < 3:
            continue
        xy = model["xy"][sel]
        part = dict(xy=xy, t=t[sel], f=model["f"][sel], ang=_angles(xy))
        parts.append(_pair_energies(case, part, scene, None, span=(int(t.min()), int(t.max()))))
    return torch.stack(parts).mean(dim=0)
