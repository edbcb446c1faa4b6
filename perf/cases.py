"""The workloads this library is timed on, through its public entry points.

A case is a dict of plain values.  Kinds:

  register   TurboReg.register: one registration, waited for (device or host inputs)
  stream     TurboReg.register_async: one registration enqueued behind others
  batch      TurboReg.register_batched: many problems of uneven size in one call
  pivots     turboreg_select_pivots_noalloc: the K1 best edges of a weight matrix
  grad       MLPTrainer.grad: loss gradient of the proposal network
  train      MLPTrainer.train_step, and the weights after it

Inputs are correspondence sets of the three scene shapes the tests and the
benchmark use: a rigid motion, Gaussian inlier noise, and outliers uniform in
the bounding box of the transformed source.
"""
import math

import numpy as np
import torch

import paper_2507_01439_gb300 as trg
from paper_2507_01439_gb300.train_proposal import load_model

# box, translation range, inlier noise, tau = theta, pivots; street scenes turn
# mostly about z, the others any way
SHAPES = {
    "cube": dict(lo=(0, 0, 0), hi=(3, 3, 3), t=(1, 1, 1), sigma=0.01, tau=0.1, k1=1000, yaw=False),
    "indoor": dict(lo=(0, 0, 0), hi=(4, 4, 3), t=(1, 1, 1), sigma=0.01, tau=0.1, k1=2000, yaw=False),
    "outdoor": dict(lo=(-35, -35, -2), hi=(35, 35, 3), t=(5, 5, 0.5), sigma=0.05, tau=0.6, k1=1000, yaw=True),
}


def _single(name, kind, shape, n, ratio, **more):
    c = dict(kind=kind, shape=shape, n=n, ratio=ratio, tau=SHAPES[shape]["tau"], k1=SHAPES[shape]["k1"], k2=2,
             undirected=False, scoring=trg.SCORE_IN, host=False)
    c.update(more)
    return dict(c, name=name) if name else c


def _batch(name, num, n_lo, n_hi, k1, learned=False):
    c = dict(kind="batch", num=num, n_lo=n_lo, n_hi=n_hi, k1=k1, learned=learned)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a handful of matches left by a strict matcher, or a loop-closure check: latency only
        _single("tiny", "register", "cube", 67, 0.3, k1=64),
        # the call of the README's example: NumPy arrays in, a pose out
        _single("cube", "register", "cube", 1000, 0.1, host=True),
        # LiDAR odometry: a sequence of street-scale pairs, enqueued one behind another
        _single("outdoor", "stream", "outdoor", 2500, 0.2),
        # the benchmark's registration: room-scale pairs with few inliers, enqueued one behind another
        _single("indoor", "stream", "indoor", 5000, 0.05),
        # a loose threshold (dense graph) with the undirected search, three cliques per pivot and a
        # capped-error score, as the ablations run it; odd size
        _single("dense", "register", "indoor", 4333, 0.1, tau=0.3, k2=3, undirected=True, scoring=trg.SCORE_MSE),
        # every keypoint of a scan pair kept: a large single problem
        _single("large", "register", "indoor", 20000, 0.05),
        # offline evaluation of a data set: 256 pairs of uneven size in one call, default pivots
        _batch("batch mixed", 256, 500, 5000, 0),
        # many small problems at once (object poses, submap candidates)
        _batch("batch small", 64, 60, 600, 100),
        # the learned proposal on a batch, with the few pivots it is meant for
        _batch("learned", 32, 500, 5000, 100, learned=True),
        # pivot selection alone, as a plugin without allocation calls it
        dict(kind="pivots", name="pivots", n=5000, k1=2000),
        # training the proposal network: the gradient of a small batch, a step on a large one
        dict(kind="grad", name="grad", m=16384),
        dict(kind="train", name="train", m=131072),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["register", "register", "stream", "stream", "batch", "learned", "pivots", "grad", "train"])
    if kind in ("register", "stream"):
        shape = rng.choice(sorted(SHAPES))
        return _single(None, kind, shape, log(40, 18000), rng.uniform(0.05, 0.3),
                       tau=SHAPES[shape]["tau"] * rng.choice([0.5, 1.0, 1.0, 2.0, 3.0]), k1=log(50, 2000),
                       k2=rng.choice([1, 2, 2, 2, 3, 5]), undirected=rng.random() < 0.25,
                       scoring=rng.choice([trg.SCORE_IN, trg.SCORE_IN, trg.SCORE_MAE, trg.SCORE_MSE]),
                       host=kind == "register" and rng.random() < 0.5)
    if kind == "batch":
        lo = log(50, 2000)
        return _batch(None, log(4, 128), lo, rng.randint(lo, 5000), rng.choice([0, log(10, 2000)]))
    if kind == "learned":
        lo = log(300, 2000)
        return _batch(None, log(4, 32), lo, rng.randint(lo, 5000), log(10, 1000), learned=True)
    if kind == "pivots":
        return dict(kind=kind, n=log(100, 8192), k1=log(10, 8192))
    return dict(kind=kind, m=log(500, 131072))


# ---- inputs ----

def _rotation(rng, yaw):
    if yaw:
        a = rng.uniform(-math.pi, math.pi)
        b, c = np.deg2rad(rng.uniform(-5, 5, 2))
        rz = np.array([[math.cos(a), -math.sin(a), 0], [math.sin(a), math.cos(a), 0], [0, 0, 1]])
        ry = np.array([[math.cos(b), 0, math.sin(b)], [0, 1, 0], [-math.sin(b), 0, math.cos(b)]])
        rx = np.array([[1, 0, 0], [0, math.cos(c), -math.sin(c)], [0, math.sin(c), math.cos(c)]])
        return rz @ ry @ rx
    q = rng.normal(size=4)
    w, x, y, z = q / np.linalg.norm(q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _problem(rng, shape, n, ratio):
    sh = SHAPES[shape]
    x = rng.uniform(sh["lo"], sh["hi"], size=(n, 3))
    moved = x @ _rotation(rng, sh["yaw"]).T + rng.uniform(-np.array(sh["t"]), sh["t"])
    y = rng.uniform(moved.min(axis=0), moved.max(axis=0), size=(n, 3))
    inl = rng.permutation(n)[:max(3, int(round(ratio * n)))]
    y[inl] = moved[inl] + rng.normal(size=(len(inl), 3)) * sh["sigma"]
    return x.astype(np.float32), y.astype(np.float32)


def _problems(case, seed):
    """The (x, y, tau, k1) of a case's problems."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] != "batch":
        x, y = _problem(rng, case["shape"], case["n"], case["ratio"])
        return [(x, y, case["tau"], case["k1"])]
    out = []
    for _ in range(case["num"]):
        shape = "indoor" if rng.random() < 0.5 else "outdoor"
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        x, y = _problem(rng, shape, n, rng.uniform(0.02, 0.2))
        out.append((x, y, SHAPES[shape]["tau"], case["k1"] or SHAPES[shape]["k1"]))
    return out


def _weights(case, seed):
    """SC^2 weights of an indoor problem above the diagonal, uint16 [n, n rounded up to 8]."""
    n = case["n"]
    rng = np.random.Generator(np.random.PCG64(seed))
    x, y = (torch.from_numpy(a).cuda() for a in _problem(rng, "indoor", n, 0.05))
    g = ((torch.cdist(x, x) - torch.cdist(y, y)).abs() <= 0.1).float().fill_diagonal_(0)
    w = torch.zeros(n, (n + 7) // 8 * 8, dtype=torch.int32, device="cuda")
    w[:, :n] = torch.triu(g * (g @ g), 1).int()
    return w.to(torch.uint16)


def _samples(case, seed):
    """Features and labels of inliers and outliers, half of each, and a network some way into training."""
    rng = np.random.Generator(np.random.PCG64(seed))
    m = case["m"]
    label = (rng.random(m) < 0.5).astype(np.float32)
    feat = rng.normal(size=(m, 8)).astype(np.float32)
    feat[:, 6] = np.abs(feat[:, 6]) * 0.02 + 0.03 * label
    feat[:, 7] = np.clip(0.1 * np.abs(feat[:, 7]) + 0.5 * label, 0, 1)
    w = []
    for out, inp in ((64, 8), (128, 64), (64, 128), (1, 64)):
        w += [rng.normal(size=out * inp) * math.sqrt(2 / inp), rng.normal(size=out) * 0.05]
    w = np.concatenate(w).astype(np.float32)
    mom = (rng.normal(size=w.size) * 1e-3).astype(np.float32)
    vel = (rng.uniform(0.5, 1.5, size=w.size) * 1e-4).astype(np.float32)
    return feat, label, w, mom, vel


STEP, LR = 200, 1e-3


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "pivots":
        s.update(w=_weights(case, seed), n=case["n"], k1=case["k1"],
                 piv=torch.zeros(case["k1"], 4, dtype=torch.int32, device="cuda"),
                 count=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif kind in ("grad", "train"):
        feat, label, w, mom, vel = _samples(case, seed)
        s["net"] = trg.MLPTrainer(max_samples=case["m"])
        s["net"].set_params(w)
        s["net"].set_state(mom, vel, STEP)
        s["feat"], s["label"] = torch.from_numpy(feat).cuda(), torch.from_numpy(label).cuda()
    else:
        probs = _problems(case, seed)
        learned = case.get("learned", False)
        prm = [trg.default_params(tau, k1, tau, k2=case.get("k2", 2), scoring=case.get("scoring", trg.SCORE_IN),
                                  graph_mode=trg.GRAPH_SC2 if case.get("undirected") else trg.GRAPH_O2,
                                  proposal=trg.PROPOSAL_LEARNED if learned else trg.PROPOSAL_PLAIN)
               for _, _, tau, k1 in probs]
        s["ctx"] = trg.TurboReg(max_n=max(len(p[0]) for p in probs), max_batch=len(probs))
        if learned:
            s["ctx"].set_proposal_model(load_model())
        x, y = (np.concatenate([p[k] for p in probs]) for k in (0, 1))
        s["x"], s["y"] = (x, y) if case.get("host") else (torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
        if kind == "batch":
            s["prm"] = prm
            s["offsets"] = np.cumsum([0] + [len(p[0]) for p in probs]).astype(np.int64)
        else:
            s["prm"] = prm[0]
            if kind == "stream":
                s["slots"] = trg.ResultSlots(1)
                s["out"] = trg.turboreg_result.from_address(s["slots"].address(0).value)
    torch.cuda.synchronize()
    return s


# ---- one pass ----

def _results(rs):
    """A call's results as arrays."""
    return {"pose": np.stack([np.concatenate([r.R.ravel(), r.t]) for r in rs]),
            "score": np.array([r.score for r in rs], dtype=np.float32),
            "whole": np.array([[*r.clique, r.inlier_count, r.hypothesis, r.n_pivots, r.n_valid, r.used_fp64,
                                r.used_fallback, r.status] for r in rs], dtype=np.int32)}


def run(s):
    kind = s["kind"]
    if kind == "register":
        return _results([s["ctx"].register(s["x"], s["y"], s["prm"])])
    if kind == "stream":
        s["ctx"].register_async(s["x"], s["y"], s["prm"], s["slots"], 0)
        # the page-locked slot itself: filled when the stream gets there
        return {"pose": np.frombuffer(s["out"], np.float32, 12).reshape(1, 12),
                "score": np.frombuffer(s["out"], np.float32, 1, 88),
                "whole": np.frombuffer(s["out"], np.int32, 10, 48).reshape(1, 10)}
    if kind == "batch":
        return _results(s["ctx"].register_batched(s["x"], s["y"], s["offsets"], s["prm"]))
    if kind == "pivots":
        rc = trg.turboreg_select_pivots_noalloc(s["w"], s["n"], s["w"].shape[1], s["k1"], s["piv"], s["count"])
        if rc != trg.OK:
            raise RuntimeError(trg.status_string(rc))
        return {"pivots": s["piv"], "count": s["count"]}
    if kind == "grad":
        g, loss = s["net"].grad(s["feat"], s["label"])
        return {"grad": g, "loss": loss}
    loss = s["net"].train_step(s["feat"], s["label"], LR, want_loss=True)
    return {"weights": s["net"].get_params(), "loss": loss}


# ---- what a pass cannot do without ----

def _register_work(n, k1, k2, tau, shape):
    density = {"cube": 0.055, "indoor": 0.045, "outdoor": 0.02}[shape] * tau / SHAPES[shape]["tau"]
    edges = density * n * n / 2
    # pair distances, AND + count over the edges' rows, residuals of the hypotheses
    return 24 * n + 92, 17 * n * n / 2 + 2 * edges * n / 32 + 25 * min(k1, edges) * k2 * n


def work(case):
    kind = case["kind"]
    if kind in ("register", "stream"):
        b, f = _register_work(case["n"], case["k1"], case["k2"], case["tau"], case["shape"])
    elif kind == "batch":
        n2 = (case["n_lo"] ** 2 + case["n_lo"] * case["n_hi"] + case["n_hi"] ** 2) / 3   # mean square size
        parts = [_register_work(math.sqrt(n2), case["k1"] or SHAPES[sh]["k1"], 2, SHAPES[sh]["tau"], sh)
                 for sh in ("indoor", "outdoor")]
        b, f = (case["num"] * (parts[0][k] + parts[1][k]) / 2 for k in (0, 1))
    elif kind == "pivots":
        b, f = case["n"] ** 2 + 16 * case["k1"], 0   # the upper triangle of 16-bit weights
    else:
        p = trg.TURBOREG_MLP_PARAMS
        b, f = 36 * case["m"] + 4 * p * (1 if kind == "grad" else 7), 6 * 16960 * case["m"]
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits ----

def _exact_pose(x, y, tau, k1, k2, undirected, scoring):
    """(pose [12], score) of one problem."""
    dev = "cuda"
    n = len(x)
    tau = float(np.float32(tau))
    x, y = torch.from_numpy(x).to(dev).double(), torch.from_numpy(y).to(dev).double()
    g = torch.empty(n, n, dtype=torch.bool, device=dev)
    for a in range(0, n, 1024):
        dx = (x[a:a + 1024, None] - x[None]).square().sum(-1).sqrt()
        dy = (y[a:a + 1024, None] - y[None]).square().sum(-1).sqrt()
        g[a:a + 1024] = (dx - dy).abs() <= tau
    g.fill_diagonal_(False)
    gf = g.float()
    w = gf @ gf   # whole numbers below 2^24: exact in 32 bits
    w *= gf
    i, j = torch.triu(w, 1).nonzero(as_tuple=True)
    key = w[i, j].long() * n * n - (i * n + j)   # heavier first, then lower (i, j)
    top = key.topk(min(k1, key.numel())).indices
    i, j = i[top], j[top]
    z = torch.arange(n, device=dev)
    cl = []
    for a in range(0, len(i), 256):
        ii, jj = i[a:a + 256], j[a:a + 256]
        s = (w[ii] + w[jj]).long() + w[ii, jj].long()[:, None]
        ok = g[ii] & g[jj] if undirected else g[ii] & g[jj] & (z > jj[:, None])
        best = torch.where(ok, s * n + (n - 1 - z), -1).topk(min(k2, n), dim=1).values
        cl.append(torch.where(best >= 0, n - 1 - best % n, -1))
    cl = torch.cat(cl).T.reshape(-1)             # h = r |P| + p
    i, j = i.repeat(k2), j.repeat(k2)
    tri = torch.stack([i, j, cl.clamp(min=0)], 1)
    X, Y = x[tri], y[tri]
    mx, my = X.mean(1, keepdim=True), Y.mean(1, keepdim=True)
    u, sv, vt = np.linalg.svd(((X - mx).transpose(1, 2) @ (Y - my)).cpu().numpy())
    fix = np.ones((len(u), 3))
    fix[:, 2] = np.sign(np.linalg.det(u) * np.linalg.det(vt))
    r = torch.from_numpy(np.einsum("hji,hj,hkj->hik", vt, fix, u)).to(dev)
    t = my[:, 0] - (r @ mx[:, 0, :, None])[..., 0]
    ok = (cl >= 0) & torch.from_numpy(sv[:, 1] > 1e-12 * sv[:, 0]).to(dev)
    score = torch.empty(len(r), dtype=torch.float64, device=dev)
    for a in range(0, len(r), 256):
        e2 = (r[a:a + 256] @ x.T + t[a:a + 256, :, None] - y.T).square().sum(1)
        if scoring == trg.SCORE_IN:
            score[a:a + 256] = (e2 <= tau * tau).sum(1)
        elif scoring == trg.SCORE_MAE:
            score[a:a + 256] = e2.sqrt().clamp(max=tau).mean(1)
        else:
            score[a:a + 256] = e2.clamp(max=tau * tau).mean(1)
    rank = torch.where(ok, score if scoring == trg.SCORE_IN else -score, -math.inf)
    h = int((rank == rank.max()).nonzero()[0])
    return np.concatenate([r[h].cpu().numpy().ravel(), t[h].cpu().numpy()]), float(score[h])


def _exact_grad(feat, label, w):
    dims, at, p = ((64, 8), (128, 64), (64, 128), (1, 64)), 0, []
    w = torch.from_numpy(w).cuda().double().requires_grad_()
    for out, inp in dims:
        p.append((w[at:at + out * inp].reshape(out, inp), w[at + out * inp:at + out * inp + out]))
        at += out * inp + out
    h = torch.from_numpy(feat).cuda().double()
    for a, b in p[:-1]:
        h = torch.relu(h @ a.T + b)
    z = (h @ p[-1][0].T + p[-1][1])[:, 0]
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, torch.from_numpy(label).cuda().double())
    loss.backward()
    return w.grad.cpu().numpy(), float(loss)


def exact(case, seed):
    kind = case["kind"]
    if kind == "pivots" or case.get("learned"):
        return None   # whole numbers; pivots ranked through a 16-bit network
    if kind in ("grad", "train"):
        feat, label, w, mom, vel = _samples(case, seed)
        g, loss = _exact_grad(feat, label, w)
        if kind == "grad":
            return {"grad": g, "loss": loss}
        mom, vel = 0.9 * mom + 0.1 * g, 0.999 * vel + 0.001 * g * g   # Adam
        step = STEP + 1
        return {"weights": w - LR * (mom / (1 - 0.9 ** step)) / (np.sqrt(vel / (1 - 0.999 ** step)) + 1e-8), "loss": loss}
    got = [_exact_pose(*p, case.get("k2", 2), case.get("undirected", False), case.get("scoring", trg.SCORE_IN))
           for p in _problems(case, seed)]
    return {"pose": np.stack([p for p, _ in got]), "score": np.array([s for _, s in got]), "whole": None}
