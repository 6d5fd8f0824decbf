"""Performance cases: the work a user of this package has it do, through its
public entry points, over the range of sizes the repository's configurations,
tests and benchmark use.

Colonies (`kind` "colony"): a context is created in prepare(), as a program
that runs many iterations does once; one pass is `iters` iterations followed by
reading the best tour and length of every instance. The launch shape is the
library's default. "solve" is the whole call from host coordinates: create,
iterate, read the best tour, close. The learned prior has three kinds: "prior"
(features and scores of one instance), "score" (the network alone on a large
feature array) and "train" (one mini-batch: gradients and an Adam step).

The relaxed construction mode is not among the cases: its results depend on
timing, so two runs cannot be compared.
"""
import math
import random

import numpy as np
import torch

from paper_1605_02669_gb300 import acs, instances, prior

MATRIX, SPM = "matrix", "spm"


def _colony(name, sizes, layout, m, memory, iters, **more):
    case = {"name": name, "kind": "colony", "sizes": sizes, "layout": layout, "m": m,
            "memory": memory, "iters": iters, "slots": 8, "cl": 32, "q0": 0.9, "period": 1,
            "side": 10000, "keep": 0}
    case.update(more)
    return case


def listed():
    return [
        # one n=198 instance, 32 ants, one iteration at a time (a program that
        # watches every iteration): the smallest call, bound by latency
        _colony("small_matrix", "198", "uniform", 32, MATRIX, 1),
        # the paper's scale on both pheromone memories: two clustered instances
        # in one context, 128 ants, a few iterations between looks at the best
        _colony("paper_matrix", "1002,2392", "clustered", 128, MATRIX, 5),
        _colony("paper_spm", "1002,2392", "clustered", 128, SPM, 5),
        # the whole call from coordinates: context creation (candidate lists,
        # nearest-neighbour tour, tables), ten iterations, the best tour
        _colony("solve_paper", "2392", "clustered", 128, SPM, 10, kind="solve"),
        # 256 instances of uneven n, half uniform and half clustered, 64 ants:
        # the batched configuration on both memories
        _colony("batch_matrix", "mixed:256:100:2500", "mixed", 64, MATRIX, 2),
        _colony("batch_spm", "mixed:256:100:2500", "mixed", 64, SPM, 2),
        # large instances: eight of 10000 and eight of 20000 nodes, 256 ants
        _colony("large_matrix", "8x10000,8x20000", "uniform", 256, MATRIX, 1, side=100000),
        _colony("large_spm", "8x10000,8x20000", "uniform", 256, SPM, 1, side=100000),
        # replicas of one instance whose lists a prior has pruned to 16: lists
        # run out sooner, so the full-scan rule works more
        _colony("pruned_replicas", "rep:5:5000", "uniform", 128, MATRIX, 2, keep=16),
        # scoring one instance before pruning its lists: features and scores
        {"name": "prior_instance", "kind": "prior", "n": 5000},
        # scoring a large set of edges
        {"name": "score_large", "kind": "score", "rows": 1 << 24},
        # one training step at the prior's default mini-batch
        {"name": "train_step", "kind": "train", "total": 300001, "batch": 4096},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over the listed ones' range."""
    r = rng.random()
    if r < 0.06:
        return {"kind": "score", "rows": _log_uniform(rng, 1000, 1 << 24)}
    if r < 0.12:
        total = _log_uniform(rng, 20000, 2000000)
        return {"kind": "train", "total": total, "batch": min(total, _log_uniform(rng, 256, 65536))}
    if r < 0.18:
        return {"kind": "prior", "n": _log_uniform(rng, 200, 6000)}
    m = _log_uniform(rng, 8, 256)
    hi = _log_uniform(rng, 100, 20000)
    memory = rng.choice([MATRIX, SPM])
    keep = rng.choice([0, 0, 0, 16])
    more = {"slots": rng.choice([4, 8, 8, 16]), "cl": rng.choice([20, 32, 32, 32]),
            "q0": rng.choice([0.5, 0.9, 0.9, 0.98]), "period": rng.choice([1, 1, 1, 4]),
            "side": 10000 if hi < 8000 else 100000, "keep": keep if hi < 8000 else 0}
    if more["keep"]:
        more["cl"] = 32
    if rng.random() < 0.2:
        return _drawn(_colony("", str(hi), rng.choice(["uniform", "clustered"]), m, memory,
                              rng.randint(1, 10) if hi < 5000 else 1, kind="solve", **more))
    B = _log_uniform(rng, 1, max(1, min(256, 200000 // hi)))
    if B == 1:
        sizes, layout = str(hi), rng.choice(["uniform", "clustered"])
    elif B <= 8 and rng.random() < 0.3:
        sizes, layout = "rep:%d:%d" % (B, hi), "uniform"
    else:
        sizes, layout = "mixed:%d:%d:%d" % (B, max(40, int(hi * rng.uniform(0.1, 0.9))), hi), "mixed"
    iters = 1 if hi > 3000 or B > 64 else rng.randint(1, 4)
    return _drawn(_colony("", sizes, layout, m, memory, iters, **more))


def _drawn(case):
    del case["name"]
    return case


def _size_list(case):
    """Nodes of every instance: they belong to the case, the seed only draws coordinates."""
    s = case["sizes"]
    if s.startswith("rep:"):
        _, k, n = s.split(":")
        return [int(n)] * int(k)
    if s.startswith("mixed:"):
        _, k, lo, hi = s.split(":")
        return [int(n) for n in np.random.default_rng(3).integers(int(lo), int(hi) + 1, int(k))]
    out = []
    for part in s.split(","):
        k, _, n = part.rpartition("x")
        out += [int(n)] * int(k or 1)
    return out


def _coords(case, seed):
    """(xy [sum n, 2], offsets [B + 1]): seeded instances."""
    sizes = _size_list(case)
    if case["layout"] == "mixed":
        kinds = ["clustered" if b % 2 else "uniform" for b in range(len(sizes))]
        return instances.batch(sizes, kinds, side=case["side"], seed=seed)
    if case["sizes"].startswith("rep:"):
        one = _points(sizes[0], case, seed, 0)
        parts = [one] * len(sizes)
    else:
        parts = [_points(n, case, seed, 1 + b) for b, n in enumerate(sizes)]
    return np.concatenate(parts), np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _points(n, case, seed, stream):
    if case["layout"] == "clustered":
        return instances.clustered(n, side=case["side"], sigma=0.03 * case["side"], seed=seed, stream=stream)
    return instances.uniform(n, side=case["side"], seed=seed, stream=stream)


def _params(case, seed):
    return acs.params(m=case["m"], cl=case["cl"], q0=case["q0"],
                      memory=acs.ACS_MEM_MATRIX if case["memory"] == MATRIX else acs.ACS_MEM_SPM,
                      spm_slots=case["slots"], local_period=case["period"], seed=1 + seed)


def _distance_prior():
    """A network that prefers short edges, as a trained one does: the score
    falls with the distance relative to the list's mean."""
    P = {k: np.zeros(shape, np.float32) for k, (_, shape) in prior.LAYOUT.items()}
    P["W1"][1, 0] = 1.0
    P["W2"][0, 0] = 1.0
    P["w3"][0] = -2.0
    P["b3"][0] = 2.0
    return torch.from_numpy(prior.pack(P)).cuda()


def _net(seed):
    """Weights of a trained network's size: all layers at work, some units off."""
    g = np.random.default_rng([int(seed), 5])
    P = {k: (0.3 * g.standard_normal(shape)).astype(np.float32) for k, (_, shape) in prior.LAYOUT.items()}
    return torch.from_numpy(prior.pack(P)).cuda()


def _bf16_features(rows, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 17)
    x = torch.randn((rows, 8), generator=g, device="cuda", dtype=torch.float32)
    return x.to(torch.bfloat16).view(torch.int16)


def _train_inputs(case, seed):
    feat = _bf16_features(case["total"], seed)
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 29)
    label = torch.randint(0, 9, (case["total"],), generator=g, device="cuda").float() / 8
    r = random.Random(int(seed))
    a = r.randrange(1, case["total"])
    while math.gcd(a, case["total"]) != 1:
        a = r.randrange(1, case["total"])
    return prior.init_params(seed), feat, label, a, r.randrange(case["total"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "score":
        return {"kind": kind, "net": _net(seed), "feat": _bf16_features(case["rows"], seed)}
    if kind == "train":
        net, feat, label, a, c = _train_inputs(case, seed)
        return {"kind": kind, "trainer": prior.Trainer(net), "feat": feat, "label": label,
                "batch": case["batch"], "a": a, "c": c}
    if kind == "prior":
        xy = instances.clustered(case["n"], seed=seed)
        return {"kind": kind, "net": _net(seed), "colony": acs.Colony(xy, acs.params(m=8, cl=32, seed=1))}
    xy, off = _coords(case, seed)
    p = _params(case, seed)
    if kind == "solve":
        return {"kind": kind, "xy": xy, "p": p, "iters": case["iters"],
                "net": _distance_prior() if case["keep"] else None, "keep": case["keep"]}
    col = acs.Colony(xy, p, offsets=off)
    if case["keep"]:
        prior.apply(col, _distance_prior(), keep=case["keep"])
    return {"kind": kind, "colony": col, "iters": case["iters"]}


def _best(col):
    tours, lens = zip(*(col.best(b) for b in range(len(col.sizes))))
    return {"tours": np.concatenate(tours), "lengths": np.array(lens, np.int64)}


def run(state):
    kind = state["kind"]
    if kind == "colony":
        state["colony"].run(state["iters"])
        return _best(state["colony"])
    if kind == "solve":
        col = acs.Colony(state["xy"], state["p"])
        if state["net"] is not None:
            prior.apply(col, state["net"], keep=state["keep"])
        col.run(state["iters"])
        out = _best(col)
        col.close()
        return out
    if kind == "prior":
        feat = prior.colony_features(state["colony"])
        return {"features": feat, "scores": prior.score(state["net"], feat)}
    if kind == "score":
        return {"scores": prior.score(state["net"], state["feat"])}
    tr = state["trainer"]
    loss = tr.batch(state["feat"], state["label"], 0, state["batch"], state["a"], state["c"])
    return {"loss": loss, "grad": tr.grad, "params": tr.params, "m": tr.m, "v": tr.v}


def work(case):
    """Bytes and operations one pass cannot do without.

    Colony, per iteration: every candidate row (32 nodes, 32 weights) and the
    candidates' trails read once, every ant's tour written once; a multiply and
    a compare per candidate of every ant step. "solve" adds the coordinates and
    one distance (about ten operations) for every pair of nodes."""
    kind = case["kind"]
    layers = 2 * (8 * 64 + 64 * 64 + 64)
    if kind == "score":
        return {"bytes": 20 * case["rows"], "flops": layers * case["rows"]}
    if kind == "train":
        return {"bytes": 20 * case["batch"] + 7 * 4 * acs.ACS_MLP_PARAMS, "flops": 3 * layers * case["batch"]}
    if kind == "prior":
        rows = 32 * case["n"]
        return {"bytes": 8 * case["n"] + 4 * rows + 20 * rows, "flops": layers * rows}
    n = sum(_size_list(case))
    state = 128 if case["memory"] == MATRIX else 8 * case["slots"] + 4
    nbytes = case["iters"] * (n * (256 + state) + 4 * case["m"] * n)
    flops = case["iters"] * 64 * case["m"] * n
    if kind == "solve":
        nbytes += 8 * n
        flops += 10 * n * n
    return {"bytes": nbytes, "flops": flops}


# ---- the values in 64 bits, by plain torch and numpy

def _unpack64(vec):
    v = vec.detach().cpu().double() if isinstance(vec, torch.Tensor) else torch.as_tensor(np.asarray(vec, np.float64))
    return {k: v[o:o + int(np.prod(shape))].reshape(shape).cuda() for k, (o, shape) in prior.LAYOUT.items()}


def _layers64(P, x):
    h1 = torch.relu(x @ P["W1"] + P["b1"])
    h2 = torch.relu(h1 @ P["W2"] + P["b2"])
    return h1, h2, h2 @ P["w3"] + P["b3"]


def _scores64(net, x):
    P, out = _unpack64(net), torch.empty(x.shape[0], dtype=torch.float64, device="cuda")
    for i in range(0, x.shape[0], 1 << 20):
        out[i:i + (1 << 20)] = torch.sigmoid(_layers64(P, x[i:i + (1 << 20)].double())[2])
    return out


def _features64(xy):
    """The eight features of every candidate edge of one instance, cl = 32."""
    n, p = xy.shape[0], xy.astype(np.float64)
    d = np.floor(np.sqrt(((p[:, None, :] - p[None, :, :]) ** 2).sum(-1)) + 0.5)
    np.fill_diagonal(d, np.inf)
    nn = np.argsort(d, axis=1, kind="stable")[:, :32]
    dist = np.take_along_axis(d, nn, 1)
    mean, last = np.maximum(dist.mean(1), 1.0), np.maximum(dist[:, -1], 1.0)
    indeg = np.bincount(nn.reshape(-1), minlength=n)
    rank = np.full((n, n), 32, np.int8)
    np.put_along_axis(rank, nn, np.arange(32, dtype=np.int8)[None, :].repeat(n, 0), 1)
    f = np.zeros((n, 32, 8))
    f[..., 0] = np.arange(32) / 32.0
    f[..., 1] = dist / mean[:, None]
    f[..., 2] = dist / last[:, None]
    f[..., 3] = (p[nn, 0] - p[:, None, 0]) / last[:, None]
    f[..., 4] = (p[nn, 1] - p[:, None, 1]) / last[:, None]
    f[..., 5] = rank[nn, np.arange(n)[:, None]] / 32.0
    f[..., 6] = dist / last[nn]
    f[..., 7] = indeg[nn] / 32.0
    return torch.from_numpy(f.reshape(-1, 8)).cuda()


def exact(case, seed):
    kind = case["kind"]
    if kind == "score":
        return {"scores": _scores64(_net(seed), _bf16_features(case["rows"], seed).view(torch.bfloat16))}
    if kind == "prior":
        xy = instances.clustered(case["n"], seed=seed)
        return {"features": None, "scores": _scores64(_net(seed), _features64(xy))}
    if kind == "train":
        net, feat, label, a, c = _train_inputs(case, seed)
        P, nb = _unpack64(net), case["batch"]
        rows = torch.tensor([(a * i + c) % case["total"] for i in range(nb)], device="cuda")
        x, y = feat[rows].view(torch.bfloat16).double(), label[rows].double()
        h1, h2, z = _layers64(P, x)
        loss = (torch.clamp(z, min=0) - z * y + torch.log1p(torch.exp(-z.abs()))).mean()
        dz = (torch.sigmoid(z) - y) / nb
        dh2 = dz[:, None] * P["w3"] * (h2 > 0)
        dh1 = (dh2 @ P["W2"].T) * (h1 > 0)
        grad = torch.cat([(x.T @ dh1).reshape(-1), dh1.sum(0), (h1.T @ dh2).reshape(-1), dh2.sum(0),
                          h2.T @ dz, dz.sum()[None]])
        # Adam's first step: the bias corrections cancel the decay factors
        vec = torch.as_tensor(np.asarray(net, np.float64)).cuda()
        return {"loss": loss[None], "grad": grad, "params": vec - 1e-3 * grad / (grad.abs() + 1e-8),
                "m": 0.1 * grad, "v": 0.001 * grad * grad}
    return None   # tours and lengths: whole numbers
