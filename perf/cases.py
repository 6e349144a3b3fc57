"""Performance cases of the library: what its users run, at the sizes they run it.

Graphs come from the repository's own workloads (Erdos-Renyi, Barabasi-Albert
and R-MAT; the small, the heavy-tailed and the social-network shapes, and the
uneven batch), at their sizes or scaled so that one pass stays below a second.
Every case goes through the Python binding's public calls.

``exact`` states in plain torch, in 64 bits, what a pass returns: the sampled
estimates (for small graphs) by popping all cycles of all samples at once, the
network and its gradients in FP64, the linear solve by conjugate gradients.
"""
import math

import numpy as np
import torch

from paper_2311_10290_gb300 import cv, inputs
from paper_2311_10290_gb300.lap import (LAP_MLP_PARAMS, LAP_OPT_PATHS, LapBatch, LapGraph, lap_mlp_forward,
                                        lap_mlp_loss_grad)

WORKSPACE = 16 << 30            # Wilson-state workspace lent to a handle, at most


def listed():
    return [
        # All-node ECC and Kemeny's constant on the small workload: 10,000
        # samples of a 1000-node graph; a latency-bound call.
        {"name": "er_1k", "kind": "ecc", "family": "er", "n": 1000, "deg": 10.0, "samples": 10000, "form": "plain"},
        # A quick look at a mid-size graph with few samples: the smallest
        # sampling call, an odd sample count.
        {"name": "rmat_16k_quick", "kind": "ecc", "family": "rmat", "n": 16384, "deg": 16.0, "samples": 257,
         "form": "plain"},
        # The README's call: 16,384 samples of a 100,000-node graph.
        {"name": "ba_100k", "kind": "ecc", "family": "ba", "n": 100000, "deg": 10.0, "samples": 16384, "form": "plain"},
        # The heavy-tailed workload's graph (10^6 nodes, 5 * 10^6 edges); the
        # number of samples of a fraction of its time-to-accuracy run.
        {"name": "ba_1m", "kind": "ecc", "family": "ba", "n": 1000000, "deg": 10.0, "samples": 4096, "form": "plain"},
        # The social-network shape, with arrays larger than the L2 cache.
        {"name": "rmat_1m", "kind": "ecc", "family": "rmat", "n": 1 << 20, "deg": 32.0, "samples": 2048, "form": "plain"},
        # The control variate on the loop-included paths.
        {"name": "ba_200k_cv_paths", "kind": "ecc", "family": "ba", "n": 200000, "deg": 10.0, "samples": 2048,
         "form": "cv_paths"},
        # Many uneven graphs in one launch.
        {"name": "batch_24", "kind": "batch", "graphs": 24, "n_lo": 1000, "n_hi": 100000, "samples": 512},
        # Features and training targets of one training graph of the control variate.
        {"name": "targets_30k", "kind": "targets", "family": "ba", "n": 30011, "deg": 12.0, "samples": 512, "reps": 16},
        # Loss and gradient of one minibatch of the network's training.
        {"name": "mlp_train_8k", "kind": "mlp_train", "rows": 8192},
        # The network on every node of a large graph.
        {"name": "mlp_predict_1m", "kind": "mlp_predict", "rows": 1000003},
        # Exact row sums of L_v^{-1} (ground truth of the large graphs).
        {"name": "solve_300k", "kind": "solve", "family": "ba", "n": 300000, "deg": 10.0},
        # The SpanTree estimators.
        {"name": "spantree_50k", "kind": "spantree", "family": "ba", "n": 50000, "deg": 8.0, "trees": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ecc", "ecc", "ecc", "batch", "targets", "mlp_train", "mlp_predict", "solve", "spantree"])
    deg = round(rng.uniform(6.0, 32.0), 1)
    # Walks to the root of a large Erdos-Renyi graph are long (its highest
    # degree is low): that family stays below 20,000 nodes.
    family = rng.choice(["er", "ba", "rmat"])
    top = 20000 if family == "er" else 1000000
    if kind == "ecc":
        n = _log(rng, 700, top)
        # At most a quarter of the largest case's node visits.
        samples = _log(rng, 64, max(65, min(16384, int(1.0e9 / n))))
        return {"kind": kind, "family": family, "n": n, "deg": deg, "samples": samples,
                "form": rng.choice(["plain", "plain", "paths", "cv", "cv_paths"])}
    if kind == "batch":
        return {"kind": kind, "graphs": rng.randint(3, 40), "n_lo": 1000, "n_hi": _log(rng, 3000, 100000),
                "samples": _log(rng, 64, 512)}
    if kind == "targets":
        return {"kind": kind, "family": family, "n": _log(rng, 5000, min(60000, top)), "deg": deg, "samples": 512, "reps": 16}
    if kind in ("mlp_train", "mlp_predict"):
        return {"kind": kind, "rows": _log(rng, 999, 1000000)}
    if kind == "solve":
        return {"kind": kind, "family": family, "n": _log(rng, 3000, 300000), "deg": deg}
    return {"kind": kind, "family": family, "n": _log(rng, 2000, min(50000, top)), "deg": deg, "trees": _log(rng, 32, 512)}


# ------------------------------------------------------------------ inputs

def _rmat_gpu(n, deg, seed):
    """Largest component of an R-MAT graph (0.57, 0.19, 0.19, 0.05) with about
    deg / 2 * n generated edges, as int32 CSR tensors on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(1 + seed)
    scale = max(4, int(math.ceil(math.log2(n))))
    m = int(round(deg / 2 * n))
    s = torch.zeros(m, dtype=torch.int64, device="cuda")
    t = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(m, device="cuda", generator=gen)
        down = r >= 0.76                                   # quadrants c, d: the source's bit
        right = ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)   # quadrants b, d: the target's bit
        s = 2 * s + down
        t = 2 * t + right
    size = 1 << scale
    keep = s != t
    s, t = s[keep], t[keep]
    key = torch.unique(torch.cat([s * size + t, t * size + s]))
    s, t = key // size, key % size
    # Components: every node takes the smallest label around it until none changes.
    lab = torch.arange(size, device="cuda")
    while True:
        new = lab.scatter_reduce(0, s, lab[t], "amin")
        new = torch.minimum(new, new[new])
        if bool((new == lab).all()):
            break
        lab = new
    big = torch.bincount(lab, minlength=size).argmax()
    inside = lab == big
    ids = torch.cumsum(inside, 0) - 1
    keep = inside[s]
    s, t = ids[s[keep]], ids[t[keep]]
    nn = int(inside.sum())
    rp = torch.zeros(nn + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(s, minlength=nn), 0)
    return rp.int(), t.int()


def _graph(case, seed):
    """(row_ptr, col) of the case's graph: CUDA tensors (R-MAT) or host arrays.
    A largest component's size depends on its graph's seed, so those families
    keep one graph per case and take `seed` for the samples alone."""
    n, deg = case["n"], case["deg"]
    if case["family"] == "rmat":
        return _rmat_gpu(n, deg, 0)
    if case["family"] == "er":
        g = inputs.er(n, min(1.0, deg / max(n - 1, 1)), seed=0, lcc=True)
    else:
        g = inputs.ba(n, max(1, int(round(deg / 2))), seed=seed)
    return g.row_ptr, g.col


def _handle(case, seed, paths=False):
    rp, col = _graph(case, seed)
    n = len(rp) - 1
    G = LapGraph(rp, col, workspace_bytes=min(WORKSPACE, 8 * n * 152 * 2048))
    if paths:
        G.set_option(LAP_OPT_PATHS, 1)
    G.set_root()
    return G


def _mlp_inputs(rows, seed):
    """Packed parameters, features and targets with the spread of the node
    features (logarithms, shares) and of mean visits and hitting times."""
    gen = torch.Generator(device="cuda").manual_seed(7 + seed)
    rnd = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)  # noqa: E731
    params = torch.cat([0.5 * rnd(64 * 8), 0.1 * rnd(64), 0.177 * rnd(64 * 64), 0.1 * rnd(64),
                        0.125 * rnd(2 * 64), 0.1 * rnd(2)]).contiguous()
    x = rnd(rows, 8)
    t = 1.0 + 0.3 * rnd(rows, 2)
    return params, x.contiguous(), t.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ecc":
        form = case["form"]
        G = _handle(case, seed, paths=form in ("paths", "cv_paths"))
        st = {"kind": kind, "G": G, "samples": case["samples"], "seed": 1000003 + seed, "cv": form.startswith("cv"),
              "counts": G.n <= 20000, "ecc": torch.empty(G.n, dtype=torch.float64, device="cuda"),
              "ldiag": torch.empty(G.n, dtype=torch.float64, device="cuda")}
        if st["cv"]:
            # Potentials with the network's shape: about 1.2 / d, and a hitting
            # time near 2m / d_max, both with a spread.
            gen = torch.Generator(device="cuda").manual_seed(11 + seed)
            d = torch.from_numpy(np.diff(G.row_ptr_host).astype(np.float64)).cuda()
            noise = torch.rand(2, G.n, device="cuda", dtype=torch.float64, generator=gen)
            G.cv_set_potentials((1.1 + 0.2 * noise[0]) / d, d.sum() / d.max() * (0.8 + 0.4 * noise[1]))
        return st
    if kind == "batch":
        spec = inputs.batch_spec(case["graphs"], case["n_lo"], case["n_hi"], seed0=0)
        gs = inputs.batch_graphs(spec)
        B = LapBatch([(g.row_ptr, g.col) for g in gs], workspace_bytes=4 << 30)
        return {"kind": kind, "B": B, "samples": case["samples"], "seed": 1000003 + seed,
                "ecc": torch.empty(B.total_n, dtype=torch.float64, device="cuda")}
    if kind == "targets":
        return {"kind": kind, "G": _handle(case, seed), "samples": case["samples"], "reps": case["reps"],
                "seed": 1000003 + seed}
    if kind in ("mlp_train", "mlp_predict"):
        params, x, t = _mlp_inputs(case["rows"], seed)
        return {"kind": kind, "rows": case["rows"], "params": params, "x": x, "t": t,
                "y": torch.empty(case["rows"], 2, device="cuda"),
                "grad": torch.empty(LAP_MLP_PARAMS, device="cuda"), "loss": torch.empty(1, device="cuda")}
    if kind == "solve":
        G = _handle(case, seed)
        return {"kind": kind, "G": G, "b": _rhs(G.n, seed)}
    return {"kind": kind, "G": _handle(case, seed), "trees": case["trees"], "seed": 1000003 + seed}


def _rhs(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(13 + seed)
    return 1.0 + 0.5 * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)


# ------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "batch":
        B = state["B"]
        B.run(state["samples"], state["seed"])
        return {"ecc": B.ecc(out=state["ecc"]), "kemeny": B.kemeny()}
    if kind == "mlp_train":
        lap_mlp_loss_grad(state["params"], state["x"], state["t"], state["rows"], 1.0, 1.0, state["grad"],
                          state["loss"])
        return {"grad": state["grad"], "loss": state["loss"]}
    if kind == "mlp_predict":
        lap_mlp_forward(state["params"], state["x"], state["rows"], state["y"])
        return {"y": state["y"]}
    G = state["G"]
    if kind == "solve":
        return {"x": G.lv_solve(state["b"], rtol=1e-10)[0]}
    G.set_root()
    if kind == "targets":
        features, targets, _ = cv.training_targets(G, state["samples"], state["reps"], state["seed"])
        return {"features": features, "targets": targets}
    if kind == "spantree":
        G.spantree_sample(state["trees"], state["seed"])
        ldiag, ecc, kemeny = G.spantree_estimates()
        return {"ldiag": ldiag, "ecc": ecc, "kemeny": kemeny}
    G.sample(state["samples"], state["seed"])
    if state["cv"]:
        _, ecc, kemeny, m2 = G.cv_estimates(0.9, 0.8, ecc_out=state["ecc"])
        return {"ecc": ecc, "kemeny": kemeny, "m2": m2}
    out = {"ecc": G.ecc(out=state["ecc"]), "ldiag": G.ldiag(out=state["ldiag"]), "kemeny": G.kemeny()}
    if state["counts"]:
        out["cnt1"], out["cnt2"], out["sums"] = (a.view(np.int64) for a in G.counts())
    return out


def work(case):
    """Bytes and operations a pass cannot do without.  A sampled Wilson run
    visits every node at least once: its row record (8 B), one column entry
    (4 B) and one state byte written; a draw is about 80 integer operations."""
    kind = case["kind"]
    if kind in ("mlp_train", "mlp_predict"):
        r, macs = case["rows"], 8 * 64 + 64 * 64 + 64 * 2
        if kind == "mlp_train":
            return {"bytes": 4.0 * (r * (8 + 2) + 2 * LAP_MLP_PARAMS), "flops": 6.0 * macs * r}
        return {"bytes": 4.0 * (r * (8 + 2) + LAP_MLP_PARAMS), "flops": 2.0 * macs * r}
    if kind == "batch":
        # Mean of n log-uniform in [n_lo, n_hi].
        lo, hi = case["n_lo"], case["n_hi"]
        visits = case["graphs"] * case["samples"] * (hi - lo) / math.log(hi / lo)
        return {"bytes": 13.0 * visits, "flops": 80.0 * visits}
    n, deg = case["n"], case["deg"]
    if kind == "solve":
        # About 30 iterations on these graphs, each reading the columns and
        # six vectors.
        return {"bytes": 30.0 * n * (4 * deg + 8 + 6 * 8), "flops": 30.0 * n * (deg + 12)}
    draws = case["trees"] if kind == "spantree" else case["samples"]
    visits = float(n) * draws
    if kind == "targets":
        return {"bytes": 13.0 * visits + 10.0 * n * (4 * deg + 16), "flops": 80.0 * visits}
    if kind == "spantree":
        return {"bytes": 21.0 * visits, "flops": 90.0 * visits}
    return {"bytes": 13.0 * visits, "flops": 80.0 * visits}


# ------------------------------------------------------------------ 64-bit statements

_M32 = 0xFFFFFFFF


def _mulhilo(a, b):
    """High and low 32 bits of a * b (a: a constant below 2^32, b: int64 tensor)."""
    return (a * (b >> 16) + ((a * (b & 0xFFFF)) >> 16)) >> 16, (a * b) & _M32


def _philox(c0, c1, c2, c3, seed):
    """Low 64 bits (low word, high word) of Philox4x32-10 blocks (SC'11)."""
    k0, k1 = seed & _M32, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c0)
        h2, l2 = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h2 ^ c1 ^ k0, l2, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1


def _below(x, r):
    """High 64 bits of the 64-bit x = (low, high) times r (< 2^31)."""
    lo, hi = x
    low = (r * (lo >> 16) + ((r * (lo & 0xFFFF)) >> 16)) >> 16
    return (hi * r + low) >> 32


def _wilson_visits(rp, col, root, first, count, seed):
    """Visits of every node in samples first .. first + count - 1: all cycles of
    all samples' arrows are popped at once until none is left (the popped
    cycles do not depend on the order)."""
    n = len(rp) - 1
    deg = rp[1:] - rp[:-1]
    node = torch.arange(n, device="cuda")
    i = torch.arange(first, first + count, device="cuda")
    z = torch.zeros((), dtype=torch.int64, device="cuda")

    def arrows(u, k, ii):
        return col[rp[u] + _below(_philox(u, k, ii, z, seed), deg[u])]

    uu, ii = node.repeat(count), i.repeat_interleave(n)
    nxt = arrows(uu, torch.zeros_like(uu), ii).view(count, n)
    nxt[:, root] = root
    k = torch.zeros((count, n), dtype=torch.int64, device="cuda")
    total = torch.full((n,), count, dtype=torch.int64, device="cuda")
    total[root] = 0
    y1 = count * (n - 1)
    live = torch.arange(count, device="cuda")
    while live.numel():
        f = nxt[live]
        for _ in range(max(1, math.ceil(math.log2(n)))):
            f = f.gather(1, f)
        on = torch.zeros_like(f, dtype=torch.bool).scatter_(1, f, True)   # the cycles' nodes and the root
        on[:, root] = False
        rows, us = on.nonzero(as_tuple=True)
        if rows.numel() == 0:
            break
        s = live[rows]
        k[s, us] += 1
        nxt[s, us] = arrows(us, k[s, us], i[s])
        total += on.sum(0)
        y1 += int(rows.numel())
        live = live[on.any(1)]
    return total, y1


def _walks(rp, col, root, start, count, seed, kind, passes):
    """Absorbed walks from `start` ([count]): adds their passes, returns the total length."""
    deg = rp[1:] - rp[:-1]
    z = torch.zeros((), dtype=torch.int64, device="cuda")
    i = torch.arange(count, device="cuda")
    u, t, length = start, 0, 0
    while True:
        keep = u != root
        u, i = u[keep], i[keep]
        if u.numel() == 0:
            return length
        t += 1
        length += int(u.numel())
        passes += torch.bincount(u, minlength=passes.numel())
        u = col[rp[u] + _below(_philox(torch.full_like(u, t), z, i, z + kind, seed), deg[u])]


def _exact_plain(case, seed):
    """The plain estimates of one graph from its samples' counts."""
    rp, col = _graph(case, seed)
    rp = torch.as_tensor(rp, device="cuda").long()
    col = torch.as_tensor(col, device="cuda").long()
    n, arcs, omega, key = len(rp) - 1, int(rp[-1]), case["samples"], 1000003 + seed
    deg = rp[1:] - rp[:-1]
    root = int((deg == deg.max()).nonzero()[0])
    cnt1 = torch.zeros(n, dtype=torch.int64, device="cuda")
    y1 = 0
    step = max(1, int(4e6 / n))
    for first in range(0, omega, step):
        c, y = _wilson_visits(rp, col, root, first, min(step, omega - first), key)
        cnt1 += c
        y1 += y
    i = torch.arange(omega, device="cuda")
    z = torch.zeros((), dtype=torch.int64, device="cuda")
    cnt2 = torch.zeros(n, dtype=torch.int64, device="cuda")
    start = _below(_philox(z, z, i, z + 1, key), torch.tensor(n, device="cuda"))
    _walks(rp, col, root, start, omega, key, 1, cnt2)
    start = col[_below(_philox(z, z, i, z + 2, key), torch.tensor(arcs, device="cuda"))]
    y2 = _walks(rp, col, root, start, omega, key, 2, torch.zeros_like(cnt2))
    v1, v2 = (c.double() / (omega * deg.double()) for c in (cnt1, cnt2))
    mean = v2.sum() / n
    ldiag = v1 - 2.0 * v2 + mean
    ldiag[root] = mean
    return {"ecc": (n - 1) / (n * ldiag + ldiag.sum()), "ldiag": ldiag, "kemeny": (y1 - y2) / omega,
            "cnt1": None, "cnt2": None, "sums": None}


def _exact_network(case, seed):
    """The network (no rounding to 16 bits) and its mean-square gradients in FP64."""
    params, x, t = (v.double() for v in _mlp_inputs(case["rows"], seed))
    params.requires_grad_(case["kind"] == "mlp_train")
    sizes = [64 * 8, 64, 64 * 64, 64, 2 * 64, 2]
    w1, b1, w2, b2, w3, b3 = params.split(sizes)
    h = torch.relu(x @ w1.view(64, 8).T + b1)
    h = torch.relu(h @ w2.view(64, 64).T + b2)
    y = h @ w3.view(2, 64).T + b3
    if case["kind"] == "mlp_predict":
        return {"y": y}
    loss = ((y - t) ** 2).sum() / case["rows"]
    loss.backward()
    return {"grad": params.grad, "loss": loss.detach().reshape(1)}


def _exact_solve(case, seed):
    """L_v x = b by conjugate gradients in FP64, to a residual far below the case's."""
    rp, col = _graph(case, seed)
    rp = torch.as_tensor(rp, device="cuda").long()
    col = torch.as_tensor(col, device="cuda").long()
    n = len(rp) - 1
    deg = rp[1:] - rp[:-1]
    root = int((deg == deg.max()).nonzero()[0])
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    d = deg.double()

    def mul(x):
        y = d * x - torch.zeros_like(x).index_add_(0, row, x[col])
        y[root] = 0.0
        return y

    b = _rhs(n, seed)
    b[root] = 0.0
    x = torch.zeros_like(b)
    r, p = b.clone(), b / d
    rz = (r * p).sum()
    for _ in range(10000):
        q = mul(p)
        a = rz / (p * q).sum()
        x, r = x + a * p, r - a * q
        if float(r.norm() / b.norm()) < 1e-14:
            break
        z = r / d
        new = (r * z).sum()
        p, rz = z + (new / rz) * p, new
    return {"x": x}


def _exact_features(case, seed):
    """The node features in FP64 (the targets come from random walks: None)."""
    rp, col = _graph(case, seed)
    rp = torch.as_tensor(rp, device="cuda").long()
    col = torch.as_tensor(col, device="cuda").long()
    n = len(rp) - 1
    deg = rp[1:] - rp[:-1]
    d = deg.double()
    root = int((deg == deg.max()).nonzero()[0])
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    around = lambda v: torch.zeros_like(d).index_add_(0, row, v[col])  # noqa: E731
    hops = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    hops[root], level = 0.0, 0.0
    while bool((hops < 0).any()):
        reached = torch.zeros(n, dtype=torch.bool, device="cuda")
        reached[col[(hops == level)[row]]] = True
        level += 1.0
        hops[reached & (hops < 0)] = level
    s1 = around(d)
    hit = torch.zeros_like(d)
    hit[root] = 1.0
    for _ in range(8):
        hit = around(hit) / d
        hit[root] = 1.0
    f = [d.log(), 1.0 / d, torch.log1p(hops), (hops == 1).double(), (s1 / d).log(), around((deg == 1).double()) / d,
         (around(s1) / s1).log(), hit]
    return {"features": torch.stack(f, 1), "targets": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mlp_train", "mlp_predict"):
        return _exact_network(case, seed)
    if kind == "solve":
        return _exact_solve(case, seed)
    if kind == "targets":
        return _exact_features(case, seed)
    # The sampled estimates as far as all samples' arrows are popped in seconds.
    if kind == "ecc" and case["form"] == "plain" and case["n"] <= 20000 and case["n"] * case["samples"] <= 1.2e7:
        return _exact_plain(case, seed)
    return None
