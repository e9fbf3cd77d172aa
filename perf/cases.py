"""The calls whose speed this framework is judged by, over the range of its use.

Each case is one call through the public entry points (the C ABI of
``include/hp.h`` by way of ``paper_2605_20497_gb300.hp``), on synthetic
hypergraphs made on the GPU from a seed: random, layered and Gaussian-local
spiking networks of the families in ``paper_2605_20497_gb300.inputs``, and
irregular circuit-like hypergraphs with several sources per hyperedge.

``listed()`` are the named cases, ``draw(rng)`` gives further ones of the same
ranges, ``prepare`` makes what a user's program holds before the call, ``run``
is the call, ``work`` the bytes and operations it cannot do without, and
``exact`` the same outputs in 64 bits where they are computed numbers (a part
vector has no such value: it is whole numbers, defined by the method alone).
"""
import ctypes
import math
import os

import numpy as np
import torch

from paper_2605_20497_gb300 import hp, train_merge

_MODEL = os.path.join(os.path.dirname(os.path.abspath(hp.__file__)), "merge_random_snn_16k.npz")


def listed():
    return [
        # the smallest partition: a placement tool's unit-sized netlist, several sources per
        # hyperedge, weights, distinct incident hyperedges bounded; launches and latency only
        dict(name="irregular_1k", kind="irregular", nodes=1021, hedges=1531, max_size=24, omega=32, delta=256),
        # the small random network
        dict(name="random_4k", kind="random", nodes=4096, targets=31, omega=256, delta=1024),
        # the 16k random network of the paper's Table I: wide neighbourhoods, binding Delta, refinement-bound
        dict(name="random_16k", kind="random", nodes=16384, targets=127, omega=1024, delta=4096),
        # a mid-sized irregular hypergraph of the first kind
        dict(name="irregular_20k", kind="irregular", nodes=20011, hedges=30011, max_size=64, omega=256, delta=4096),
        # a layered network with spike-rate weights, held in host memory by its program
        dict(name="layered_65k_host", kind="layered_host", layers=8, h=16, w=16, ch=32, omega=4096, delta=65536),
        # the default benchmark: the layered network with 262,144 nodes, 63.6 M pins
        dict(name="layered_262k", kind="layered", layers=8, h=32, w=32, ch=32, omega=4096, delta=65536),
        # the large sparse layered network, no shared destination lists, 80 M pins
        dict(name="gaussian_1m", kind="gaussian", layers=16, h=256, w=256, mean=84, omega=4096, delta=65536),
        # the learned merge priority with the trained weights on the first level of a Gaussian-local network
        dict(name="gaussian_262k_learned", kind="gaussian_learned", layers=16, h=128, w=128, mean=84, omega=4096,
             delta=65536),
        # many small uneven networks in one call
        dict(name="batch_24", kind="batch", count=24, n_min=1000, n_max=64000, flight=16),
        # the objective of a given part vector on the large network
        dict(name="connectivity_gaussian_1m", kind="connectivity", layers=16, h=256, w=256, mean=84, parts=391),
        # the learned priority's MLP on the pairs of a large level
        dict(name="merge_scores_8m", kind="scores", rows=8388608),
        # one minibatch of the priority's training: loss and gradient
        dict(name="merge_grad_64k", kind="grad", rows=65536),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["irregular", "random", "layered", "layered_host", "gaussian", "gaussian_learned", "batch",
                       "connectivity", "scores", "grad"])
    if kind == "irregular":
        n = _log(rng, 1000, 20011)
        return dict(kind=kind, nodes=n, hedges=int(n * rng.uniform(1.2, 1.5)), max_size=rng.randint(16, 64),
                    omega=rng.randint(32, 256), delta=4096)
    if kind == "random":
        om = 1 << rng.randint(8, 10)
        return dict(kind=kind, nodes=_log(rng, 1000, 16384), targets=_log(rng, 7, 127), omega=om, delta=4 * om)
    if kind in ("layered", "layered_host"):
        return dict(kind=kind, layers=rng.randint(3, 8), h=rng.randint(7, 32), w=rng.randint(7, 32),
                    ch=rng.randint(5, 32), omega=4096, delta=65536)
    if kind in ("gaussian", "gaussian_learned"):
        side = 256 if kind == "gaussian" else 128
        return dict(kind=kind, layers=rng.randint(4, 16), h=_log(rng, 32, side), w=_log(rng, 32, side),
                    mean=rng.randint(20, 84), omega=4096, delta=65536)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 24), n_min=1000, n_max=_log(rng, 2000, 64000), flight=16)
    if kind == "connectivity":
        return dict(kind=kind, layers=rng.randint(4, 16), h=_log(rng, 32, 256), w=_log(rng, 32, 256),
                    mean=rng.randint(20, 84), parts=_log(rng, 2, 400))
    if kind == "scores":
        return dict(kind=kind, rows=_log(rng, 1000, 8388608))
    return dict(kind="grad", rows=_log(rng, 4096, 65536))


# ------------------------------------------------------------------ hypergraphs
class Graph:
    """CSR of a hypergraph on the GPU (int32 tensors; None: one source, unit weights)."""

    def __init__(self, num_nodes, sizes, pins, src_counts=None, weights=None):
        self.num_nodes, self.num_hedges = num_nodes, sizes.numel()
        off = torch.zeros(sizes.numel() + 1, dtype=torch.int64, device=pins.device)
        torch.cumsum(sizes, 0, out=off[1:])
        self.offsets, self.pins = off.int(), pins.int()
        self.src_counts, self.weights = src_counts, weights


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rows_of_targets(src, need, targets_of, n, g):
    """Hyperedges {src} + up to `need` distinct targets, ascending: rows and
    draws are flat, `targets_of(rows)` gives one candidate (or -1) for each."""
    rows = torch.repeat_interleave(torch.arange(need.numel(), device="cuda"), (need * 3) // 2 + 8)
    t = targets_of(rows)
    key = rows * n + t
    key = torch.unique(key[t >= 0])                      # distinct targets of each row
    rows = key // n
    # where a row has too many, a random choice of them stays
    order = torch.argsort(rows * (1 << 24) + torch.randint(0, 1 << 24, rows.shape, generator=g, device="cuda"))
    cnt = torch.bincount(rows, minlength=need.numel())
    rank = torch.arange(rows.numel(), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[rows]
    key = torch.sort(key[order[rank < need[rows]]])[0]
    rows, t = key // n, key % n
    cnt = torch.bincount(rows, minlength=need.numel())
    off = torch.cumsum(cnt + 1, 0) - (cnt + 1)
    pins = torch.empty(rows.numel() + need.numel(), dtype=torch.int64, device="cuda")
    pins[off] = src
    pins[torch.arange(rows.numel(), device="cuda") + rows + 1] = t
    return cnt + 1, pins


def _random(n, need, g):
    """Node i owns {i} + need[i] distinct uniform targets."""
    def targets(rows):
        t = torch.randint(0, n - 1, rows.shape, generator=g, device="cuda")
        return t + (t >= rows)
    return Graph(n, *_rows_of_targets(torch.arange(n, device="cuda"), need, targets, n, g))


def _powerlaw(n, g):
    """Hyperedge sizes from P(s) ~ s^-2.2 on [2, 1024], uniform targets."""
    s = torch.arange(2, min(1024, n // 2) + 1, dtype=torch.float64, device="cuda")
    cdf = torch.cumsum(s ** -2.2, 0)
    u = torch.rand(n, dtype=torch.float64, generator=g, device="cuda") * cdf[-1]
    return _random(n, 1 + torch.searchsorted(cdf, u).clamp(max=s.numel() - 1), g)


def _gaussian(c, g):
    """Node of every layer but the last owns {itself} + geometric(mean) targets
    around its position in the next layer, 4 cells wide."""
    h, w, cells = c["h"], c["w"], c["h"] * c["w"]
    n, E = c["layers"] * cells, (c["layers"] - 1) * cells
    u = torch.rand(E, dtype=torch.float64, generator=g, device="cuda").clamp(min=1e-12)
    need = (torch.log(u) / math.log(1 - 1 / c["mean"])).long().clamp(1, 400)

    def targets(rows):
        y = torch.randn(rows.shape, generator=g, device="cuda").mul_(4).round_().long() + (rows // w) % h
        x = torch.randn(rows.shape, generator=g, device="cuda").mul_(4).round_().long() + rows % w
        ok = (y >= 0) & (y < h) & (x >= 0) & (x < w)
        return torch.where(ok, (rows // cells + 1) * cells + y * w + x, -1)

    return Graph(n, *_rows_of_targets(torch.arange(E, device="cuda"), need, targets, n, g))


def _layered(c, g, pruned):
    """Neurons of a layer reach all channels of the 3x3 window in the next
    one; `pruned`: one hyperedge in 64 has lost one random target."""
    h, w, ch = c["h"], c["w"], c["ch"]
    P = (c["layers"] - 1) * h * w
    pos = torch.arange(P, device="cuda")
    d = torch.arange(-1, 2, device="cuda")
    y = ((pos // w) % h)[:, None, None] + d[:, None]
    x = (pos % w)[:, None, None] + d
    ok = ((y >= 0) & (y < h) & (x >= 0) & (x < w)).reshape(P, 9)
    t = (((pos // (h * w) + 1)[:, None, None] * h + y) * w + x).reshape(P, 9)
    t = (t[:, :, None] * ch + torch.arange(ch, device="cuda")).reshape(P, 1, 9 * ch).expand(P, ch, 9 * ch)
    E = P * ch
    full = torch.cat([torch.arange(E, device="cuda").reshape(P, ch, 1), t], 2).reshape(E, 1 + 9 * ch).int()
    keep = torch.ones(P, ch, 1 + 9 * ch, dtype=torch.bool, device="cuda")
    keep[:, :, 1:] = ok[:, None, :, None].expand(P, ch, 9, ch).reshape(P, ch, 9 * ch)
    keep = keep.reshape(E, 1 + 9 * ch)
    if pruned:
        rows = torch.randperm(E, generator=g, device="cuda")[: max(1, E // 64)]
        # the window's middle position lies inside the grid for every neuron
        keep[rows, 1 + 4 * ch + torch.randint(0, ch, rows.shape, generator=g, device="cuda")] = False
    return Graph(c["layers"] * h * w * ch, keep.sum(1), full[keep])


def _irregular(c, g):
    """Hyperedges of 1..max_size distinct nodes, about a quarter of them
    sources, weights 1..100."""
    n, E = c["nodes"], c["hedges"]
    want = torch.randint(1, c["max_size"] + 1, (E,), generator=g, device="cuda")
    rows = torch.repeat_interleave(torch.arange(E, device="cuda"), want)
    key = torch.unique(rows * n + torch.randint(0, n, rows.shape, generator=g, device="cuda"))
    rows, t = key // n, key % n
    dst = (torch.rand(rows.shape, generator=g, device="cuda") >= 0.25).long()
    key = torch.sort((rows * 2 + dst) * n + t)[0]            # sources first, each half ascending
    src = torch.bincount(rows[dst == 0], minlength=E).int()
    wgt = torch.randint(1, 101, (E,), generator=g, device="cuda", dtype=torch.int32)
    return Graph(n, torch.bincount(rows, minlength=E), key % n, src, wgt)


def _batch_sizes(c):
    """Nodes and Omega of the instances: node counts evenly spread over the
    logarithm of the range, Omega cycling through 2^8 .. 2^12."""
    ratio = c["n_max"] / c["n_min"]
    return [(int(c["n_min"] * ratio ** ((i + 0.5) / c["count"])), 1 << (8 + i * 3 % 5)) for i in range(c["count"])]


def _batch(c, g):
    """Instances with power-law hyperedge sizes, Delta = 4 Omega."""
    return [(_powerlaw(n, g), om, 4 * om) for n, om in _batch_sizes(c)]


# ------------------------------------------------------------------ state, call, outputs
def _ptr(t):
    return None if t is None else t.data_ptr()


def _ok(rc):
    if rc != hp.HP_OK:
        raise RuntimeError(f"{hp.hp_status_string(rc)}: {hp.hp_last_error()}")


def prepare(case, seed):
    g, kind = _generator(seed), case["kind"]
    s = dict(case=case, kind=kind, seed=int(seed), stats=hp.hp_stats())
    if kind in ("scores", "grad"):
        # log codes and ratios of pairs lie all over 0..255
        s["feat"] = torch.randint(0, 256, (case["rows"], 16), generator=g, device="cuda", dtype=torch.uint8)
        if kind == "scores":
            s["model"] = train_merge.load(_MODEL)
        else:
            s["label"] = (torch.rand(case["rows"], generator=g, device="cuda") < 0.1).float()
            s["params"] = torch.from_numpy(train_merge.init_params(int(seed) & 0x7FFFFFFF)).cuda()
        return s
    if kind == "batch":
        s["graphs"] = _batch(case, g)
        s["opt"] = hp.options()
        total = sum(x.num_nodes for x, _, _ in s["graphs"])
        s["part"] = torch.empty(total, dtype=torch.int32, device="cuda")
        s["inst"] = (hp.hp_instance * case["count"])()
        at = 0
        for i, (x, om, de) in enumerate(s["graphs"]):
            s["inst"][i] = hp.hp_instance(_ptr(x.pins), _ptr(x.offsets), None, None, x.num_hedges, x.num_nodes, om, de,
                                          i, s["part"][at:].data_ptr())
            at += x.num_nodes
        s["batch_stats"] = (hp.hp_stats * case["count"])()
        return s
    if kind == "irregular":
        s["graph"], s["opt"] = _irregular(case, g), hp.options(count_kind=hp.HP_COUNT_INCIDENT)
    elif kind == "random":
        need = torch.full((case["nodes"],), case["targets"], device="cuda")
        s["graph"], s["opt"] = _random(case["nodes"], need, g), hp.options()
    elif kind in ("layered", "layered_host"):
        s["graph"], s["opt"] = _layered(case, g, kind == "layered"), hp.options()
    else:
        s["graph"], s["opt"] = _gaussian(case, g), hp.options()
    x = s["graph"]
    if kind == "gaussian_learned":
        s["opt"] = hp.options(learned_k=16, learned_levels=1, model=train_merge.load(_MODEL))
    if kind == "connectivity":
        # a part vector such as a partition leaves: blocks of neighbouring nodes, with some strays
        n, k = x.num_nodes, case["parts"]
        part = torch.arange(n, device="cuda") * k // n
        stray = torch.rand(n, generator=g, device="cuda") < 0.1
        s["part"] = torch.where(stray, torch.randint(0, k, (n,), generator=g, device="cuda"), part).int()
    elif kind == "layered_host":
        x.weights = torch.randint(1, 1001, (x.num_hedges,), generator=g, device="cuda", dtype=torch.int32)
        s["host"] = [t.cpu().numpy() for t in (x.pins, x.offsets, x.weights)]
        s["part"] = np.zeros(x.num_nodes, dtype=np.int32)
        s["graph"] = None
        s["sizes"] = (x.num_hedges, x.num_nodes)
    else:
        s["part"] = torch.empty(x.num_nodes, dtype=torch.int32, device="cuda")
    return s


def run(s):
    case, kind, stream = s["case"], s["kind"], torch.cuda.current_stream().cuda_stream
    if kind == "scores":
        rc, out = hp.merge_scores(s["feat"], s["model"], stream)
        _ok(rc)
        return out
    if kind == "grad":
        rc, grad, loss = hp.merge_grad(s["feat"], s["label"], s["params"], stream)
        _ok(rc)
        return {"grad": grad, "loss": loss}
    if kind == "connectivity":
        x = s["graph"]
        rc, conn, cut = hp.hp_connectivity(_ptr(x.pins), _ptr(x.offsets), x.num_hedges, None, _ptr(s["part"]),
                                           x.num_nodes, case["parts"], stream)
        _ok(rc)
        return {"connectivity": conn, "cut_net": cut}
    if kind == "batch":
        _ok(hp.load().hp_partition_batch(s["inst"], case["count"], ctypes.byref(s["opt"]), case["flight"],
                                         s["batch_stats"], None, stream))
        return {"part": s["part"], "connectivity": np.array([t.connectivity for t in s["batch_stats"]])}
    st = s["stats"]
    if kind == "layered_host":
        pins, off, wgt = s["host"]
        _ok(hp.hp_partition_host(pins.ctypes.data, off.ctypes.data, s["sizes"][0], s["sizes"][1], None,
                                 wgt.ctypes.data, case["omega"], case["delta"], s["seed"], ctypes.byref(s["opt"]),
                                 s["part"].ctypes.data, ctypes.byref(st), stream))
    else:
        x = s["graph"]
        _ok(hp.hp_partition(_ptr(x.pins), _ptr(x.offsets), x.num_hedges, x.num_nodes, _ptr(x.src_counts),
                            _ptr(x.weights), case["omega"], case["delta"], s["seed"], ctypes.byref(s["opt"]),
                            _ptr(s["part"]), ctypes.byref(st), stream))
    return {"part": s["part"], "connectivity": st.connectivity, "cut_net": st.cut_net, "parts": st.num_parts,
            "moves": st.moves_applied}


# ------------------------------------------------------------------ bounds and 64-bit values
def _shape(case):
    """(nodes, hyperedges, expected pins) of a case's hypergraph."""
    kind = case["kind"]
    if kind == "irregular":
        return case["nodes"], case["hedges"], int(case["hedges"] * (case["max_size"] + 1) / 2)
    if kind == "random":
        return case["nodes"], case["nodes"], case["nodes"] * (case["targets"] + 1)
    if kind == "batch":
        n = sum(x for x, _ in _batch_sizes(case))
        s = np.arange(2, 1025, dtype=np.float64)
        return n, n, int(n * (s ** -1.2).sum() / (s ** -2.2).sum())
    if kind in ("layered", "layered_host"):
        h, w, ch, pairs = case["h"], case["w"], case["ch"], case["layers"] - 1
        return (case["layers"] * h * w * ch, pairs * h * w * ch,
                pairs * ch * (h * w + (3 * h - 2) * (3 * w - 2) * ch))
    cells = case["h"] * case["w"]
    return case["layers"] * cells, (case["layers"] - 1) * cells, (case["layers"] - 1) * cells * case["mean"]


def work(case):
    kind = case["kind"]
    if kind == "scores":    # 16 B of features in, a 32-bit score out; 16 x 64 + 64 x 64 + 64 products a row
        return {"bytes": case["rows"] * 20, "flops": case["rows"] * 2 * (1024 + 4096 + 64)}
    if kind == "grad":      # forward; two more products of W2's size and one of W1's
        return {"bytes": case["rows"] * 20 + 2 * 4 * hp.HP_MERGE_NPARAM,
                "flops": case["rows"] * 2 * (2 * 1024 + 3 * 4096 + 2 * 64)}
    n, e, pins = _shape(case)
    extra = 4 * e if kind == "layered_host" else 8 * e if kind == "irregular" else 0   # weights, source counts
    return {"bytes": 4 * (pins + e + 1 + n) + extra, "flops": 0}


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("scores", "grad", "connectivity"):
        return None
    s = prepare(case, seed)
    if kind == "connectivity":
        x, parts = s["graph"], case["parts"]
        rows = torch.repeat_interleave(torch.arange(x.num_hedges, device="cuda"), x.offsets.diff().long())
        key = torch.unique(rows * parts + s["part"].long()[x.pins.long()])
        lam = torch.bincount(key // parts, minlength=x.num_hedges)
        return {"connectivity": int((lam - 1).sum()), "cut_net": int((lam > 1).sum())}
    f64 = lambda a: torch.as_tensor(np.asarray(a), device="cuda").double()
    if kind == "scores":
        m, out = s["model"], []
        for f in s["feat"].split(1 << 20):      # whole numbers below 2^53: exact in doubles
            a = ((f.double() @ f64(m.w1).T + f64(m.b1)) / 2.0 ** int(m.shift1)).floor().clamp(0, 255)
            a = ((a @ f64(m.w2).T + f64(m.b2)) / 2.0 ** int(m.shift2)).floor().clamp(0, 255)
            out.append((a @ f64(m.w3) + float(m.b3)).to(torch.int32))
        return torch.cat(out)
    p = s["params"].double().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = p.split([1024, 64, 4096, 64, 64, 1])
    h1 = torch.relu(s["feat"].double() / 256 @ w1.view(64, 16).T + b1)
    o = torch.relu(h1 @ w2.view(64, 64).T + b2) @ w3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(o, s["label"].double())
    loss.backward()
    return {"grad": p.grad, "loss": float(loss)}
