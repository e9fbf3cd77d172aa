"""GPU parity of one refinement repetition at the edges of its kernels'
classes: hyperedges of 2, 8, 9, 32, 33, 128, 129, 512 and 513 pins, part counts
on both sides of 1,024 (bit and part-indexed forms) and 2,048 (per-CTA part
sums), nodes with few, 256, 1,024 and more cut hyperedges, and single-pin
hyperedges."""
import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_20497_gb300 import build
    build.build()
    oracle.build()
    hp.load()
    return t


def graph(n, sizes, seed, hub=0):
    """One hyperedge per entry of sizes; node 0 is in the first `hub` ones;
    up to a third of the pins are sources, weights 1..50."""
    rng = np.random.default_rng(seed)
    rows, src = [], []
    for i, k in enumerate(sizes):
        r = rng.choice(n - 1, size=k, replace=False) + 1
        if i < hub:
            r[0] = 0
        s = int(rng.integers(0, k // 3 + 2)) if k > 1 else int(rng.integers(0, 2))
        rows.append(np.concatenate([np.sort(r[:s]), np.sort(r[s:])]))
        src.append(min(s, k))
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    return inputs.Hypergraph(n, off.astype(np.int32), np.concatenate(rows).astype(np.int32), np.asarray(src, np.int32),
                             rng.integers(1, 51, size=len(rows)).astype(np.int32))


def check(torch, g, nparts, seed, second_half=False, spread=1.0):
    from test_gpu_steps import gpu_refine
    rng = np.random.default_rng(seed)
    n = g.num_nodes
    # spread < 1: most nodes in few parts, so that lists are short and counts high
    rho = (nparts * rng.random(n) ** (1 / spread)).astype(np.int32)
    rho[:nparts] = np.arange(min(nparts, n))
    size = rng.integers(1, 4, n).astype(np.int32)
    omega, delta = 2 * n // nparts + 8, 10 ** 6
    r = gpu_refine(torch, g, size, rho, nparts, second_half, omega, delta)
    node, src, dst, gain = oracle.propose_moves(g, size, rho, nparts, omega, second_half)
    assert np.array_equal(r["node"], node) and np.array_equal(r["src"], src)
    assert np.array_equal(r["dst"], dst) and np.array_equal(r["gain"], gain)
    if len(node) == 0:
        return
    seq = oracle.sequence(g, size, nparts, node, src, dst, gain)
    assert np.array_equal(r["seq"], seq)
    gseq, k, bg = oracle.inseq_and_prefix(g, size, rho, nparts, node[seq], dst[seq], omega, delta)
    assert np.array_equal(r["gseq"], gseq)
    assert (r["k"], r["best"]) == (k, bg)


@pytest.mark.parametrize("nparts", [2, 31, 32, 33, 128, 1023, 1024, 1025, 2048, 2049])
def test_part_counts(torch, nparts):
    sizes = [1] * 40 + [2, 3, 8, 9, 32, 33, 128, 129] * 40
    g = graph(max(2500, nparts), sizes, nparts)
    for seed, half in ((1, False), (2, True)):
        check(torch, g, nparts, seed, half)


@pytest.mark.parametrize("size", [1, 2, 7, 8, 9, 31, 32, 33, 64, 65, 127, 128, 129, 511, 512, 513, 700])
def test_hyperedge_sizes(torch, size):
    g = graph(900, [size] * 300, size)
    for nparts in (3, 40, 1100 if size < 100 else 300):
        if nparts <= g.num_nodes:
            check(torch, g, nparts, size)
    check(torch, g, 60, size + 1, spread=0.2)


@pytest.mark.parametrize("hub", [0, 31, 32, 33, 256, 257, 1024, 1025, 3000])
def test_cut_degrees(torch, hub):
    g = graph(1500, [5] * 3100, hub, hub)
    check(torch, g, 20, hub)
    check(torch, g, 1200, hub)


# few coarsening levels: many parts at the start, most of them empty soon, so that the rest is renumbered
@pytest.mark.parametrize("max_levels", [0, 1, 3])
@pytest.mark.parametrize("omega", [40, 700])
def test_renumbered_parts(torch, max_levels, omega):
    g = inputs.random_hypergraph(1500, 2600, 7, seed=omega, multi_src=True, weights=True)
    r = hp.partition(g, omega, 10 ** 5, seed=4, trace=True, max_levels=max_levels)
    o = oracle.partition(g, omega, 10 ** 5, seed=4, trace=True, max_levels=max_levels)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
    for k, v in o.stats.items():
        assert r.stats[k] == v, k
    assert [t["moves"] for t in r.trace] == [t["moves"] for t in o.trace]


# several repetitions a level that apply moves: the state updated for them (levels of 2^19 pins or more, so
# here down to the level that falls below that) equals the rebuilt one
@pytest.mark.parametrize("weights,kind", [(False, 0), (True, 1)])
def test_updated_repetitions(torch, weights, kind):
    n, e, max_size = 20000, 26000, 60
    rng = np.random.default_rng(5)
    # hyperedges around a ring: moves between neighbouring parts, a few at a time
    rows, src = [], []
    for i in range(e):
        k = int(rng.integers(1, max_size + 1)) if i % 3 else int(rng.integers(1, 9))
        r = np.unique((rng.integers(0, n) + np.round(rng.normal(0, 90, size=k)).astype(np.int64)) % n)
        rng.shuffle(r)
        s = int(rng.integers(0, len(r) + 1)) if weights else 1
        rows.append(np.concatenate([np.sort(r[:s]), np.sort(r[s:])]))
        src.append(s)
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    assert off[-1] >= 1 << 19
    g = inputs.Hypergraph(n, off.astype(np.int32), np.concatenate(rows).astype(np.int32),
                          np.asarray(src, np.int32), rng.integers(1, 30, size=len(rows)).astype(np.int32) if weights else None)
    r = hp.partition(g, 300, 6000, seed=3, trace=True, count_kind=kind)
    o = oracle.partition(g, 300, 6000, seed=3, trace=True, count_kind=kind)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
    for k, v in o.stats.items():
        assert r.stats[k] == v, k
    assert [(t["moves"], t["reps"], t["conn"]) for t in r.trace] == [(t["moves"], t["reps"], t["conn"]) for t in o.trace]
    assert any(t["reps"] > 3 and t["pins"] >= 1 << 19 for t in o.trace)
