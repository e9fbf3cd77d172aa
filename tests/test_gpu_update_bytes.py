"""hp_stats.alg_bytes counts what the refinement repetitions do: a rebuilt
repetition every pin and list entry of its level, an updated one those of the
hyperedges with a moved pin, a reused one neither.  The repetitions are replayed
by the oracle, so the count is exact, and it tells that the updates ran: on two
consecutive levels, with hyperedges of up to 512 pins, and after renumbering."""
import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs

UPDATE_PINS, MAX_PARTS, MAX_PINS = 1 << 19, 1024, 512


def ring(n, sizes, seed, width):
    """Hyperedges of nearby nodes on a ring; weights 1..9, several sources."""
    rng = np.random.default_rng(seed)
    rows, src = [], []
    for k in sizes:
        off = np.unique(np.round(rng.normal(0, width, size=4 * k)).astype(np.int64) % n)
        r = (rng.integers(0, n) + rng.permutation(off)[:k]) % n
        s = int(rng.integers(0, len(r) // 4 + 2)) if len(r) > 1 else 1
        rows.append(np.concatenate([np.sort(r[:s]), np.sort(r[s:])]))
        src.append(s)
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    return inputs.Hypergraph(n, off.astype(np.int32), np.concatenate(rows).astype(np.int32), np.asarray(src, np.int32),
                             rng.integers(1, 10, size=len(rows)).astype(np.int32))


def lists(g, rho):
    """|e| and lambda(e) of every hyperedge."""
    sz = np.diff(g.offsets)
    rows = np.repeat(np.arange(g.num_hedges), sz)
    key = np.unique(rows * np.int64(g.num_nodes) + rho[g.pins])
    return sz, np.bincount(key // g.num_nodes, minlength=g.num_hedges)


def replay(levels, omega, delta, theta):
    """Bytes of the refinement of the levels (coarsest first: graph, size,
    gamma to the next coarser one), and the repetitions by kind and level."""
    total, kinds, rho, nparts = 0, [], None, levels[0][0].num_nodes
    for g, size, gamma in levels:
        rho = np.arange(nparts, dtype=np.int32) if rho is None else rho[gamma]
        used = np.unique(rho)
        if 2 * len(used) <= nparts:
            rho, nparts = np.searchsorted(used, rho).astype(np.int32), len(used)
        sz = np.diff(g.offsets)
        may = g.num_pins >= UPDATE_PINS and sz.max() <= MAX_PINS and nparts <= MAX_PARTS
        k, same, rep, kind = 0, False, 0, {"rebuilt": 0, "updated": 0, "reused": 0}
        cuts = cut_lam = 0
        prev = rho
        while rep < theta:
            half = rep >= theta // 2
            if same:
                kind["reused"] += 1
            else:
                _, lam = lists(g, rho)
                multi = sz >= 2
                if may and 0 < 8 * k <= g.num_nodes:
                    kind["updated"] += 1
                    rows = np.repeat(np.arange(g.num_hedges), sz)
                    touched = np.bincount(rows[(prev != rho)[g.pins]], minlength=g.num_hedges) > 0
                    multi_t = multi & touched
                    total += 4 * g.num_pins + 8 * int(sz[multi_t].sum()) + 12 * int(lam[multi_t].sum())
                else:
                    kind["rebuilt"] += 1
                    total += 12 * g.num_pins + 12 * int(lam[multi].sum())
                cut = multi & (lam >= 2)
                cuts, cut_lam = int(sz[cut].sum()), int((sz[cut].astype(np.int64) * lam[cut]).sum())
            node, *_ = oracle.propose_moves(g, size, rho, nparts, omega, half)
            total += 4 * cuts + 12 * cut_lam + 48 * len(node)
            prev = rho
            k, rho = oracle.refine_rep(g, size, rho, nparts, half, omega, delta)
            same = k == 0
            if same:
                if half:
                    break
                rep = theta // 2 - 1
            rep += 1
        kinds.append(kind)
    return total, kinds, rho


def hierarchy(g, omega, delta, seed, max_levels):
    """The levels as the partitioner builds them, coarsest first."""
    out, cur, size = [], g, np.ones(g.num_nodes, np.int32)
    for level in range(max_levels):
        cand, score = oracle.propose(cur, size, omega, delta, seed, level)
        _, mate = oracle.pair_isolated(cur, size, omega, delta, cand, np.full(cur.num_nodes, -1, np.int32))
        _, mate = oracle.match_all(cand, score, mate)
        gamma, csize, off, pins, nsrc = oracle.contract(cur, size, mate)
        out.append((cur, size, gamma))
        cur, size = inputs.Hypergraph(len(csize), off.astype(np.int32), pins.astype(np.int32), nsrc.astype(np.int32),
                                      cur.weights), csize
    out.append((cur, size, None))
    return out[::-1]


CASES = {
    # every node a part at first, hyperedges of up to 512 pins
    "one_level": dict(n=1024, sizes=[2, 7, 8, 9, 129, 300, 511, 512] * 356, width=150, omega=64, max_levels=0),
    # updates on both levels of two
    "two_levels": dict(n=1700, sizes=[3, 8, 9, 31, 64, 100, 128, 300] * 1150, width=60, omega=60, max_levels=1),
    # most of the coarsest level's parts are empty at the finer one
    "renumbered": dict(n=1700, sizes=[4, 8, 16, 64, 120, 200] * 1650, width=60, omega=500, max_levels=1),
}
THETA = 8


def case(name):
    c = CASES[name]
    g = ring(c["n"], c["sizes"], 7, c["width"])
    return g, c["omega"], 10 ** 6, c["max_levels"]


# the cases reach what they are for (no GPU)
@pytest.mark.parametrize("name", CASES)
def test_cases_reach_the_updates(name):
    oracle.build()
    g, omega, delta, max_levels = case(name)
    levels = hierarchy(g, omega, delta, 3, max_levels)
    _, kinds, rho = replay(levels, omega, delta, THETA)
    o = oracle.partition(g, omega, delta, seed=3, max_levels=max_levels, theta=THETA)
    assert np.array_equal(np.unique(rho, return_inverse=True)[1], o.part)   # the replay is the method
    assert kinds[-1]["updated"] > 0 and kinds[0]["rebuilt"] > 0
    if name == "two_levels":
        assert kinds[0]["updated"] > 0
    if name == "renumbered":
        assert levels[0][0].num_nodes >= 2 * len(np.unique(rho))


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_bytes_of_updated_repetitions(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_20497_gb300 import build
    build.build()
    oracle.build()
    hp.load()
    g, omega, delta, max_levels = case(name)
    want, kinds, rho = replay(hierarchy(g, omega, delta, 3, max_levels), omega, delta, THETA)
    r = hp.partition(g, omega, delta, seed=3, max_levels=max_levels, theta=THETA)
    coarsening = hp.partition(g, omega, delta, seed=3, max_levels=max_levels, theta=0).stats["alg_bytes"]
    assert r.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, np.unique(rho, return_inverse=True)[1])
    assert r.stats["alg_bytes"] - coarsening == want, kinds
