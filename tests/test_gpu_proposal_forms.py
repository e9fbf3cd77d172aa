"""GPU parity of the candidate proposal over its dispatch: level sizes on both
sides of the dense-table limits, narrow and wide neighbour counters (node
degrees on both sides of the limit, unit and largest weights), hyperedges
around the 12 pins walked a lane each, and top-4 and top-16 lists."""
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


def fixed_size(n, e, size, hubs, seed, weight):
    """e hyperedges of `size` distinct nodes; node h < hubs is in every
    (2 + h)-th one."""
    rng = np.random.default_rng(seed)
    rows = rng.integers(hubs, n, size=(e, size))
    for h in range(hubs):
        rows[h % 2::2 + h, h] = h
    rows = [np.unique(r) for r in rows]
    off = np.zeros(e + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    pins = np.concatenate(rows).astype(np.int32)
    # any distinct order is a valid one: the source is the first pin
    w = None if weight is None else rng.integers(max(1, weight - 9), weight + 1, size=e).astype(np.int32)
    return inputs.Hypergraph(n, off.astype(np.int32), pins, None, w)


def check_level(torch, g, level, omega=12, delta=10 ** 6, pi=4):
    from test_gpu_steps import gpu_coarsen
    rng = np.random.default_rng(7)
    size = np.ones(g.num_nodes, np.int32) if level == 0 else rng.integers(1, 9, size=g.num_nodes).astype(np.int32)
    cand, score, _, _ = gpu_coarsen(torch, g, size, omega, delta, 3, level, pi=pi)
    oc, ocs = oracle.propose(g, size, omega, delta, seed=3, level=level, pi=pi)
    assert np.array_equal(cand, oc)
    assert np.array_equal(score[oc >= 0], ocs[oc >= 0])


# dense tables for every node up to 4,096 nodes, for large neighbourhoods up to 16,384
@pytest.mark.parametrize("n", [1, 2, 33, 4096, 4097, 16384, 16385, 26624, 26625])
@pytest.mark.parametrize("pi", [4, 16])
def test_level_sizes(torch, n, pi):
    g = fixed_size(n, 2 * n + 1, min(n, 13), min(3, n - 1), n, None) if n > 1 else inputs.random_hypergraph(1, 3, 1)
    check_level(torch, g, 0, pi=pi)
    check_level(torch, g, 2, pi=pi)


@pytest.mark.parametrize("size", [2, 11, 12, 13, 31, 32, 33, 64, 65])
def test_hyperedge_sizes(torch, size):
    check_level(torch, fixed_size(900, 1500, size, 2, size, 5), 1)
    check_level(torch, fixed_size(20000, 9000, size, 2, size, 5), 1)


# step calls assume weights up to 65,536: narrow counters up to 255 hyperedges a node
@pytest.mark.parametrize("e", [508, 510, 512, 514])
@pytest.mark.parametrize("n", [300, 5000, 17000])
def test_degrees_at_the_narrow_limit(torch, e, n):
    check_level(torch, fixed_size(n, e, 9, 3, e, 65536), 0)
    check_level(torch, fixed_size(n, e, 40, 3, e, 65536), 3, pi=16)


# whole calls take the limit from the largest weight: 8,191 hyperedges with unit weights
@pytest.mark.parametrize("e,weight", [(16380, None), (16384, None), (2046, 1000), (2050, 1000), (600, 65536)])
def test_partitions_at_the_narrow_limit(torch, e, weight):
    for n in (200, 5000):
        g = fixed_size(n, e, 5, 3, e, weight)
        r = hp.partition(g, 64, 10 ** 6, seed=1, trace=True)
        o = oracle.partition(g, 64, 10 ** 6, seed=1, trace=True)
        assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
        assert np.array_equal(r.part, o.part)
        assert [t["pairs"] for t in r.trace] == [t["pairs"] for t in o.trace]


# the noise is reduced by a reciprocal: caps from 0 to the largest
@pytest.mark.parametrize("permille", [0, 1, 1000])
def test_noise_caps(torch, permille):
    for weight in (None, 65536):
        g = fixed_size(700, 1100, 7, 2, permille, weight)
        r = hp.partition(g, 16, 10 ** 6, seed=9, noise_permille=permille)
        o = oracle.partition(g, 16, 10 ** 6, seed=9, noise_permille=permille)
        assert r.status == o.status == hp.HP_OK and np.array_equal(r.part, o.part)


# large neighbourhoods: dense tables up to 26,624 nodes, then the hashed tables' limits (2,560, 6,144 neighbours)
@pytest.mark.parametrize("n", [16400, 26624, 26625, 40000])
@pytest.mark.parametrize("pi", [4, 16])
def test_large_neighbourhoods(torch, n, pi):
    rng = np.random.default_rng(n)
    rows = [rng.choice(n, size=k, replace=False) for k in [40] * 3000 + [700] * 30]
    # nodes 0..5 in 64 to 280 hyperedges of 40 pins: 2,500 to 9,000 neighbours
    for h, reps in enumerate((64, 66, 72, 158, 170, 280)):
        for i in rng.choice(3000, size=reps, replace=False):
            rows[i][h] = h
    rows = [np.unique(r) for r in rows]
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    g = inputs.Hypergraph(n, off.astype(np.int32), np.concatenate(rows).astype(np.int32), None, None)
    check_level(torch, g, 0, pi=pi)
    check_level(torch, g, 2, pi=pi)
