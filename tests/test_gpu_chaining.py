"""GPU parity of the chaining rounds: window lengths around the 32 moves a warp
scans at a time, many moves of equal gain (unit weights) and few (weights),
the device-wide form, and move counts on both sides of the cluster kernel's
shared-memory copy (10,240 moves)."""
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


def check(g, omega, delta, **opts):
    r = hp.partition(g, omega, delta, seed=2, trace=True, **opts)
    o = oracle.partition(g, omega, delta, seed=2, trace=True, **opts)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
    assert [t["moves"] for t in r.trace] == [t["moves"] for t in o.trace]


@pytest.mark.parametrize("window", [1, 2, 31, 32, 33, 64, 65, 256, 5000])
@pytest.mark.parametrize("weights", [False, True])
def test_windows(torch, window, weights):
    g = inputs.random_hypergraph(2500, 4000, 7, seed=window, multi_src=True, weights=weights, max_weight=1000)
    check(g, 500, 10 ** 6, chain_window=window)


# 45,056 moves is the most one cluster sorts
@pytest.mark.parametrize("n,least,most", [(12000, 4097, 45056), (70000, 45057, 70000)])
@pytest.mark.parametrize("window", [1, 33, 256])
@pytest.mark.parametrize("weights", [False, True])
def test_one_repetition_device_wide(torch, n, least, most, window, weights):
    # a random part vector: most nodes propose a move, more than one cluster sequences on a step call
    from test_gpu_steps import gpu_refine
    g = inputs.random_hypergraph(n, 3 * n // 2, 6, seed=5, weights=weights, max_weight=9)
    rng = np.random.default_rng(window)
    size = rng.integers(1, 4, size=g.num_nodes).astype(np.int32)
    rho = rng.integers(0, 7, size=g.num_nodes).astype(np.int32)
    omega, delta = n, 10 ** 6
    r = gpu_refine(torch, g, size, rho, 7, False, omega, delta, chain_window=window)
    assert least <= r["m"] <= most
    seq = oracle.sequence(g, size, 7, r["node"], r["src"], r["dst"], r["gain"], window=window)
    assert np.array_equal(r["seq"], seq)


# Omega = 1: every node is its own part and every node with a hyperedge proposes a move
@pytest.mark.parametrize("n", [10240, 10241])
def test_moves_at_the_shared_memory_limit(torch, n):
    check(inputs.random_snn(n, 2, seed=n), 1, 64)
