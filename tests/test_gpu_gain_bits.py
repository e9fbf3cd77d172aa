"""GPU parity of the gains computed from part bits (refinement of levels whose
cut hyperedges span many parts): whole partitions against the oracle at part
counts on both sides of every row width (128, 256, 512 and 1,024 parts), and
at weight sums on both sides of the 32-bit counters' limit."""
import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_20497_gb300 import build
    build.build()
    oracle.build()
    hp.load()


def check(g, omega, delta, **opts):
    r = hp.partition(g, omega, delta, seed=5, trace=True, **opts)
    o = oracle.partition(g, omega, delta, seed=5, trace=True, **opts)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
    for k, v in o.stats.items():
        assert r.stats[k] == v, k
    assert [t["conn"] for t in r.trace] == [t["conn"] for t in o.trace]
    assert [t["moves"] for t in r.trace] == [t["moves"] for t in o.trace]


# nodes = parts when Omega = 1 (one coarsening attempt forms no pair): exact part counts
@pytest.mark.parametrize("n", [2, 31, 127, 128, 129, 256, 257, 512, 513, 1024, 1025])
def test_part_counts_at_row_edges(n):
    check(inputs.random_snn(n, min(n - 1, 40), seed=n), 1, 4096)


@pytest.mark.parametrize("omega", [2, 3, 5, 9, 40])
@pytest.mark.parametrize("weights", [False, True])
def test_moves_at_every_row_width(omega, weights):
    g = inputs.random_hypergraph(1300, 1700, 40, seed=omega, multi_src=True, weights=weights, isolated=7)
    check(g, omega, 100000)
    check(g, omega, 400 * omega, count_kind=1)


# 65,536 weights of 65,536 sum to 2^32: the list form from there on
@pytest.mark.parametrize("e", [65535, 65536])
def test_weight_sum_at_the_counter_limit(e):
    rng = np.random.default_rng(e)
    pins = np.argsort(rng.random((e, 40)), axis=1)[:, :20].astype(np.int32)   # 20 of 40 nodes each
    off = np.arange(0, 20 * e + 1, 20, dtype=np.int32)
    g = inputs.Hypergraph(40, off, pins.reshape(-1), None, np.full(e, 65536, np.int32))
    check(g, 4, 10 ** 6)
