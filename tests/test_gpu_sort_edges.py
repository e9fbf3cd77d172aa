"""The sorts at the edges of their forms: move counts around what one cluster
sorts with 64-bit keys (46,592), event counts around what it sorts with 32-bit
keys (65,536), and item counts at which a direct ranking gives way to radix
passes, at every number of passes.  Moves come with many equal gains, so that
an unstable sort would show; sequence, in-sequence gains and best prefix are the
oracle's."""
import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs
from test_gpu_steps import gpu_refine

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


def moves(m, nparts, seed):
    """Exactly m moves: hyperedge i joins a node alone in its part with two nodes of another part."""
    rng = np.random.default_rng(seed)
    node = rng.permutation(3 * m).reshape(m, 3)
    pins = np.concatenate([node[:, :1], np.sort(node[:, 1:], 1)], 1)
    own = rng.integers(0, nparts, m)
    other = (own + rng.integers(1, nparts, m)) % nparts
    rho = np.empty(3 * m, np.int32)
    rho[node[:, 0]], rho[node[:, 1]], rho[node[:, 2]] = own, other, other
    g = inputs.Hypergraph(3 * m, np.arange(0, 3 * m + 1, 3, dtype=np.int32), pins.reshape(-1).astype(np.int32),
                          np.ones(m, np.int32), rng.integers(1, 4, m).astype(np.int32))
    return g, rho


# n items are ranked directly while n^2 <= passes << 19
RANKED = [int((p << 19) ** 0.5) + d for p in range(1, 9) for d in (0, 1)]


@pytest.mark.parametrize("m", RANKED + [32767, 32768, 32769, 46591, 46592, 46593])
@pytest.mark.parametrize("nparts", [5, 300])
def test_moves(torch, m, nparts):
    g, rho = moves(m, nparts, m)
    size = np.ones(3 * m, np.int32)
    omega, delta = 3 * m, 10 ** 6
    r = gpu_refine(torch, g, size, rho, nparts, False, omega, delta)
    node, src, dst, gain = oracle.propose_moves(g, size, rho, nparts, omega, False)
    assert r["m"] == len(node) == m
    assert np.array_equal(r["node"], node) and np.array_equal(r["src"], src)
    assert np.array_equal(r["dst"], dst) and np.array_equal(r["gain"], gain)
    seq = oracle.sequence(g, size, nparts, node, src, dst, gain)
    assert np.array_equal(r["seq"], seq)
    gseq, k, bg = oracle.inseq_and_prefix(g, size, rho, nparts, node[seq], dst[seq], omega, delta)
    assert np.array_equal(r["gseq"], gseq)
    assert (r["k"], r["best"]) == (k, bg)


# the incidence is sorted by node: one, two and three passes
@pytest.mark.parametrize("n", [100, 3000, 40000])
@pytest.mark.parametrize("pins", RANKED[:6] + [65535, 65536, 65537])
def test_incidence(torch, n, pins):
    rng = np.random.default_rng(pins + n)
    sizes = []
    while sum(sizes) < pins:
        sizes.append(min(int(rng.integers(1, 30)), pins - sum(sizes)))
    rows = [rng.choice(n, size=k, replace=False) for k in sizes]
    off = np.zeros(len(rows) + 1, np.int32)
    off[1:] = np.cumsum(sizes)
    g = inputs.Hypergraph(n, off, np.concatenate([np.concatenate([r[:1], np.sort(r[1:])]) for r in rows]).astype(np.int32),
                          np.ones(len(rows), np.int32), None)
    assert g.num_pins == pins
    r = hp.partition(g, 50, 10 ** 6, seed=1, max_levels=2, theta=2)
    o = oracle.partition(g, 50, 10 ** 6, seed=1, max_levels=2, theta=2)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
