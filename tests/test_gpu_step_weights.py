"""The step calls take weights beyond the 65,536 of hp_partition: sums that pass
the 32-bit counters of the forms chosen for small weights still equal the
oracle's."""
import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs
from test_gpu_steps import gpu_coarsen, gpu_refine

pytestmark = pytest.mark.gpu
HEAVY = (1 << 25, 1 << 26)


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


def heavy(n, e, max_size, seed):
    """Hyperedges of 2..max_size pins with weights in HEAVY."""
    rng = np.random.default_rng(seed)
    rows = [rng.choice(n, size=int(rng.integers(2, max_size + 1)), replace=False) for _ in range(e)]
    rows = [np.concatenate([r[:1], np.sort(r[1:])]) for r in rows]
    off = np.zeros(e + 1, np.int32)
    off[1:] = np.cumsum([len(r) for r in rows])
    return inputs.Hypergraph(n, off, np.concatenate(rows).astype(np.int32), np.ones(e, np.int32),
                             rng.integers(*HEAVY, size=e).astype(np.int32))


@pytest.mark.parametrize("n,e,max_size", [(5, 200, 2), (12, 250, 3), (40, 2000, 12), (300, 3000, 40)])
@pytest.mark.parametrize("pi", [4, 16])
def test_coarsen_step(torch, n, e, max_size, pi):
    g = heavy(n, e, max_size, n)
    size = np.ones(n, np.int32)
    cand, score, mate, pairs = gpu_coarsen(torch, g, size, 4, 10 ** 6, 1, 0, pi=pi)
    ocand, oscore = oracle.propose(g, size, 4, 10 ** 6, 1, 0, pi, 100)
    assert np.array_equal(cand, ocand)
    assert np.array_equal(score[ocand >= 0], oscore[ocand >= 0])


# short lists (by part) and long ones (by bits), part counts on both sides of 1,024
@pytest.mark.parametrize("n,e,max_size,nparts", [(300, 12000, 6, 4), (300, 6000, 60, 40), (1200, 9000, 6, 1100)])
def test_refine_step(torch, n, e, max_size, nparts):
    g = heavy(n, e, max_size, n + nparts)
    size = np.ones(n, np.int32)
    # most nodes in part 0: the others' gains there pass 2^32
    rho = np.where(np.arange(n) < nparts, np.arange(n), 0).astype(np.int32)
    omega, delta = n, 10 ** 6
    r = gpu_refine(torch, g, size, rho, nparts, False, omega, delta)
    node, src, dst, gain = oracle.propose_moves(g, size, rho, nparts, omega, False)
    assert len(node) and (nparts > 1024 or gain.max() >= 1 << 32)
    assert np.array_equal(r["node"], node) and np.array_equal(r["src"], src)
    assert np.array_equal(r["dst"], dst) and np.array_equal(r["gain"], gain)
    seq = oracle.sequence(g, size, nparts, node, src, dst, gain)
    assert np.array_equal(r["seq"], seq)
    gseq, k, bg = oracle.inseq_and_prefix(g, size, rho, nparts, node[seq], dst[seq], omega, delta)
    assert np.array_equal(r["gseq"], gseq)
    assert (r["k"], r["best"]) == (k, bg)
