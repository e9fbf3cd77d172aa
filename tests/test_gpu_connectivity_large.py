"""hp_connectivity (and the statistics of a partition) with hyperedges that a
CTA takes: sizes around the limit of 8,192 pins and around a CTA's 4,096 pins a
step, few and many of them, beside small ones, every error in them, and no
slower than their pins are worth."""
import time

import numpy as np
import pytest

import oracle
from paper_2605_20497_gb300 import hp, inputs
from test_gpu_connectivity_forms import call, count, make

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


SIZES = [8191, 8192, 8193, 12287, 12288, 12289, 20001, 3, 1, 130, 30000]


@pytest.mark.parametrize("nparts", [1, 2, 33, 1024, 1025, 32768])
@pytest.mark.parametrize("ordered", [True, False])
def test_large_hyperedges(torch, nparts, ordered):
    n = 34000
    off, pins = make(n, SIZES * 2, nparts, ordered)
    rng = np.random.default_rng(nparts)
    w = rng.integers(1, 65537, len(off) - 1).astype(np.int32)
    for part in (rng.integers(0, nparts, n).astype(np.int32), np.zeros(n, np.int32)):
        for weights in (None, w):
            st, c, cn = call(torch, off, pins, n, part, nparts, weights)
            assert st == hp.HP_OK and (c, cn) == count(off, pins, part, weights)


def test_errors_in_large_hyperedges(torch):
    n, nparts = 40000, 9
    off, pins = make(n, [5, 9000, 30000, 3], 1)
    part = np.random.default_rng(2).integers(0, nparts, n).astype(np.int32)
    ok = call(torch, off, pins, n, part, nparts)
    assert ok[0] == hp.HP_OK
    e2 = int(off[2])
    for at, value in ((e2, n), (e2 + 1, -1), (e2 + 4096, 2**31 - 1), (e2 + 29999, -2**31)):
        p = pins.copy()
        p[at] = value
        assert call(torch, off, p, n, part, nparts)[0] == hp.HP_ERR_BAD_CSR
    for i, j in ((e2, e2 + 1), (e2, e2 + 29999), (e2 + 1023, e2 + 1024), (e2 + 4095, e2 + 4096), (e2 + 1, e2 + 20000)):
        p = pins.copy()
        p[j] = p[i]
        assert call(torch, off, p, n, part, nparts)[0] == hp.HP_ERR_BAD_CSR
    for v, value in ((pins[e2 + 7], -1), (pins[e2 + 20000], nparts)):
        q = part.copy()
        q[v] = value
        assert call(torch, off, pins, n, q, nparts)[0] == hp.HP_ERR_INVALID_ARG
    assert call(torch, off, pins, n, part, nparts) == ok


@pytest.mark.parametrize("kind", [0, 1])
def test_statistics_of_a_partition(torch, kind):
    off, pins = make(9000, [8500, 2, 3, 4, 5, 6] * 3, 4)
    g = inputs.Hypergraph(9000, off, pins, np.maximum(np.diff(off) // 3, 1).astype(np.int32), None)
    r = hp.partition(g, 600, 10 ** 6, seed=1, max_levels=5, trace=True, count_kind=kind)
    o = oracle.partition(g, 600, 10 ** 6, seed=1, max_levels=5, trace=True, count_kind=kind)
    assert r.status == o.status == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(r.part, o.part)
    for k, v in o.stats.items():
        assert r.stats[k] == v, k
    assert [t["conn"] for t in r.trace] == [t["conn"] for t in o.trace]


def test_one_hyperedge_against_many(torch):
    # the same 16 M pins as one hyperedge and as 4,000: a warp alone with them takes 5,000 times as long
    n, total = 17_000_000, 16_000_000
    pins = torch.arange(total, device="cuda", dtype=torch.int32)
    part = (torch.arange(n, device="cuda") % 300).int()
    best = []
    for size in (total, 4000):
        off = torch.arange(0, total + 1, size, device="cuda").int()
        t = []
        for _ in range(4):
            torch.cuda.synchronize()
            a = time.perf_counter()
            rc, conn, cut = hp.hp_connectivity(pins.data_ptr(), off.data_ptr(), off.numel() - 1, None, part.data_ptr(), n, 300)
            t.append(time.perf_counter() - a)
            assert rc == hp.HP_OK and conn == (off.numel() - 1) * 299
        best.append(min(t))
    assert best[0] < 400 * best[1]
