"""hp_connectivity over what its one-pass form and its general form take:
part counts around the bit rows' sizes and beyond them, hyperedge sizes around
a warp's loads, sorted and unsorted destinations, weights, and every error
against the general form's answer."""
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


def call(torch, off, pins, n, part, nparts, weights=None):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()
    o, p, q = t(off), t(pins), t(part)
    w = None if weights is None else t(weights)
    return hp.hp_connectivity(p.data_ptr(), o.data_ptr(), len(off) - 1, None if w is None else w.data_ptr(),
                              q.data_ptr(), n, nparts)


def count(off, pins, part, weights=None):
    conn = cut = 0
    for e in range(len(off) - 1):
        lam = len(set(part[pins[off[e]:off[e + 1]]].tolist()))
        w = 1 if weights is None else int(weights[e])
        conn += w * (lam - 1)
        cut += w * (lam > 1)
    return conn, cut


def make(n, sizes, seed, ordered=True):
    rng = np.random.default_rng(seed)
    rows = []
    for k in sizes:
        r = rng.choice(n, size=k, replace=False)
        rows.append(np.concatenate([r[:1], np.sort(r[1:])]) if ordered else r)
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([len(r) for r in rows])
    return off.astype(np.int32), np.concatenate(rows).astype(np.int32)


@pytest.mark.parametrize("nparts", [1, 2, 32, 33, 1023, 1024, 1025, 2049, 32768, 32769])
@pytest.mark.parametrize("ordered", [True, False])
def test_part_counts(torch, nparts, ordered):
    n = 3000
    off, pins = make(n, [1, 2, 3, 31, 32, 33, 64, 65, 127, 128, 129, 130, 257, 700] * 12, nparts, ordered)
    rng = np.random.default_rng(nparts)
    part = rng.integers(0, nparts, n).astype(np.int32)
    w = rng.integers(1, 65537, len(off) - 1).astype(np.int32)
    for weights in (None, w):
        st, c, cn = call(torch, off, pins, n, part, nparts, weights)
        assert st == hp.HP_OK and (c, cn) == count(off, pins, part, weights)


def test_errors(torch):
    n, nparts = 200, 9
    off, pins = make(n, [5, 40, 140, 3] * 9, 1)
    rng = np.random.default_rng(2)
    part = rng.integers(0, nparts, n).astype(np.int32)
    ok = call(torch, off, pins, n, part, nparts)
    assert ok[0] == hp.HP_OK
    bad_csr, bad_arg = hp.HP_ERR_BAD_CSR, hp.HP_ERR_INVALID_ARG
    e2 = int(off[2])
    cases = []
    for at, value in ((e2 + 100, n), (e2 + 100, -1), (0, 2**31 - 1), (len(pins) - 1, -2**31)):   # pins out of range
        p = pins.copy()
        p[at] = value
        cases.append((off, p, part, None, bad_csr))
    for i, j in ((e2, e2 + 139), (e2 + 31, e2 + 32), (e2 + 127, e2 + 128), (e2 + 1, e2 + 139)):   # a pin twice
        p = pins.copy()
        p[j] = p[i]
        cases.append((off, p, part, None, bad_csr))
    for i in (0, 3, len(off) - 1):   # offsets
        o = off.copy()
        o[i] = o[i - 1] if i else 1
        cases.append((o, pins, part, None, bad_csr))
    for value in (0, -5, 65537):
        w = np.ones(len(off) - 1, np.int32)
        w[7] = value
        cases.append((off, pins, part, w, bad_arg))
        p = pins.copy()
        p[e2 + 139] = p[e2 + 138]
        cases.append((off, p, part, w, bad_csr))
    for v, value in ((0, -1), (n - 1, nparts)):
        q = part.copy()
        q[v] = value
        cases.append((off, pins, q, None, bad_arg))
        p = pins.copy()
        p[5] = n
        cases.append((off, p, q, None, bad_csr))
    for o, p, q, w, want in cases:
        assert call(torch, o, p, n, q, nparts, w)[0] == want
    assert call(torch, off, pins, n, part, nparts) == ok
    # no hyperedges, no nodes
    assert call(torch, np.zeros(1, np.int32), np.zeros(1, np.int32), n, part, nparts) == (hp.HP_OK, 0, 0)
