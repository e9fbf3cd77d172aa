"""A hypergraph whose pins end at the last position an int32 offset can hold:
the kernels' strides past a hyperedge's end must not wrap."""
import pytest

from paper_2605_20497_gb300 import hp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_20497_gb300 import build
    build.build()
    hp.load()
    return t


def test_connectivity_at_the_last_pin_position(torch):
    last = 2 ** 31 - 1
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 24 GB")
    n, size, nparts = 100_000, 4096, 321
    # hyperedges of 4,096 consecutive nodes, the last 4,095 pins cut into 3,690 + 200 + 200 + 5
    off = torch.arange(0, last, size, device="cuda", dtype=torch.int64)
    tail = last - 405 + torch.tensor([0, 200, 400], device="cuda")
    off = torch.cat([off, tail, torch.tensor([last], device="cuda")])
    e = off.numel() - 1
    start = torch.randint(0, n - size, (e,), device="cuda", generator=torch.Generator("cuda").manual_seed(1)).int()
    whole = last // size
    pins = torch.empty(last, dtype=torch.int32, device="cuda")
    pins[: whole * size].view(whole, size).copy_(torch.arange(size, device="cuda", dtype=torch.int32))
    pins[: whole * size].view(whole, size).add_(start[:whole, None])
    for i in range(whole, e):
        a, b = int(off[i]), int(off[i + 1])
        pins[a:b] = torch.arange(b - a, device="cuda", dtype=torch.int32) + start[i]
    part = (torch.arange(n, device="cuda") * nparts // n).int()
    weights = torch.randint(1, 9, (e,), device="cuda", generator=torch.Generator("cuda").manual_seed(2)).int()
    lam = part[(start + off.diff().int() - 1).long()] - part[start.long()] + 1   # parts are runs of nodes
    want = (int(((lam - 1).long() * weights).sum()), int(weights[lam > 1].long().sum()))
    off = off.int()
    for call in (hp.hp_connectivity, hp.hp_connectivity_noalloc):
        rc, conn, cut = call(pins.data_ptr(), off.data_ptr(), e, weights.data_ptr(), part.data_ptr(), n, nparts)
        assert rc == hp.HP_OK, hp.hp_last_error()
        assert (conn, cut) == want
