"""A process that has seen many hypergraphs of different sizes is as fast as one
that has seen few: what the library keeps per kernel and size is bounded."""
import ctypes
import statistics
import time

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


def test_calls_after_many_level_sizes(torch):
    most = 16_300   # every level size asks for its own table sizes
    i32 = lambda *a: torch.tensor(a, dtype=torch.int32, device="cuda")
    off, pins, src, w = i32(0, 2), i32(0, 1), i32(1), i32(1)
    size = torch.ones(most, dtype=torch.int32, device="cuda")
    cand = torch.empty(most * 4, dtype=torch.int32, device="cuda")
    score = torch.empty(most * 4, dtype=torch.int64, device="cuda")
    mate = torch.empty(most, dtype=torch.int32, device="cuda")
    opt = hp.options()

    def step(n):
        a = time.perf_counter()
        rc, pairs = hp.hp_debug_coarsen_level(n, 1, off.data_ptr(), pins.data_ptr(), src.data_ptr(), w.data_ptr(),
                                              size.data_ptr(), 4, 4, 1, 0, ctypes.byref(opt), cand.data_ptr(),
                                              score.data_ptr(), mate.data_ptr())
        assert rc == hp.HP_OK and pairs >= 1
        return time.perf_counter() - a

    median = lambda n: statistics.median([step(n) for _ in range(60)][20:])
    median(502)                        # a size the process sees first
    for n in range(most, 500, -1):
        step(n)
    assert median(501) < 1.2 * median(502)   # the one it sees last
