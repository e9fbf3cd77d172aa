"""GPU parity of the MLP's two forms: row counts around a warp's 32 rows,
rows that do not start on a word, and biases and shifts on both sides of what
the fp16 form takes (the offset b / 2^s + 1024 a float), with pre-activations
far below and above the activation range."""
import ctypes

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


@pytest.mark.parametrize("count", [1, 31, 32, 33, 255, 256, 257, 40001])
@pytest.mark.parametrize("start", [0, 1, 2, 4])
def test_counts_and_alignment(torch, count, start):
    rng = np.random.default_rng(count)
    feat = rng.integers(0, 256, size=(count, 16)).astype(np.uint8)
    buf = torch.zeros(count * 16 + 16, dtype=torch.uint8, device="cuda")
    buf[start:start + count * 16] = torch.from_numpy(feat.reshape(-1)).cuda()
    out = torch.full((count + 1,), 77, dtype=torch.int32, device="cuda")
    m = inputs.random_merge_model(count)
    mm = hp.merge_model(m)
    assert hp.hp_merge_scores(buf.data_ptr() + start, count, ctypes.byref(mm), out.data_ptr()) == hp.HP_OK
    assert np.array_equal(out.cpu().numpy()[:count].astype(np.int64), oracle.mlp_scores(feat, m))
    assert int(out[count]) == 77


@pytest.mark.parametrize("shift1,shift2", [(0, 0), (1, 30), (6, 8), (12, 13), (13, 14), (14, 15), (20, 21), (30, 5)])
@pytest.mark.parametrize("bias", [0, 1, 1 << 12, (1 << 23) - 1, 1 << 23, (1 << 24) - 1024, (1 << 24) + 1, 1 << 30])
def test_biases_and_shifts(torch, shift1, shift2, bias):
    rng = np.random.default_rng(bias + shift1)
    feat = rng.integers(0, 256, size=(997, 16)).astype(np.uint8)
    feat[:40] = 255
    feat[40:60] = 0
    m = inputs.random_merge_model(shift1 + 100, bias_scale=64, shift1=shift1, shift2=shift2)
    m.b1[::3] += bias
    m.b1[1::3] -= bias
    m.b2[::4] += bias
    m.b2[1::4] -= bias
    np.clip(m.b1, -2**30, 2**30, out=m.b1)
    np.clip(m.b2, -2**30, 2**30, out=m.b2)
    rc, s = hp.merge_scores(torch.from_numpy(feat).cuda(), m)
    assert rc == hp.HP_OK, hp.hp_last_error()
    assert np.array_equal(s.cpu().numpy().astype(np.int64), oracle.mlp_scores(feat, m))
