"""The batched quantizer's exponents and items, bit for bit against the oracle: maxima on both sides of
every rounding line of the exponent (powers of two times the largest code, subnormals, the largest
float), zero and negative tensors, and sizes at the edges of its items, in calls of at most 32 tensors
and of more."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import ORACLE_TYPE, dev

pytestmark = pytest.mark.gpu

QMAX = {"u8": 255, "s8": 127, "u4": 15, "s4": 7}


@pytest.fixture(autouse=True)
def _clean_status():
    yield
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


def _check(xs, ts):
    got = fgq.fgq_quantize_act_batch([torch.from_numpy(x).to(dev()) for x in xs], ts)
    for x, t, (q, sc) in zip(xs, ts, got):
        qo, so, _, _ = O.quantize(x, ORACLE_TYPE[t])
        assert float(sc.item()) == float(so), (t, x.max())
        assert np.array_equal(q.cpu().numpy(), O.pack_act(qo, ORACLE_TYPE[t])), (t, x.size)


@pytest.mark.parametrize("t", list(QMAX))
def test_exponent_edges(t):
    tops = []
    for e in (-149, -146, -140, -133, -127, -126, -3, 0, 1, 60, 119):
        v = np.float32(QMAX[t]) * np.float32(2.0) ** np.float32(e) if e > -126 else np.ldexp(np.float32(QMAX[t]), e)
        v = np.float32(v)
        tops += [np.nextafter(v, np.float32(0)), v, np.nextafter(v, np.float32(np.inf))]
    tops += [np.float32(2.0 ** -149), np.finfo(np.float32).max, np.float32(0), np.float32(-3.5)]
    xs = [np.array([0.25 * top, -top, 0.0, top], np.float32) for top in tops if np.isfinite(top)]
    _check(xs, [t] * len(xs))          # more than 32 tensors
    _check(xs[:32], [t] * len(xs[:32]))


@pytest.mark.parametrize("n", [16383, 16384, 16385, 32768 + 1027, 3 * 16384 + 4])
def test_item_edges(n):
    rng = np.random.default_rng(n)
    xs, ts = [], []
    for i, t in enumerate(QMAX):
        x = (rng.standard_normal(n) * 3).astype(np.float32)
        x[[0, n - 1][i & 1]] = 77.7  # the maximum in the first or the last item
        xs.append(x)
        ts.append(t)
    _check(xs, ts)


@pytest.mark.parametrize("dtype", [torch.float16, torch.float64, torch.int32])
def test_inputs_are_fp32(dtype):
    """A tensor of another type would be read as fp32, an fp16 one past its end."""
    with pytest.raises(TypeError):
        fgq.fgq_quantize_act_batch([torch.ones(64, device=dev()), torch.ones(64, device=dev()).to(dtype)], ["u8", "u8"])
