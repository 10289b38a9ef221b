"""The batched quantizer's cooperative launch where the context keeps fewer blocks resident than the device
would (a test control refuses the larger launches as the runtime does), and its wait for a tensor's
maximum, run out on purpose."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import ORACLE_TYPE, dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _restore():
    yield
    fgq.fgq_debug_set_resident_blocks(-1)
    fgq.fgq_debug_set_wait_limit_us(-1)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


@pytest.mark.parametrize("blocks", [1, 3, 200])
def test_fewer_resident_blocks(blocks):
    rng = np.random.default_rng(blocks)
    ts = ["u8", "s4", "s8", "u4"]
    xs = [(rng.standard_normal(n) * 3).astype(np.float32) for n in (5, 7 * 16384 + 5, 16384, 40 * 16384 - 2)]
    fgq.fgq_debug_set_resident_blocks(blocks)
    got = fgq.fgq_quantize_act_batch([torch.from_numpy(x).to(dev()) for x in xs], ts)
    for x, t, (q, sc) in zip(xs, ts, got):
        qo, so, _, _ = O.quantize(x, ORACLE_TYPE[t])
        assert float(sc.item()) == float(so)
        assert np.array_equal(q.cpu().numpy(), O.pack_act(qo, ORACLE_TYPE[t])), (t, x.size)


def test_no_resident_block_is_an_error():
    x = torch.ones(100, device=dev())
    fgq.fgq_debug_set_resident_blocks(0)
    with pytest.raises(fgq.FGQError) as e:
        fgq.fgq_quantize_act_batch([x], ["u8"])
    assert e.value.code == fgq.FGQ_ERR_CUDA
    fgq.fgq_debug_set_resident_blocks(-1)
    q, sc = fgq.fgq_quantize_act_batch([x], ["u8"])[0]
    assert (q == 128).all() and float(sc.item()) == 2.0 ** -7


def test_wait_for_the_maximum_expires():
    """One tensor of more items than blocks: some block reaches its codes while another still reduces."""
    x = torch.randn(1 << 25, device=dev(), generator=torch.Generator(device="cuda").manual_seed(5))
    q0, s0 = fgq.fgq_quantize_act(x, "s8")
    fgq.fgq_debug_set_wait_limit_us(0)
    seen = []
    for _ in range(12):
        fgq.fgq_quantize_act_batch([x], ["s8"])
        seen.append(fgq.fgq_stream_status())
        if seen[-1] == fgq.FGQ_ERR_TIMEOUT:
            break
    assert seen[-1] == fgq.FGQ_ERR_TIMEOUT, seen
    fgq.fgq_debug_set_wait_limit_us(-1)
    q, s = fgq.fgq_quantize_act_batch([x], ["s8"])[0]
    assert fgq.fgq_stream_status() == fgq.FGQ_OK
    assert torch.equal(q, q0) and torch.equal(s, s0)
