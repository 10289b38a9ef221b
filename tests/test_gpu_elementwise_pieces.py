"""Residual additions and max pooling at the edges of their 16-byte pieces: sizes around 16, addresses
that are not 16-byte aligned, channel counts that are and are not multiples of 16."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,off", [(1, 0), (15, 0), (16, 0), (17, 0), (4099, 0), (4099, 1), (4096, 8)])
def test_add_codes_pieces(n, off):
    rng = np.random.default_rng(n + off)
    ra, rb = rng.integers(0, 256, n + 16, dtype=np.uint8), rng.integers(0, 256, n + 16, dtype=np.uint8)
    da, db = to_dev(ra)[off:off + n], to_dev(rb)[:n]
    qa, qb = ra[off:off + n].view(np.int8).astype(np.int64), rb[:n].astype(np.int64)
    sa, sb = np.float32(0.25), np.float32(0.125)
    dsa, dsb = to_dev(np.array([sa])), to_dev(np.array([sb]))
    want = O.add_codes(qa, sa, qb, sb)
    assert np.array_equal(fgq.fgq_add_codes(da, "s8", dsa, db, "u8", dsb).cpu().numpy(), want)
    so = np.float32(2.0 ** O.dfp_exponent(want, O.U8))
    out = torch.empty(n + 16, dtype=torch.uint8, device=da.device)[off:off + n]
    got = fgq.fgq_add_codes(da, "s8", dsa, db, "u8", dsb, "u8", to_dev(np.array([so])), out=out)
    assert np.array_equal(got.cpu().numpy().astype(np.int64), O.quantize(want, O.U8, scale_in=so)[0])


@pytest.mark.parametrize("C,off", [(16, 0), (48, 0), (20, 0), (32, 4)])
def test_maxpool_pieces(C, off):
    shape = (2, 9, 7, C)
    raw = np.random.default_rng(C + off).integers(0, 256, int(np.prod(shape)) + 16, dtype=np.uint8)
    q = raw[off:off + int(np.prod(shape))].reshape(shape)
    x = to_dev(raw)[off:off + int(np.prod(shape))].view(shape)
    assert np.array_equal(fgq.fgq_maxpool_u8(x, *shape, 3, 2, 1).cpu().numpy(), O.maxpool_codes(q, 3, 2, 1))
