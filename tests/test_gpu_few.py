"""8-bit-weight convolutions of few channels read in place from rows of fp16 pixels: every sum is an exact
integer, so the outputs equal the oracle's values rounded once (and the dp4a path's), at the edges of
the form: one and eight channels, runs of 32 and 64 elements, strides that divide nothing, one and 256
output columns, partial row tiles, no padding and more padding than needed, ragged filter counts."""
import zlib

import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import quantize_oracle, random_acts, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _clean_status():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    yield
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


CASES = [
    # B, H, W, C, M, R, S, stride, pad, act
    (2, 67, 67, 3, 64, 11, 11, 4, 2, "u8"),   # 11 taps of 4 channels: runs of 64
    (3, 19, 23, 3, 70, 3, 3, 1, 1, "s8"),     # odd stride: 8 channels per pixel; M % 4 != 0
    (1, 33, 29, 8, 132, 5, 5, 1, 2, "u8"),    # 8 channels, two filter tiles
    (1, 3, 256, 1, 64, 1, 1, 1, 0, "s8"),     # 256 output columns, one product
    (3, 9, 5, 4, 32, 7, 5, 2, 0, "u8"),       # one output column
    (2, 20, 23, 5, 64, 3, 3, 3, 4, "u8"),     # stride 3, windows that lie wholly in the padding
    (2, 31, 30, 2, 64, 1, 16, 6, 1, "s8"),    # one filter row of 16 taps, stride 6
    (2, 51, 51, 3, 96, 11, 11, 4, 0, "s8"),   # 96 operand rows, two output boxes a warp
    (1, 40, 44, 6, 64, 8, 8, 2, 3, "u8"),     # 8 pieces a run in two planes
    (1, 12, 260, 3, 64, 3, 3, 1, 1, "u8"),    # 260 output columns: not covered, im2col rows
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_few_conv2d_w8_exact(case):
    B, H, W, C, M, R, S, stride, pad, act = case
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    w = rng.standard_normal((M, R * S * C)).astype(np.float32)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    wq, ws = O.quantize_weights_w8(w)
    y, _ = O.conv2d_w8(q, sc, R, S, stride, pad, 1, wq, ws)
    args = (to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, R, S, stride, pad, 1, to_dev(wq),
            to_dev(ws), M)
    got = fgq.fgq_conv2d_w8(*args).cpu().numpy()
    assert fgq.fgq_last_path() == fgq.PATH_DENSE
    assert np.array_equal(got, y.astype(np.float32))
    y32 = y.astype(np.float32).reshape(-1)
    scale = np.float32(2.0 ** O.dfp_exponent(y32, O.S8))
    rq = fgq.fgq_conv2d_w8_rq(*args, "s8", to_dev(np.array([scale], np.float32))).cpu().numpy()
    want, _, _, _ = O.quantize(y32, O.S8, scale_in=scale)
    assert np.array_equal(rq.reshape(-1).view(np.int8).astype(np.int64), want.astype(np.int64))


def test_few_largest_sums():
    """8 x 8 taps of 8 channels at full scale: 512 products of 255 * 127, sums just below 2^24."""
    B, H, W, C, M, R, S = 1, 9, 10, 8, 64, 8, 8
    wq = np.full((M, R * S * C), 127, np.int8)
    wq[::2] = -127
    x = np.full((B, H, W, C), 255, np.uint8)
    ws = np.full(M, 0.25, np.float32)
    got = fgq.fgq_conv2d_w8(to_dev(x), "u8", to_dev(np.array([0.5], np.float32)), B, H, W, C, R, S, 1, 0, 1, to_dev(wq),
                            to_dev(ws), M).cpu().numpy().reshape(-1, M)
    want = 0.125 * 512 * 255 * 127
    assert (got[:, ::2] == -want).all() and (got[:, 1::2] == want).all()
