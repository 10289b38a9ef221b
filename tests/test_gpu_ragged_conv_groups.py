"""Conv groups whose filters are no multiple of 4 while all filters together are: the second group's rows
start between the four-output stores of the CUDA-core kernel."""
import zlib

import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import check_within, make_codes, quantize_oracle, random_acts, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _clean_status():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    yield
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


@pytest.mark.parametrize("path", [fgq.PATH_SIMT, fgq.PATH_AUTO])
@pytest.mark.parametrize("case", [(2, 66, 32, 4, "u8"), (2, 130, 20, 8, "s8"), (4, 65, 16, 16, "u8"), (2, 70, 64, 64, "u4"),
                                  (2, 6, 64, 128, "u8"), (4, 33, 24, 32, "s4"), (2, 2, 3, 4, "u8")],
                         ids=lambda c: "x".join(map(str, c)))
def test_ragged_filters_of_conv_groups(case, path):
    groups, Mg, Cg, G, act = case
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    B, H, W, R, M, C = 2, 9, 11, 3, groups * Mg, groups * Cg
    t, al, codes = make_codes(rng.standard_normal((M, R * R * Cg)).astype(np.float32), G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    y, ym = O.conv2d(q, sc, R, R, 1, 1, groups, t, al, G)
    args = (to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, 1, 1, groups,
            to_dev(codes.view(np.int32)), to_dev(al), M, G)
    fgq.fgq_set_path(path)
    got = fgq.fgq_conv2d(*args).cpu().numpy()
    check_within(got, y, ym, f"ragged conv groups {case}")
    y32 = got.reshape(-1)
    scale = np.float32(2.0 ** O.dfp_exponent(y32, O.S8))
    rq = fgq.fgq_conv2d_rq(*args, "s8", to_dev(np.array([scale], np.float32))).cpu().numpy().reshape(-1).view(np.int8)
    want, _, _, _ = O.quantize(y32, O.S8, scale_in=scale)
    diff = np.abs(rq.astype(np.int64) - want.astype(np.int64))
    assert diff.max() == 0 or (G >= 64 and diff.max() <= 1)


@pytest.mark.parametrize("groups,Mg", [(2, 66), (4, 65), (1, 66)])
def test_ragged_filters_w8(groups, Mg):
    rng = np.random.default_rng(groups + Mg)
    B, H, W, R, Cg = 2, 9, 11, 3, 5
    M, C = groups * Mg, groups * Cg
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), "u8", rng), "u8")
    wq, ws = O.quantize_weights_w8(rng.standard_normal((M, R * R * Cg)).astype(np.float32))
    y, _ = O.conv2d_w8(q, sc, R, R, 1, 1, groups, wq, ws)
    got = fgq.fgq_conv2d_w8(to_dev(packed), "u8", to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, 1, 1, groups,
                            to_dev(wq), to_dev(ws), M).cpu().numpy()
    assert np.array_equal(got, y.astype(np.float32))
