"""The folded kernel where a filter has few groups (G = 8 to 32: units take both pairs of parts) and at
G = 64 on channel counts that fill no whole K-tiles (18 groups or more; fewer stay on dp4a):
against the oracle, and no further from it than the dp4a kernel is."""
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


CASES = [
    # B, H, W, C, M, R, stride, pad, groups, G, act, expected path
    (2, 28, 28, 128, 64, 3, 1, 1, 1, 64, "u8", fgq.PATH_TC),    # 18 whole groups (the per-group kernel)
    (1, 20, 20, 96, 64, 4, 1, 1, 1, 64, "u8", fgq.PATH_TC),     # 24 groups of 64 over 96 channels
    (1, 20, 20, 72, 64, 4, 1, 1, 1, 64, "u8", fgq.PATH_SIMT),   # 18 groups, but 8 units: dp4a
    (1, 20, 20, 68, 64, 4, 1, 1, 1, 64, "u8", fgq.PATH_SIMT),   # 17 groups: dp4a
    (2, 13, 13, 200, 130, 3, 1, 1, 1, 64, "s8", fgq.PATH_TC),   # 29 groups, M % 4 != 0
    (2, 13, 13, 144, 130, 4, 1, 2, 1, 128, "s8", fgq.PATH_SIMT),
    (2, 14, 14, 96, 128, 5, 1, 2, 2, 64, "s4", fgq.PATH_TC),    # conv groups of 48 channels, 4-bit codes
    (1, 24, 24, 64, 64, 3, 1, 1, 1, 32, "u8", fgq.PATH_TC),     # 18 groups
    (1, 24, 24, 60, 64, 3, 1, 1, 1, 32, "u8", fgq.PATH_TC),     # 17 groups
    (1, 20, 20, 272, 64, 1, 1, 0, 1, 16, "s8", fgq.PATH_TC),    # 17 groups, two units
    (1, 20, 20, 264, 64, 1, 2, 0, 1, 128, "u8", fgq.PATH_SIMT),  # 3 groups
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_few_groups(case):
    B, H, W, C, M, R, stride, pad, groups, G, act, path = case
    rng = np.random.default_rng(zlib.crc32(repr(case[:-1]).encode()))
    Kred = R * R * (C // groups)
    w = (rng.standard_normal((M, Kred)) * np.sqrt(2.0 / Kred)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    y, ym = O.conv2d(q, sc, R, R, stride, pad, groups, t, al, G)
    args = (to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, stride, pad, groups,
            to_dev(codes.view(np.int32)), to_dev(al), M, G)
    got = fgq.fgq_conv2d(*args).cpu().numpy()
    assert fgq.fgq_last_path() == path
    check_within(got, y, ym, f"few groups {case}")
    fgq.fgq_set_path(fgq.PATH_SIMT)
    simt = fgq.fgq_conv2d(*args).cpu().numpy()
    err = np.sqrt(np.mean((got.astype(np.float64) - y) ** 2))
    ref = np.sqrt(np.mean((simt.astype(np.float64) - y) ** 2))
    rms = np.sqrt(np.mean(y ** 2))
    # an error that is not the smaller one is within the spread of two draws of such roundings
    assert err <= 1.1 * ref + 0.05 * 2.0 ** -24 * rms, (err / rms, ref / rms)
