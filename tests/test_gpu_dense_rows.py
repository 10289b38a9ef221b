"""Fixed-point alphas on the two dense kernels: unpadded stride-1 rows, few filters -- many rows on the
kernel that converts in flight, fewer on the one that reads an fp16 copy.  Every sum is below 2^24, so
both give the exact value rounded once, on either side of the line between them."""
import zlib

import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import make_codes, quantize_oracle, random_acts, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _clean_status():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    yield
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


@pytest.mark.parametrize("case", [(80001, 64, 64, 4, "u8"), (80001, 64, 70, 8, "s8"),   # at least two whole waves
                                  (60001, 320, 64, 4, "u8"), (60001, 256, 66, 4, "s8"),  # 18 and 15 MB of rows
                                  (257, 128, 640, 16, "u8"),
                                  # fewer tiles than SMs: 256 channels and more; whole waves: 256 filters and more
                                  (3001, 256, 130, 4, "u8"), (3001, 320, 130, 4, "s8"), (20001, 128, 256, 8, "u8"),
                                  (20001, 128, 260, 8, "s8")], ids=lambda c: "x".join(map(str, c)))
def test_gemm_qa_rows_exact(case):
    P, K, M, G, act = case
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    w = (rng.standard_normal((M, K)) * np.sqrt(2.0 / K)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    a, asc, _ = O.quantize_alpha(al, 8)
    q, sc, packed = quantize_oracle(random_acts((P, K), act, rng), act)
    sums = q.astype(np.int64) @ (np.repeat(a, G, axis=1)[:, :K].astype(np.int64) * t.astype(np.int64)).T
    assert np.abs(sums).max() < 2 ** 24
    want = (sums * (asc.astype(np.float64) * float(sc))).astype(np.float32)
    got = fgq.fgq_gemm_qa(to_dev(packed), act, to_dev(np.array([sc], np.float32)), P, K, to_dev(codes.view(np.int32)),
                          to_dev(a.astype(np.uint8)), 8, to_dev(asc), M, G)
    assert fgq.fgq_last_path() == fgq.PATH_DENSE
    assert np.array_equal(got.cpu().numpy(), want)
