"""The folded tensor-core kernel (G = 4, 8, 16, 32: alphas on a common grid per about 256 reduction
elements, in one or two pairs of fp16 parts) against the oracle, inside the contraction tolerance: channel counts that are no multiple of the K-tile,
groups that straddle filter taps, the edges of units and tiles, strided pixels, conv groups,
4-bit codes, and alphas and activations chosen so that only small alphas contribute."""
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
    # B, H, W, C, M, R, S, stride, pad, groups, G, act
    (2, 9, 11, 96, 128, 5, 5, 1, 2, 2, 4, "s8"),      # 48 channels per conv group: padded K-tiles
    (1, 13, 9, 72, 70, 3, 3, 1, 1, 1, 8, "u8"),       # 72 channels: a K-tile of 8 real channels
    (1, 9, 9, 20, 64, 5, 5, 1, 1, 1, 16, "u8"),       # 20 channels: groups of 16 straddle taps
    (1, 7, 8, 18, 66, 5, 5, 2, 2, 1, 4, "u4"),        # groups of 4 straddle taps, M % 4 != 0, 4-bit
    (1, 8, 7, 90, 64, 3, 1, 1, 0, 1, 32, "s4"),       # 90 channels, no padding
    (2, 15, 15, 272, 64, 1, 1, 2, 0, 1, 8, "u8"),     # strided 1x1 on padded channels
    (3, 14, 14, 128, 256, 3, 3, 1, 1, 1, 32, "s8"),   # 18 K-tiles: units of 4 and a rest of 2
    (2, 16, 16, 64, 192, 1, 1, 1, 0, 1, 4, "u8"),     # one K-tile, P = 512: whole tiles
    (1, 17, 19, 256, 64, 1, 1, 1, 0, 1, 4, "u8"),     # one whole unit
    (1, 17, 19, 320, 64, 1, 1, 1, 0, 1, 4, "s4"),     # a unit and one K-tile
    (1, 40, 40, 64, 130, 3, 3, 1, 1, 1, 8, "u8"),     # M % 4 != 0: direct stores
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_fold_conv2d_parity(case):
    B, H, W, C, M, R, S, stride, pad, groups, G, act = case
    rng = np.random.default_rng(zlib.crc32(repr(case).encode()))
    Kred = R * S * (C // groups)
    w = (rng.standard_normal((M, Kred)) * np.sqrt(2.0 / Kred)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    y, ym = O.conv2d(q, sc, R, S, stride, pad, groups, t, al, G)
    args = (to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, R, S, stride, pad, groups,
            to_dev(codes.view(np.int32)), to_dev(al), M, G)
    if Kred <= 256:  # the automatic choice is the dp4a kernel
        fgq.fgq_set_path(fgq.PATH_TC)
    got = fgq.fgq_conv2d(*args)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got.cpu().numpy(), y, ym, f"fold conv2d {case}")
    # the requantized codes are the quantizer applied to the same fp32 output
    y32 = got.cpu().numpy().reshape(-1)
    scale = np.float32(2.0 ** O.dfp_exponent(y32, O.U8))
    rq = fgq.fgq_conv2d_rq(*args, "u8", to_dev(np.array([scale], np.float32))).cpu().numpy().reshape(-1)
    want, _, _, _ = O.quantize(y32, O.U8, scale_in=scale)
    assert np.array_equal(rq.astype(np.int64), want.astype(np.int64)), f"fold conv2d_rq {case}"


@pytest.mark.parametrize("P,K,M,G,act", [(9, 300, 64, 4, "u8"), (200, 1000, 100, 8, "s8"), (65, 520, 64, 16, "u4"),
                                         (300, 2048, 1000, 32, "u8"), (64, 9216, 128, 4, "s8")])
def test_fold_gemm_parity(P, K, M, G, act):
    rng = np.random.default_rng(P + K)
    w = rng.standard_normal((M, K)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    q, sc, packed = quantize_oracle(random_acts((P, K), act, rng), act)
    y, ym = O.gemm(q, sc, t, al, G)
    got = fgq.fgq_gemm(to_dev(packed), act, to_dev(np.array([sc], np.float32)), P, K, to_dev(codes.view(np.int32)),
                       to_dev(al), M, G)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got.cpu().numpy(), y, ym, f"fold gemm {(P, K, M, G, act)}")


@pytest.mark.parametrize("G,spread", [(4, 30), (8, 16), (16, 8), (4, 6), (32, 0)])
def test_fold_spread_alphas(G, spread):
    """Alphas down to 2^-spread of the row's largest, and activations for which every group with a
    large alpha sums to zero (equal values, codes +1 and -1) while its products are as large as
    they get: the output is carried by the small alphas alone, inside the tolerance of their own
    sum.  Positions whose every group sum is zero must give exactly zero."""
    P, K, M = 130, 768, 128
    rng = np.random.default_rng(100 * G + spread)
    ng = K // G
    al = (rng.uniform(1.0, 2.0, (M, ng)) * 2.0 ** -rng.integers(0, spread + 1, (M, ng))).astype(np.float32)
    t = rng.integers(-1, 2, (M, ng, G)).astype(np.int8)
    big = al >= 2.0 ** -(spread // 2)
    half = np.concatenate([np.ones(G // 2), -np.ones(G // 2)]).astype(np.int8)
    t[big] = half
    al[:3] = 0.0  # rows without any weight
    t[:3] = 0
    t = t.reshape(M, K)
    q = np.repeat(rng.integers(0, 256, (P, ng)), G, axis=1).astype(np.int32)  # equal inside a group
    q[P // 2:] = rng.integers(0, 256, (P - P // 2, K))
    q[0] = 255
    sc = np.float32(2.0 ** -6)
    y, ym = O.gemm(q, sc, t, al, G)
    got = fgq.fgq_gemm(to_dev(O.pack_act(q, O.U8)), "u8", to_dev(np.array([sc], np.float32)), P, K,
                       to_dev(O.pack_codes(t).view(np.int32)), to_dev(al), M, G).cpu().numpy()
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got, y, ym, f"spread alphas G={G} 2^-{spread}")
    assert np.all(got[ym == 0] == 0)


def test_fold_saturated_sums():
    """All codes +1, alphas and activations near their maxima: a unit's sum passes 2^24, where the
    accumulator rounds; 64 units."""
    P, K, M, G = 70, 16384, 64, 4
    rng = np.random.default_rng(7)
    t = np.ones((M, K), np.int8)
    al = rng.uniform(1.9, 2.0, (M, K // G)).astype(np.float32)
    q = rng.integers(230, 256, (P, K)).astype(np.int32)
    sc = np.float32(0.5)
    y, ym = O.gemm(q, sc, t, al, G)
    got = fgq.fgq_gemm(to_dev(O.pack_act(q, O.U8)), "u8", to_dev(np.array([sc], np.float32)), P, K,
                       to_dev(O.pack_codes(t).view(np.int32)), to_dev(al), M, G).cpu().numpy()
    check_within(got, y, ym, "saturated sums")


@pytest.mark.parametrize("G,act,C,R,path", [
    (4, "u8", 256, 1, fgq.PATH_SIMT), (4, "u8", 288, 1, fgq.PATH_TC), (8, "u8", 320, 1, fgq.PATH_SIMT),
    (8, "s8", 352, 1, fgq.PATH_TC), (16, "s8", 384, 1, fgq.PATH_SIMT), (16, "u8", 416, 1, fgq.PATH_TC),
    (32, "u8", 448, 1, fgq.PATH_SIMT), (32, "u8", 480, 1, fgq.PATH_TC), (32, "u8", 32, 3, fgq.PATH_SIMT),
    (32, "u8", 36, 3, fgq.PATH_TC), (32, "u4", 288, 1, fgq.PATH_TC)])
def test_small_layers_choice(G, act, C, R, path):
    """Both sides of the line up to which one wave of dp4a blocks is done before the folded kernel."""
    rng = np.random.default_rng(C)
    B, H, W, M = 1, 12, 14, 64
    w = rng.standard_normal((M, R * R * C)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    y, ym = O.conv2d(q, sc, R, R, 1, R // 2, 1, t, al, G)
    got = fgq.fgq_conv2d(to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, 1, R // 2, 1,
                         to_dev(codes.view(np.int32)), to_dev(al), M, G)
    assert fgq.fgq_last_path() == path
    check_within(got.cpu().numpy(), y, ym, f"small layer G={G} C={C}")
