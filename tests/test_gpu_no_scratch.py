"""Calls on a device without memory for their temporaries (the requests fail through a test control): what
the dp4a kernel or the in-flight dense kernel can run is run by them, the rest is an error, and neither
leaves an error behind for the calls after it."""
import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import check_within, make_codes, quantize_oracle, random_acts, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _restore():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    yield
    fgq.fgq_debug_set_scratch_limit(-1)
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


def _layer(C, G, act="u8", seed=3):
    rng = np.random.default_rng(seed + C + G)
    B, H, W, M = 2, 20, 20, 128
    t, al, codes = make_codes(rng.standard_normal((M, 9 * C)).astype(np.float32), G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), act, rng), act)
    y, ym = O.conv2d(q, sc, 3, 3, 1, 1, 1, t, al, G)
    return (to_dev(packed), act, to_dev(np.array([sc], np.float32)), B, H, W, C, 3, 3, 1, 1, 1,
            to_dev(codes.view(np.int32))), al, M, (q, sc, t, y, ym)


@pytest.mark.parametrize("C,G,act", [(64, 4, "u8"), (72, 4, "s8"), (64, 8, "u8"), (48, 16, "u4"), (96, 32, "u8"),
                                     (144, 64, "u8")])
def test_folded_layers_run_on_dp4a(C, G, act):
    head, al, M, (_, _, _, y, ym) = _layer(C, G, act)
    ad = to_dev(al)
    fgq.fgq_set_path(fgq.PATH_SIMT)
    want = fgq.fgq_conv2d(*head, ad, M, G).cpu().numpy()
    fgq.fgq_set_path(fgq.PATH_AUTO)
    fgq.fgq_debug_set_scratch_limit(1024)
    got = fgq.fgq_conv2d(*head, ad, M, G).cpu().numpy()
    assert fgq.fgq_last_path() == fgq.PATH_SIMT
    assert np.array_equal(got, want)
    fgq.fgq_debug_set_scratch_limit(-1)
    got = fgq.fgq_conv2d(*head, ad, M, G).cpu().numpy()
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got, y, ym, "after a call without scratch")


def test_forced_paths_and_whole_groups_fail():
    for C, G, path in ((64, 4, fgq.PATH_TC), (64, 64, fgq.PATH_AUTO)):
        head, al, M, (_, _, _, y, ym) = _layer(C, G)
        fgq.fgq_set_path(path)
        fgq.fgq_debug_set_scratch_limit(1024)
        with pytest.raises(fgq.FGQError) as e:
            fgq.fgq_conv2d(*head, to_dev(al), M, G)
        assert e.value.code == fgq.FGQ_ERR_CUDA
        fgq.fgq_debug_set_scratch_limit(-1)
        check_within(fgq.fgq_conv2d(*head, to_dev(al), M, G).cpu().numpy(), y, ym, "after the error")


@pytest.mark.parametrize("limit", [2 * 128 * 576 + 128 * 4 + 256, -1])
def test_fixed_point_alphas_without_room_for_activations(limit):
    """The folded weights need 2 * 128 * 576 bytes, the fp16 activations 2 * 800 * 64 more."""
    head, al, M, (q, sc, t, _, _) = _layer(64, 4)
    a8, asc, _ = O.quantize_alpha(al, 8)
    y, _ = O.conv2d(q, sc, 3, 3, 1, 1, 1, t, O.dequantize_alpha(a8, asc), 4)
    fgq.fgq_debug_set_scratch_limit(limit)
    got = fgq.fgq_conv2d_qa(*head, to_dev(a8.astype(np.uint8)), 8, to_dev(asc), M, 4).cpu().numpy()
    assert fgq.fgq_last_path() == fgq.PATH_DENSE
    assert np.array_equal(got, y.astype(np.float32))
