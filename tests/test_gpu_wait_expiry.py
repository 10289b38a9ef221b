"""Failure detection in the tensor-core contraction kernels themselves: every mbarrier wait
is bounded, and on expiry the kernel records FGQ_ERR_TIMEOUT, every role leaves its loop,
the copies and MMAs already issued are waited for, and the tensor memory is freed.

A test control (fgq_debug_set_wait_limit_us) shortens the waits of this thread's launches
to nothing, so waits that the kernel's own pipeline would satisfy a few microseconds later
run out: no flag is left unset on purpose and nothing faults, traps or hangs.  The next
call with the normal limits, on the same stream, must then be correct against the oracle,
which it could not be if an aborted CTA had kept its tensor memory (its allocation would
never be granted) or left a copy in flight."""
import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import check_within, make_codes, quantize_oracle, random_acts, to_dev

pytestmark = pytest.mark.gpu

TRIES = 12  # calls with the shortened limit until one of them times out


@pytest.fixture(autouse=True)
def _restore():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    fgq.fgq_debug_set_wait_limit_us(-1)
    yield
    fgq.fgq_debug_set_wait_limit_us(-1)
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


@pytest.mark.parametrize("family,G,R", [("tc4", 4, 3), ("tc4", 4, 1), ("tc", 64, 3), ("tc", 64, 1),
                                        ("dense", 4, 3), ("dense", 64, 1)])
def test_forced_wait_expiry_then_exact(family, G, R):
    rng = np.random.default_rng(31 + G + R)
    B, H, W, C, M = 8, 14, 14, 256, 256
    pad = R // 2
    Kred = R * R * C
    w = (rng.standard_normal((M, Kred)) * np.sqrt(2.0 / Kred)).astype(np.float32)
    t, al, codes = make_codes(w, G)
    x = random_acts((B, H, W, C), "u8", rng)
    q, sc, packed = quantize_oracle(x, "u8")
    geo = (B, H, W, C, R, R, 1, pad, 1)
    qd, sd, cd = to_dev(packed), to_dev(np.array([sc], np.float32)), to_dev(codes.view(np.int32))
    if family == "dense":  # 8-bit fixed-point alphas: 3x3 on the dense form of the G >= 64 kernel, 1x1 in flight
        a8, asc, _ = O.quantize_alpha(al, 8)
        ad, ascd = to_dev(a8.astype(np.uint8)), to_dev(asc)

        def call():
            return fgq.fgq_conv2d_qa(qd, "u8", sd, *geo, cd, ad, 8, ascd, M, G)
        al_eff = O.dequantize_alpha(a8, asc)
        want_path = fgq.PATH_DENSE
    else:
        fgq.fgq_set_path(fgq.PATH_TC)

        def call():
            return fgq.fgq_conv2d(qd, "u8", sd, *geo, cd, to_dev(al), M, G)
        al_eff = al
        want_path = fgq.PATH_TC
    y, ym = O.conv2d(q, sc, R, R, 1, pad, 1, t, al_eff, G)

    timed_out = 0
    fgq.fgq_debug_set_wait_limit_us(0)
    for _ in range(TRIES):
        out = call()
        assert fgq.fgq_last_path() == want_path
        st = fgq.fgq_stream_status()
        assert st in (fgq.FGQ_OK, fgq.FGQ_ERR_TIMEOUT), st
        if st == fgq.FGQ_OK:  # every wait happened to be satisfied in time: the result stands
            check_within(out.cpu().numpy(), y, ym, f"{family} unexpired call")
        else:
            timed_out += 1
            break
    fgq.fgq_debug_set_wait_limit_us(-1)
    assert timed_out, f"no wait of {family} ran out in {TRIES} calls"
    # the same stream, normal limits: the kernel runs whole and exact
    for _ in range(2):
        out = call().cpu().numpy()
        assert fgq.fgq_stream_status() == fgq.FGQ_OK
        check_within(out, y, ym, f"{family} after an expired call")


@pytest.mark.parametrize("limit_us", [0, 1, 200])
def test_warp_wait_is_decided_once(limit_us):
    """The lanes of a warp leave a wait together, also where some of them see their phase complete and
    others run out of time: what follows a wait in the kernels are warp-collective instructions."""
    assert fgq.fgq_debug_selftest_warp_wait(limit_us) == fgq.FGQ_ERR_TIMEOUT


@pytest.mark.parametrize("family,G,R", [("tc4", 4, 3), ("tc", 64, 3), ("tc", 64, 1)])
@pytest.mark.parametrize("limit_us", [1, 5])
def test_short_wait_limits(family, G, R, limit_us):
    """Limits near the waits' own lengths, so that the timer decides: some calls expire and some do not,
    those that do not are right, and so is the next call with the normal limits."""
    rng = np.random.default_rng(57 + G + R)
    B, H, W, C, M = 8, 14, 14, 256, 256
    t, al, codes = make_codes(rng.standard_normal((M, R * R * C)).astype(np.float32), G)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), "u8", rng), "u8")
    y, ym = O.conv2d(q, sc, R, R, 1, R // 2, 1, t, al, G)
    args = (to_dev(packed), "u8", to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, 1, R // 2, 1,
            to_dev(codes.view(np.int32)), to_dev(al), M, G)
    fgq.fgq_set_path(fgq.PATH_TC)
    fgq.fgq_debug_set_wait_limit_us(limit_us)
    for _ in range(TRIES):
        out = fgq.fgq_conv2d(*args)
        st = fgq.fgq_stream_status()
        assert st in (fgq.FGQ_OK, fgq.FGQ_ERR_TIMEOUT), st
        if st == fgq.FGQ_OK:
            check_within(out.cpu().numpy(), y, ym, f"{family} limit {limit_us} us")
    fgq.fgq_debug_set_wait_limit_us(-1)
    out = fgq.fgq_conv2d(*args).cpu().numpy()
    assert fgq.fgq_stream_status() == fgq.FGQ_OK
    check_within(out, y, ym, f"{family} after short limits")


def _w8_call(B, H, W, C, M, R, stride, pad):
    rng = np.random.default_rng(C)
    w = rng.standard_normal((M, R * R * C)).astype(np.float32)
    q, sc, packed = quantize_oracle(random_acts((B, H, W, C), "u8", rng), "u8")
    wq, ws = O.quantize_weights_w8(w)
    y, _ = O.conv2d_w8(q, sc, R, R, stride, pad, 1, wq, ws)
    args = (to_dev(packed), "u8", to_dev(np.array([sc], np.float32)), B, H, W, C, R, R, stride, pad, 1, to_dev(wq),
            to_dev(ws), M)
    return lambda: fgq.fgq_conv2d_w8(*args).cpu().numpy(), y.astype(np.float32)


def _sums_call(G, R):
    rng = np.random.default_rng(G + R)
    B, H, W, C, M = 4, 14, 14, 128, 64
    t, _, codes = make_codes(rng.standard_normal((M, R * R * C)).astype(np.float32), G)
    q, _, packed = quantize_oracle(random_acts((B, H, W, C), "s8", rng), "s8")
    qd, cd = to_dev(packed), to_dev(codes.view(np.int32))

    def call(path=fgq.PATH_TC):
        fgq.fgq_set_path(path)
        return fgq.fgq_conv2d_group_sums(qd, "s8", B, H, W, C, R, R, 1, R // 2, 1, cd, M, G).cpu().numpy()
    return call, call(fgq.PATH_SIMT)


@pytest.mark.parametrize("kernel", ["im2col_dense", "few_channels", "few_channels_s1", "sums_g4_3x3", "sums_g4_1x1",
                                    "sums_g64"])
def test_forced_wait_expiry_of_the_exact_kernels(kernel):
    """The kernels whose outputs are exact integers (times one scale): the dense kernel that converts its
    operands in flight, the few-channel one, and the group sums."""
    call, want = {"im2col_dense": lambda: _w8_call(4, 30, 30, 16, 64, 3, 1, 1),
                  "few_channels": lambda: _w8_call(8, 64, 64, 3, 64, 7, 2, 3),
                  "few_channels_s1": lambda: _w8_call(8, 32, 32, 8, 130, 3, 1, 1),
                  "sums_g4_3x3": lambda: _sums_call(4, 3), "sums_g4_1x1": lambda: _sums_call(4, 1),
                  "sums_g64": lambda: _sums_call(64, 3)}[kernel]()
    assert np.array_equal(call(), want)
    fgq.fgq_debug_set_wait_limit_us(0)
    seen = []
    for _ in range(TRIES):
        out = call()
        seen.append(fgq.fgq_stream_status())
        assert seen[-1] in (fgq.FGQ_OK, fgq.FGQ_ERR_TIMEOUT)
        if seen[-1] == fgq.FGQ_ERR_TIMEOUT:
            break
        assert np.array_equal(out, want)
    assert seen[-1] == fgq.FGQ_ERR_TIMEOUT, f"no wait of {kernel} ran out in {TRIES} calls"
    fgq.fgq_debug_set_wait_limit_us(-1)
    for _ in range(2):
        assert np.array_equal(call(), want)
        assert fgq.fgq_stream_status() == fgq.FGQ_OK
