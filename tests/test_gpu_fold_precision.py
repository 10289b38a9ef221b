"""What the folded tensor-core kernel keeps of a group sum and of its alpha, against the oracle: groups
that a tap boundary cuts, groups whose large halves cancel, rows whose small alphas alone contribute."""
import numpy as np
import pytest

import oracle as O
from paper_1705_01462_gb300 import fgq
from _gpu import check_within, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _clean_status():
    fgq.fgq_set_path(fgq.PATH_AUTO)
    yield
    fgq.fgq_set_path(fgq.PATH_AUTO)
    assert fgq.fgq_stream_status() == fgq.FGQ_OK


def _conv(q, act, t, al, G, R, S, stride=1, pad=0, groups=1, path=fgq.PATH_AUTO):
    B, H, W, C = q.shape
    fgq.fgq_set_path(path)
    got = fgq.fgq_conv2d(to_dev(O.pack_act(q, {"u8": O.U8, "s8": O.S8}[act])), act,
                         to_dev(np.array([1.0], np.float32)), B, H, W, C, R, S, stride, pad, groups,
                         to_dev(O.pack_codes(t).view(np.int32)), to_dev(al), t.shape[0], G).cpu().numpy()
    fgq.fgq_set_path(fgq.PATH_AUTO)
    return got


# channels, G, taps: where the K-tiles of a tap end inside groups
STRADDLE = [(72, 32, 3), (68, 16, 3), (200, 32, 3), (200, 64, 3), (130, 4, 3), (65, 4, 3), (30, 8, 5), (17, 32, 5), (132, 64, 3),
            (144, 64, 3), (48, 32, 5), (100, 64, 4)]


@pytest.mark.parametrize("C,G,R", STRADDLE)
def test_fold_groups_cut_by_taps(C, G, R):
    """Groups with codes +1 on one half and -1 on the other: over images of one value each sums to zero,
    and whatever its halves leave behind counts against the one group of a filter that does not, with
    a single code and a smaller alpha.  Filters without that group give exactly zero."""
    rng = np.random.default_rng(C + G)
    B, H, W, M = 6, R + 11, R + 23, 96
    K = R * R * C
    ng = -(-K // G)
    al = rng.uniform(5.0, 10.0, (M, ng)).astype(np.float32)
    tg = np.tile(np.concatenate([np.ones(G // 2), -np.ones(G // 2)]).astype(np.int8), (M, ng, 1))
    if K % G:
        tg[:, -1] = 0  # the ragged last group would not cancel
    for m in range(M - 8):
        g = m * (K // G) // (M - 8)
        tg[m, g] = 0
        tg[m, g, rng.integers(G)] = 1
        al[m, g] = rng.uniform(1.0, 2.0)
    t = tg.reshape(M, -1)
    q = rng.integers(0, 256, (B, H, W, C)).astype(np.int32)
    q[:B - 1] = np.array([255, 1, 97, 200, 254], np.int32)[:, None, None, None]
    y, ym = O.conv2d(q, np.float32(1.0), R, R, 1, 0, 1, t, al, G)
    got = _conv(q, "u8", t, al, G, R, R)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got, y, ym, f"groups cut by taps C={C} G={G}")
    assert np.all(got[ym == 0] == 0)


@pytest.mark.parametrize("G", [8, 16, 32, 64])
def test_fold_sums_inside_groups(G):
    """What an accumulator holds between the two halves of a group that cancels: at G = 64 32 products of
    255 with the largest alpha, 2^24 on the grid of 2^11.  A filter's output is one group's sum of 37
    with alphas whose grid value is odd, so that a unit lost there is 1.3e-5 of it; filters of
    cancelling groups alone, with alphas of many magnitudes, give exactly zero."""
    rng = np.random.default_rng(G)
    P, K, M = 140, 1184, 96
    ng = -(-K // G)
    al = np.full((M, ng), 1.999, np.float32)
    al[M // 2:] = rng.uniform(0.02, 2.0, (M // 2, ng))
    tg = np.tile(np.concatenate([np.ones(G // 2), -np.ones(G // 2)]).astype(np.int8), (M, ng, 1))
    tg[:, ::4] = 0  # every fourth group holds one code in one filter, and nothing in the others
    if K % G:
        tg[:, -1] = 0
    q = np.full((P, K), 255, np.int32)
    q[1::2] = rng.integers(200, 256, (P // 2, 1))
    q[:, ::4 * G] = 37
    for m in range(0, M, 2):
        tg[m, 4 * (m // 2 % ((K // G + 3) // 4)), 0] = 1
    t = tg.reshape(M, -1)
    y, ym = O.gemm(q, np.float32(1.0), t, al, G)
    got = _conv(q.reshape(P, 1, 1, K), "u8", t, al, G, 1, 1).reshape(P, M)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    check_within(got, y, ym, f"sums inside groups G={G}")
    assert np.all(got[ym == 0] == 0)


@pytest.mark.parametrize("ratio", [1, 2, 3, 5, 8, 45, 700, 2 ** 20])
@pytest.mark.parametrize("G,K", [(4, 2304), (4, 256), (8, 2304), (16, 2304), (32, 2304), (32, 512), (32, 1152), (8, 9216), (64, 2336)])
def test_fold_small_alphas_alone(G, K, ratio):
    """One group in 256 elements has the largest alpha, `ratio` times the others', and meets channels that
    are zero: the output's error is that of the small alphas' parts, no larger than the error of fp32
    alphas on exact group sums (the dp4a kernel)."""
    rng = np.random.default_rng(1000 * G + K + ratio)
    P, M = 200, 128
    ng = -(-K // G)
    al = rng.uniform(1.0, 2.0, (M, ng)).astype(np.float32)
    t = rng.integers(-1, 2, (M, ng * G)).astype(np.int8)
    t[:, K:] = 0
    q = rng.integers(0, 256, (P, K)).astype(np.int32)
    for k in range(0, K, 256):
        al[:, k // G] *= np.float32(ratio)
        q[:, k:k + G] = 0
    y, _ = O.gemm(q, np.float32(1.0), t, al, G)
    q = q.reshape(P, 1, 1, K)
    got = _conv(q, "u8", t, al, G, 1, 1, path=fgq.PATH_TC if G == 4 and K % 64 == 0 else fgq.PATH_AUTO).reshape(P, M)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    simt = _conv(q, "u8", t, al, G, 1, 1, path=fgq.PATH_SIMT).reshape(P, M)
    rms = np.sqrt(np.mean(y ** 2))
    err, ref = (np.sqrt(np.mean((v.astype(np.float64) - y) ** 2)) / rms for v in (got, simt))
    # both are sums of roundings; 1.1 and 0.05 ulp for the spread of two draws of them
    assert err <= 1.1 * ref + 0.05 * 2.0 ** -24, (err, ref)


@pytest.mark.parametrize("G", [4, 8, 16])
@pytest.mark.parametrize("frac", [0, 3, 6])
def test_fold_step_sums_are_exact(G, frac):
    """Groups inside one MMA step: the products of a group that cancels, as large as they get, leave nothing
    of themselves and take nothing from an alpha on the finest grid of the parts beside them."""
    rng = np.random.default_rng(10 * G + frac)
    P, K, M = 130, 1024, 128
    ng = K // G
    t = np.zeros((M, ng, G), np.int8)
    for r in t.reshape(-1, G):
        i = rng.permutation(G)
        r[i[:G // 2]], r[i[G // 2:]] = 1, -1
    al = np.full((M, ng), 2047 / 1024, np.float32)
    al[:, ::3] = 1999 / 1024
    for m in range(M):  # one group of one code: al is an odd multiple of 2^-frac / 1024, 10 bits long
        g = m * ng // M
        t[m, g] = 0
        t[m, g, rng.integers(G)] = rng.choice([-1, 1])
        al[m, g] = (rng.integers(2 ** 9, 2 ** 10) | 1) * 2.0 ** -frac / 1024
    t = t.reshape(M, K)
    q = np.full((P, K), 255, np.int32)
    q[1::2] = rng.integers(1, 256, (P // 2, 1))
    y, _ = O.gemm(q, np.float32(1.0), t, al, G)
    got = _conv(q.reshape(P, 1, 1, K), "u8", t, al, G, 1, 1).reshape(P, M)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    assert np.array_equal(got, y.astype(np.float32))


@pytest.mark.parametrize("G,K", [(4, 512), (8, 2304), (16, 512), (32, 2304), (64, 2336)])
def test_fold_nonfinite_alphas(G, K):
    """A caller's infinite and NaN alphas, on codes and on groups without any: the outputs that they reach
    are the dp4a kernel's (alpha s in fp32: infinite, or NaN where s is 0), the other filters' are as
    ever."""
    rng = np.random.default_rng(G)
    P, M = 96, 128
    ng = -(-K // G)
    al = rng.uniform(0.001, 2.0, (M, ng)).astype(np.float32)
    t = rng.integers(-1, 2, (M, ng, G)).astype(np.int8)
    t[:, -1] = 0  # (ragged where K % G)
    q = rng.integers(0, 256, (P, K)).astype(np.int32)
    q[::3, :256] = 0
    al[0, 0], al[1, 1], al[2, ng // 2] = np.inf, -np.inf, np.nan
    al[64, 0] = al[65, 0] = np.inf
    al[66, 1] = np.nan
    t[64, 0] = t[66, 1] = 0  # no codes
    t = t.reshape(M, -1)
    clean = np.ones(M, bool)
    clean[[0, 1, 2, 64, 65, 66]] = False
    y, ym = O.gemm(q, np.float32(1.0), t[clean], al[clean], G)
    q = q.reshape(P, 1, 1, K)
    got = _conv(q, "u8", t, al, G, 1, 1).reshape(P, M)
    assert fgq.fgq_last_path() == fgq.PATH_TC
    simt = _conv(q, "u8", t, al, G, 1, 1, path=fgq.PATH_SIMT).reshape(P, M)
    assert np.isnan(simt[:, [2, 64, 66]]).all() and np.isinf(simt).any()
    assert np.array_equal(got[:, ~clean], simt[:, ~clean], equal_nan=True)
    check_within(got[:, clean], y, ym, f"non-finite alphas beside, G={G}")
