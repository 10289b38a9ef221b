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
