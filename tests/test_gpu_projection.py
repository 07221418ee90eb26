"""The projection's screen division against IEEE division, on the GPU.

Every geometry kernel divides both clip coordinates of a point by w through
one reciprocal, y = RN(1/w) (one Newton step on the hardware estimate), and
corrects each quotient after Markstein (1990), for w in [2^-40, 2^40).  The
render parity tests show whole frames equal to the oracle's; these tests pin
the arithmetic itself through pcr_check_division:

- the reciprocal equals the IEEE one for every float in the window;
- the quotient equals IEEE c / w on dense grids of significands and on
  random bit patterns (all exponents, zeros, subnormals, infinities, NaNs);
- the screen coordinate equals the one from the IEEE quotient, or both are
  culled, for every pair.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2104_07526_gb300 import pcr

pytestmark = pytest.mark.gpu

WINDOW_LO = 0x2B800000  # bits of 2^-40
WINDOW_HI = 0x53800000  # bits of 2^40
ONE = 0x3F800000


@pytest.fixture(scope="module")
def ctx():
    from gpu_helpers import ensure_built
    ensure_built()
    c = pcr.Context(0, stream=torch.cuda.current_stream())
    yield c.handle
    c.close()


def test_reciprocal_exact_over_the_whole_window(ctx):
    got = pcr.pcr_check_division(ctx, WINDOW_LO, WINDOW_HI - WINDOW_LO)
    assert got["reciprocal_mismatches"] == 0
    # the bit patterns just outside the window are skipped, not checked
    edge = pcr.pcr_check_division(ctx, WINDOW_LO - 1000, 2000)
    assert edge["reciprocal_mismatches"] == 0


def test_quotient_on_a_grid_of_significands(ctx):
    """w: 8 runs of 2^15 consecutive significands spread over [1, 2); c: every
    8th significand in [1, 2).  2^38 pairs; quotients in (0.5, 2) span both
    binades next to 1."""
    for k in range(8):
        got = pcr.pcr_check_division(ctx, ONE + k * (1 << 20), 1 << 15, c_first=ONE, c_count=1 << 20, c_step=8,
                                     size=1920.0)
        assert got["pairs"] == (1 << 15) * (1 << 20)
        assert got["quotient_pairs"] == got["pairs"]
        assert got["quotient_mismatches"] == 0
        assert got["screen_mismatches"] == 0


def test_quotient_on_random_and_special_numerators(ctx):
    rng = np.random.default_rng(20260301)
    c = rng.integers(0, 2**32, size=1 << 20, dtype=np.uint64).astype(np.uint32)
    special = np.array([0x00000000, 0x80000000, 0x00000001, 0x80000001, 0x007FFFFF, 0x00800000, 0x7F7FFFFF,
                        0xFF7FFFFF, 0x7F800000, 0xFF800000, 0x7FC00000, 0xFFC00000, 0x3F800000, 0xBF800000,
                        0x4F000000, 0x30800000, 0x2F800000, 0x2E800000], dtype=np.uint32)
    c[:special.size] = special
    dev = torch.from_numpy(c.view(np.int32)).cuda()
    total = {"quotient_mismatches": 0, "screen_mismatches": 0, "quotient_pairs": 0, "pairs": 0}
    starts = rng.integers(WINDOW_LO, WINDOW_HI - 64, size=24)
    for w0 in list(starts) + [WINDOW_LO, WINDOW_HI - 64, ONE - 32]:
        for size in (1920.0, 1080.0, 7.0):
            got = pcr.pcr_check_division(ctx, int(w0), 64, c_bits=dev, size=size)
            for k in total:
                total[k] += got[k]
    assert total["pairs"] == 27 * 3 * 64 * c.size
    assert total["quotient_pairs"] > total["pairs"] // 4
    assert total["quotient_mismatches"] == 0
    assert total["screen_mismatches"] == 0


def test_check_rejects_bad_arguments(ctx):
    with pytest.raises(pcr.PcrError):
        pcr.pcr_check_division(ctx, ONE, 1, c_first=ONE, c_count=4, c_step=0)
    with pytest.raises(pcr.PcrError):
        pcr.pcr_check_division(ctx, ONE, 1, size=0.0)


SPECIAL_W = np.array([2.0**-41, np.nextafter(np.float32(2.0**-40), np.float32(0)), 2.0**-40, 2.0**40,
                      np.nextafter(np.float32(2.0**40), np.float32(0)), 2.0**41, 1e-42, 0.0, -0.0, -(2.0**-41),
                      -1.0, -(2.0**41), np.inf, -np.inf, np.nan, 3.4e38], dtype=np.float32)


@pytest.mark.parametrize("n", (1, 2, 31, 33, 127, 128, 129, 4099))
@pytest.mark.parametrize("share", (0.02, 0.5, 1.0))
def test_slots_that_leave_the_window_beside_slots_inside(ctx, oracle, n, share):
    """w is the z coordinate: a share of the points have a w outside the
    reciprocal window, zero, infinite or NaN, so lanes mix both kinds.  Key
    frames test the window once per lane, the depth and colour passes once
    per pair of slots."""
    from gpu_helpers import Renderer
    rng = np.random.default_rng(n)
    z = rng.uniform(0.5, 4.0, n).astype(np.float32)
    z = np.where(rng.random(n) < share, rng.choice(SPECIAL_W, n), z).astype(np.float32)
    scale = np.where(np.isfinite(z), np.clip(z, -1e37, 1e37), 1.0)
    xy = (rng.uniform(-1.2, 1.2, (n, 2)) * scale[:, None]).astype(np.float32)
    cloud = np.empty((n, 4), dtype=np.int32)
    cloud[:, :2], cloud[:, 2], cloud[:, 3] = xy.view(np.int32), z.view(np.int32), rng.integers(0, 1 << 31, n)
    m = np.eye(4, dtype=np.float32)
    m[3] = (0, 0, 1, 0)
    W, H = 37, 23
    r = Renderer()
    r.upload(cloud)
    r.view(m, W, H)
    expect = oracle.render_basic(cloud, m, W, H)
    for v in pcr.EXACT_VARIANTS:
        assert np.array_equal(r.render_basic(v), expect), v
    hq = oracle.render_hq(cloud, m, W, H, 1.01)
    for v in (pcr.PCR_VARIANT_ATOMICMIN, pcr.PCR_VARIANT_DEDUP_EARLYZ):
        for a, b in zip(r.render_hq(v), hq):
            assert np.array_equal(a, b), v
    r.close()
