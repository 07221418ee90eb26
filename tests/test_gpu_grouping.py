"""Where the warp deduplication and the colour grouping are switched on and
off: rows of 32 points with a chosen number of equal-pixel runs on both sides
of the limits, followed by rows of one pixel and of distinct pixels, against
the oracle."""
import numpy as np
import pytest

from gpu_helpers import Renderer
from paper_2104_07526_gb300 import pcr

pytestmark = pytest.mark.gpu

W, H = 61, 47


@pytest.fixture(scope="module")
def r():
    rend = Renderer()
    yield rend
    rend.close()


def _cloud(pixels: np.ndarray, rng) -> np.ndarray:
    """Points on the centres of the given pixels (-1: culled) at random depths
    with ties, for a camera whose w is the z coordinate."""
    n = pixels.size
    z = rng.choice(np.float32([1.0, 1.5, 2.0, 2.015625]), n).astype(np.float32)
    x = (((pixels % W) + 0.5) / W * 2 - 1) * z
    y = (((pixels // W) + 0.5) / H * 2 - 1) * z
    cloud = np.empty((n, 4), dtype=np.int32)
    cloud[:, 0], cloud[:, 1] = x.astype(np.float32).view(np.int32), y.astype(np.float32).view(np.int32)
    cloud[:, 2] = np.where(pixels < 0, np.float32(-1), z).astype(np.float32).view(np.int32)
    cloud[:, 3] = rng.integers(-(1 << 31), 1 << 31, n)
    return cloud


def _runs(rng, lanes: int, runs: int) -> np.ndarray:
    """`lanes` neighbouring points on pixels that change runs - 1 times."""
    cuts = np.zeros(lanes, dtype=np.int64)
    cuts[rng.choice(np.arange(1, lanes), runs - 1, replace=False)] = 1
    return rng.choice(W * H, runs, replace=False)[np.cumsum(cuts)]


def _check(r, oracle, cloud):
    m = np.eye(4, dtype=np.float32)
    m[3] = (0, 0, 1, 0)
    r.upload(cloud)
    r.view(m, W, H)
    keys = oracle.render_basic(cloud, m, W, H)
    rgb = oracle.render_rgb(cloud, m, W, H)
    for v in pcr.EXACT_VARIANTS:
        assert np.array_equal(r.render_basic(v), keys), pcr.VARIANT_NAMES[v]
        assert np.array_equal(r.render_rgb(v), rgb), pcr.VARIANT_NAMES[v]
    hq = oracle.render_hq(cloud, m, W, H, 1.01)
    sums = oracle.hq_channel_sums(cloud, m, W, H, hq[0], 1.01)
    for v in (pcr.PCR_VARIANT_EARLYZ, pcr.PCR_VARIANT_DEDUP, pcr.PCR_VARIANT_DEDUP_EARLYZ):
        for got, want in zip(r.render_hq(v), hq):
            assert np.array_equal(got, want), pcr.VARIANT_NAMES[v]
        for got, want in zip(r.render_hq1r_sums(v)[1:], sums):
            assert np.array_equal(got, want), pcr.VARIANT_NAMES[v]


@pytest.mark.parametrize("visible", (16, 17, 32))
@pytest.mark.parametrize("runs", (1, 15, 16, 17, 32))
def test_rows_on_both_sides_of_the_run_limit(r, oracle, runs, visible):
    rng = np.random.default_rng(100 * runs + visible)
    rows = []
    for chunk in range(5):
        first = np.full(32, -1)
        first[32 - visible:] = _runs(rng, visible, min(runs, visible))
        rows += [first, np.full(32, rng.integers(W * H)), _runs(rng, 32, 32), _runs(rng, 32, 5)]
    pixels = np.concatenate(rows)
    _check(r, oracle, _cloud(pixels, rng))
    _check(r, oracle, _cloud(pixels[: pixels.size - 45], rng))  # a ragged last chunk


@pytest.mark.parametrize("joins", (0, 7, 8, 9, 32))
def test_chunks_on_both_sides_of_the_join_limit(r, oracle, joins):
    """Lane l takes points 4l .. 4l + 3 of a chunk: `joins` lanes have their
    first two points on one pixel, the lanes' first points fall on few pixels."""
    rng = np.random.default_rng(7 + joins)
    chunks = []
    for _ in range(5):
        p = rng.choice(W * H, (32, 4))
        p[:, 0] = rng.choice(W * H, 3)[rng.integers(0, 3, 32)]
        p[:, 1] = p[:, 0] + 1
        mine = rng.choice(32, joins, replace=False)
        p[mine, 1] = p[mine, 0]
        chunks.append(np.minimum(p, W * H - 1).reshape(-1))
    pixels = np.concatenate(chunks)
    _check(r, oracle, _cloud(pixels, rng))
    _check(r, oracle, _cloud(pixels[: pixels.size - 3], rng))
