"""GPU parity for the vertex orders (Sec. 4, Sec. 5): permutation and
reordered records bit-exact against the oracle; rendering is invariant under
every order."""
import numpy as np
import pytest
import torch

import constructed as cs
from gpu_helpers import Renderer, reorder_gpu, U64_EMPTY
from paper_2104_07526_gb300 import pcr, scenes

pytestmark = pytest.mark.gpu

MODES = (pcr.PCR_ORDER_MORTON, pcr.PCR_ORDER_MORTON_SHUFFLE128, pcr.PCR_ORDER_SHUFFLE, pcr.PCR_ORDER_MORTON63,
         pcr.PCR_ORDER_MORTON63_SHUFFLE128)


@pytest.fixture(scope="module")
def r():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    rend = Renderer()
    yield rend
    rend.close()


@pytest.mark.parametrize("n", [0, 1, 2, 127, 128, 129, 1000, 5119, 5120, 5121, 6143, 6144, 6145, 8191, 8192, 8193,
                               10241, 12289, 100_003])
def test_reorder_matches_oracle(r, oracle, n):
    cloud = scenes.random_cloud(n, seed=n + 7).numpy() if n else np.zeros((0, 4), np.int32)
    for mode in MODES:
        seed = 0xC0FFEE + n
        expect = oracle.reorder(cloud, seed, mode)
        dev = torch.from_numpy(cloud.copy()).cuda() if n else torch.zeros((0, 4), dtype=torch.int32, device="cuda")
        perm = reorder_gpu(r.h, dev, seed, mode)
        assert np.array_equal(perm, expect), (n, mode)
        assert np.array_equal(dev.cpu().numpy(), oracle.gather(cloud, expect) if n else cloud), (n, mode)


@pytest.mark.parametrize("n", [300_017, 5_000_017])
def test_reorder_scene_with_duplicates(r, oracle, n):
    """Scanline scene (many equal Morton codes: stability decides) at sizes
    spanning many sort tiles with a ragged tail; 5M points is 814 tiles, more
    than the scatter kernel keeps resident at once (4 per SM), so tiles run
    in several waves."""
    cloud = scenes.scan(n, seed=1).numpy()
    for mode in MODES:
        expect = oracle.reorder(cloud, 42, mode)
        dev = torch.from_numpy(cloud.copy()).cuda()
        perm = reorder_gpu(r.h, dev, 42, mode)
        assert np.array_equal(perm, expect), mode
    assert pcr.pcr_last_device_error(r.h) == 0


@pytest.mark.parametrize("n", [129, 8193, 100_003])
def test_reorder_without_permutation(r, oracle, n):
    """Without a permutation output the last sort pass takes its other
    record-moving loops; the records must be the same."""
    cloud = scenes.random_cloud(n, seed=n + 3).numpy()
    for mode in MODES:
        expect = oracle.gather(cloud, oracle.reorder(cloud, 99, mode))
        dev = torch.from_numpy(cloud.copy()).cuda()
        ws = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device="cuda")
        pcr.pcr_reorder_morton_shuffle128(r.h, dev, n, 99, mode, ws, None)
        torch.cuda.synchronize()
        assert np.array_equal(dev.cpu().numpy(), expect), (n, mode)


def test_reorder_degenerate_and_nonfinite(r, oracle):
    same = cs.pack(np.tile([[1.0, 2.0, 3.0]], (1000, 1)), np.arange(1000, dtype=np.uint32))
    odd = scenes.random_cloud(3000, seed=4).numpy()
    odd[5, 0] = np.float32(np.nan).view(np.int32)
    odd[9, 1] = np.float32(-0.0).view(np.int32)
    odd[11, 2] = np.float32(np.nan).view(np.int32)
    for cloud in (same, odd):
        for mode in MODES:
            expect = oracle.reorder(cloud, 5, mode)
            dev = torch.from_numpy(cloud.copy()).cuda()
            assert np.array_equal(reorder_gpu(r.h, dev, 5, mode), expect), mode


def test_render_invariant_under_orders(r, oracle):
    """Sec. 4: reordering changes speed, not the image.  Depth halves match
    exactly.  Where several points share the minimum depth (the ground plane
    of this scene is at one depth) the index tie-break may pick another of
    them, so each winner is checked to be a minimum-depth point of its
    pixel; the reordered buffer also matches the oracle bit for bit."""
    cloud = scenes.sphere_plane(120_000, seed=2).numpy()
    view = scenes.sphere_plane_views()[0]
    W, H = view.width, view.height
    base = oracle.render_basic(cloud, view.matrix, W, H)
    hit = np.nonzero(base != U64_EMPTY)[0]
    p = np.ascontiguousarray(cloud[:, :3]).view(np.float32)
    for mode in MODES:
        dev = torch.from_numpy(cloud.copy()).cuda()
        perm = reorder_gpu(r.h, dev, 9, mode).astype(np.int64)
        pcr.pcr_upload_points(r.h, dev, dev.shape[0])
        r.points = dev
        r.view(view.matrix, W, H)
        got = r.render_basic(pcr.PCR_VARIANT_DEDUP_EARLYZ)
        moved = oracle.gather(cloud, perm.astype(np.uint32))
        assert np.array_equal(got, oracle.render_basic(moved, view.matrix, W, H)), mode
        assert np.array_equal(got >> np.uint64(32), base >> np.uint64(32)), mode
        for px in hit[:: max(1, hit.size // 3000)]:
            old = perm[int(got[px]) & 0xFFFFFFFF]
            pr = oracle.project(view.matrix, W, H, *p[old])
            assert pr is not None and pr[0] == px
            assert int(np.float32(pr[1]).view(np.uint32)) == int(base[px]) >> 32
        img = r.resolve(pcr.PCR_RESOLVE_BASIC, 0)
        assert np.array_equal(img, oracle.resolve_basic(got, moved, 0)), mode


def test_reorder_errors(r):
    n = 1000
    dev = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
    need = pcr.pcr_reorder_workspace_size(n)
    small = torch.empty(need - 256, dtype=torch.uint8, device="cuda")
    with pytest.raises(pcr.PcrError) as e:
        pcr.pcr_reorder_morton_shuffle128(r.h, dev, n, 0, pcr.PCR_ORDER_MORTON, small)
    assert e.value.status == pcr.PCR_ERR_WORKSPACE
    with pytest.raises(pcr.PcrError) as e:
        pcr.pcr_reorder_morton_shuffle128(r.h, dev, n, 0, pcr.PCR_ORDER_MORTON, None)
    assert e.value.status == pcr.PCR_ERR_WORKSPACE
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    with pytest.raises(pcr.PcrError) as e:
        pcr.pcr_reorder_morton_shuffle128(r.h, dev, n, 0, 5, ws)
    assert e.value.status == pcr.PCR_ERR_ARG
    with pytest.raises(pcr.PcrError) as e:
        pcr.pcr_reorder_morton_shuffle128(r.h, dev.data_ptr() + 4, n, 0, 0, ws)
    assert e.value.status == pcr.PCR_ERR_ARG


@pytest.mark.parametrize("n", [1983, 1984, 1985, 4095, 4096, 4097, 20_011, 2048 * 1984, 2048 * 1984 + 1])
def test_shuffle_at_its_pass_limits(r, oracle, n):
    """The random order's buckets hold 1984 records on average: one bucket and
    two, tiles of 4096 and one more, the most records one partition pass
    splits and the first size that takes two."""
    cloud = torch.arange(4 * n, dtype=torch.int32).reshape(n, 4)
    expect = oracle.reorder(cloud.numpy(), 11 * n, pcr.PCR_ORDER_SHUFFLE).astype(np.int64)
    dev = cloud.cuda()
    assert np.array_equal(reorder_gpu(r.h, dev, 11 * n, pcr.PCR_ORDER_SHUFFLE), expect)
    assert torch.equal(dev.cpu(), cloud[torch.from_numpy(expect)])
    ws = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device="cuda")
    dev = cloud.cuda()
    pcr.pcr_reorder_morton_shuffle128(r.h, dev, n, 11 * n, pcr.PCR_ORDER_SHUFFLE, ws)
    assert torch.equal(dev.cpu(), cloud[torch.from_numpy(expect)])


@pytest.mark.parametrize("n", [1984, 2048 * 1984])
def test_benchmark_counts_the_shuffles_passes(r, n):
    """The benchmark's bytes of a shuffle change where its launches do."""
    import bench

    def launches(n):
        points = torch.zeros((n, 4), dtype=torch.int32, device="cuda")
        ws = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device="cuda")
        before = pcr.pcr_launches()
        pcr.pcr_reorder_morton_shuffle128(r.h, points, n, 0, pcr.PCR_ORDER_SHUFFLE, ws)
        return pcr.pcr_launches() - before

    assert launches(n) < launches(n + 1)
    assert bench.shuffle_bytes_per_point(n) < bench.shuffle_bytes_per_point(n + 1)


@pytest.mark.parametrize("n", [255, 1023, 1024, 1025, 2049, 128 * 1024, 128 * 1024 + 1, 256 * 3072, 256 * 3072 + 1,
                               384 * 6144, 384 * 6144 + 1])
def test_reorder_at_the_limits_of_small_sorts(r, oracle, n):
    """One tile and two, the last size of each small tile size and the first of
    the next, the first that takes the three-kernel passes (256 * 3072 + 1),
    and whole tiles of those passes and one point more; half of the points lie
    on few cells."""
    rng = np.random.default_rng(n)
    cloud = scenes.random_cloud(n, seed=n).numpy()
    dense = rng.random(n) < 0.5
    cloud[dense, :3] = rng.uniform(-0.01, 0.01, (int(dense.sum()), 3)).astype(np.float32).view(np.int32)
    for mode in (pcr.PCR_ORDER_MORTON, pcr.PCR_ORDER_MORTON63, pcr.PCR_ORDER_MORTON_SHUFFLE128):
        expect = oracle.reorder(cloud, 5 + n, mode)
        dev = torch.from_numpy(cloud.copy()).cuda()
        assert np.array_equal(reorder_gpu(r.h, dev, 5 + n, mode), expect), mode
        assert np.array_equal(dev.cpu().numpy(), oracle.gather(cloud, expect)), mode


def test_small_reorder_of_points_without_bounds(r, oracle):
    """Every coordinate NaN, one axis NaN, infinities: the bounds' joins."""
    base = scenes.random_cloud(3001, seed=1).numpy()
    for spoil in ("all", "axis", "inf"):
        cloud = base.copy()
        if spoil == "all":
            cloud[:, :3] = np.float32(np.nan).view(np.int32)
        elif spoil == "axis":
            cloud[:, 1] = np.float32(np.nan).view(np.int32)
        else:
            cloud[::7, 0] = np.float32(np.inf).view(np.int32)
            cloud[3::7, 2] = np.float32(-np.inf).view(np.int32)
        for mode in MODES:
            expect = oracle.reorder(cloud, 3, mode)
            dev = torch.from_numpy(cloud.copy()).cuda()
            assert np.array_equal(reorder_gpu(r.h, dev, 3, mode), expect), (spoil, mode)


@pytest.mark.parametrize("spoil", ["all", "axis", "inf", "one"])
def test_large_reorder_of_points_without_bounds(r, oracle, spoil):
    """As above with the bounds that blocks join by atomics; "one": a single
    point has an extreme, in the last record."""
    n = 384 * 6144 + 261
    cloud = scenes.random_cloud(n, seed=2).numpy()
    if spoil == "all":
        cloud[:, :3] = np.float32(np.nan).view(np.int32)
    elif spoil == "axis":
        cloud[:, 1] = np.float32(np.nan).view(np.int32)
    elif spoil == "inf":
        cloud[::7, 0] = np.float32(np.inf).view(np.int32)
        cloud[3::7, 2] = np.float32(-np.inf).view(np.int32)
    else:
        cloud[-1, :3] = np.array([900.0, -700.0, 800.0], np.float32).view(np.int32)
    for mode in (pcr.PCR_ORDER_MORTON, pcr.PCR_ORDER_MORTON63):
        expect = oracle.reorder(cloud, 3, mode)
        dev = torch.from_numpy(cloud.copy()).cuda()
        assert np.array_equal(reorder_gpu(r.h, dev, 3, mode), expect), mode
