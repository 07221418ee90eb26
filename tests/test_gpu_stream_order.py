"""Launches overlap the end of the kernel before them in the stream.  Back to
back, with nothing waiting between, calls that read what the call (or the
PyTorch kernel) just before them wrote give the results they give alone."""
import numpy as np
import pytest
import torch

from gpu_helpers import Renderer
from paper_2104_07526_gb300 import pcr, scenes

pytestmark = pytest.mark.gpu

W, H = 320, 200


def _pass(r, points, workspace, source, seed, order, matrix, wait):
    """Points written by PyTorch, reordered, rendered into buffers that
    PyTorch cleared (so no kernel of the library stands between), resolved."""
    def step():
        if wait:
            torch.cuda.synchronize()
    fb = r.fb
    points.copy_(source)
    step()
    pcr.pcr_reorder_morton_shuffle128(r.h, points, points.shape[0], seed, order, workspace)
    step()
    fb["keys"].fill_(-1)
    step()
    pcr.pcr_set_matrix(r.h, matrix)
    pcr.pcr_render_basic(r.h, pcr.PCR_VARIANT_DEDUP_EARLYZ, False)
    step()
    pcr.pcr_resolve(r.h, pcr.PCR_RESOLVE_BASIC, fb["image"], 7)
    out = [points.clone(), fb["keys"].clone(), fb["image"].clone()]
    step()
    pcr.pcr_reorder_morton_shuffle128(r.h, points, points.shape[0], seed + 1, pcr.PCR_ORDER_SHUFFLE, workspace)
    step()
    pcr.pcr_render_basic(r.h, pcr.PCR_VARIANT_EARLYZ, True)
    step()
    pcr.pcr_render_hq(r.h, 1.01, pcr.PCR_VARIANT_DEDUP_EARLYZ, True)
    step()
    pcr.pcr_resolve(r.h, pcr.PCR_RESOLVE_HQ, fb["image"], 7)
    return out + [fb[k].clone() for k in ("keys", "hq_depth", "hq_rg", "hq_ba", "image")]


@pytest.mark.parametrize("n", (3_001, 100_003, 3_000_017))
@pytest.mark.parametrize("order", (pcr.PCR_ORDER_MORTON, pcr.PCR_ORDER_MORTON_SHUFFLE128, pcr.PCR_ORDER_SHUFFLE,
                                   pcr.PCR_ORDER_MORTON63))
def test_back_to_back_calls_equal_calls_alone(n, order):
    r = Renderer()
    sources = [scenes.random_cloud(n, seed=s, device="cuda") for s in range(3)]
    points = torch.empty_like(sources[0])
    workspace = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device="cuda")
    r.upload(points)
    points = r.points
    matrices = [scenes.camera((2.0 + k, 1.0 - k, 2.5), (0, 0, 0), (0, 0, 1), W, H) for k in range(3)]
    r.view(matrices[0], W, H)
    alone = [_pass(r, points, workspace, sources[k], k, order, matrices[k], True) for k in range(3)]
    got = [_pass(r, points, workspace, sources[k % 3], k % 3, order, matrices[k % 3], False) for k in range(9)]
    torch.cuda.synchronize()
    for k, outs in enumerate(got):
        for i, (a, b) in enumerate(zip(alone[k % 3], outs)):
            assert torch.equal(a, b), (k, i)
    r.close()


@pytest.mark.parametrize("size", ((2048, 2047), (2048, 2048), (1024, 1023), (1024, 1024)))
@pytest.mark.parametrize("n", (5_003, 2 * 1024 * 1024 - 1, 2 * 1024 * 1024))
def test_sums_cleared_beside_the_depth_pass(oracle, size, n):
    """High-quality frames on both sides of the limits from which the sums are
    cleared beside the depth pass, back to back with other cameras and as a
    replayed graph: the oracle's buffers and images."""
    r = Renderer()
    cloud = scenes.random_cloud(n, seed=n % 97).numpy()
    r.upload(cloud)
    matrices = [scenes.camera((1.5 + k, -2.0, 1.0), (0, 0, 0), (0, 0, 1), *size) for k in range(2)]
    expect = [oracle.render_hq(cloud, m, *size, 1.01) for m in matrices]
    images = [oracle.resolve_hq(e[1], e[2], 5) for e in expect]
    r.view(matrices[0], *size)
    fb, out = r.fb, []
    for k in (0, 1, 0, 1):
        pcr.pcr_set_matrix(r.h, matrices[k])
        pcr.pcr_render_hq(r.h, 1.01, pcr.PCR_VARIANT_DEDUP_EARLYZ, True)
        pcr.pcr_resolve(r.h, pcr.PCR_RESOLVE_HQ, fb["image"], 5)
        out.append([fb[b].clone() for b in ("hq_depth", "hq_rg", "hq_ba", "image")])
        pcr.pcr_render_hq1r(r.h, 1.01, pcr.PCR_VARIANT_EARLYZ, True)
        pcr.pcr_resolve(r.h, pcr.PCR_RESOLVE_HQ1R, fb["image"], 5)
        out[-1].append(fb["image"].clone())
    pcr.pcr_capture_begin(r.h)
    pcr.pcr_render_hq(r.h, 1.01, pcr.PCR_VARIANT_DEDUP_EARLYZ, True)
    pcr.pcr_resolve(r.h, pcr.PCR_RESOLVE_HQ, fb["image"], 5)
    graph = pcr.pcr_capture_end(r.h)
    for _ in range(3):
        pcr.pcr_graph_launch(r.h, graph)
    out.append([fb[b].clone() for b in ("hq_depth", "hq_rg", "hq_ba", "image")])
    torch.cuda.synchronize()
    pcr.pcr_graph_destroy(graph)
    for k, got in zip((0, 1, 0, 1, 1), out):
        for a, b in zip(got, (*expect[k], images[k], images[k])):
            assert np.array_equal(a.cpu().numpy().view(b.dtype), b), k
    r.close()
