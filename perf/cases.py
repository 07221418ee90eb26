"""The work this library is measured by: frames, vertex orders, batches and
served requests, from the smallest calls to the largest.

A case is a dict of plain values.  `prepare` makes what a program holds before
the call (clouds, buffers, a context, a captured graph, a server), `run` makes
one pass through the public entry points and returns the buffers it wrote.

Every output is a word or a byte with one defined value (depth keys, integer
colour sums, images, permutations, moved records), so all of them are compared
exactly and there is no 64-bit reference to be near to: the float32 projection
in its fixed order of operations decides which pixel a point lands on.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_07526_gb300 import pcr, scenes

DEVICE = "cuda:0"
POINT = scenes.POINT_BYTES
FACTOR = 1.01  # high-quality depth band

ORDERS = {"morton": pcr.PCR_ORDER_MORTON, "morton_shuffle128": pcr.PCR_ORDER_MORTON_SHUFFLE128,
          "shuffle": pcr.PCR_ORDER_SHUFFLE, "morton63": pcr.PCR_ORDER_MORTON63,
          "morton63_shuffle128": pcr.PCR_ORDER_MORTON63_SHUFFLE128}
VARIANTS = {name: v for v, name in pcr.VARIANT_NAMES.items()}


def listed() -> list[dict]:
    return [
        # A thumbnail of a small object: latency and launches only.
        _frame("frame_sphere_20k", "sphere", 20_011, "original", "front", 160, 120, "basic", "dedup+early-z"),
        # The 1M-point object of the first configuration, in the order it was made, with the plain atomic.
        _frame("frame_sphere_1m", "sphere", 1_000_000, "original", "front", 640, 480, "basic", "atomicMin"),
        # A mid-size scene straight from its generator (no preprocessing), early depth test.
        _frame("frame_boxes_50m", "boxes", 50_000_000, "original", "overview", 1920, 1080, "basic", "early-z"),
        # The headline frame: the largest scan in the recommended order and variant.
        _frame("frame_scan_800m", "scan", 800_000_000, "morton_shuffle128", "overview", 1920, 1080, "basic",
               "dedup+early-z"),
        # High-quality viewing of a mid-size scene in the recommended order.
        _frame("hq_boxes_50m", "boxes", 50_000_000, "morton_shuffle128", "mid", 1920, 1080, "hq", "dedup+early-z"),
        # High-quality frame of a small scan on a 4K screen: clears and resolves weigh as much as the points.
        _frame("hq_scan_4m_4k", "scan", 4_000_037, "original", "overview", 3840, 2160, "hq", "dedup+early-z"),
        # Preprocessing of a small upload (an interactive edit, a tile of a larger data set).
        _reorder("reorder_sphere_100k", "sphere", 100_003, "morton_shuffle128", True),
        # Preprocessing of the largest scan into the recommended order.
        _reorder("reorder_scan_800m", "scan", 800_000_000, "morton_shuffle128", False),
        # The random order of a mid-size scene, with its permutation (attributes kept beside the points).
        _reorder("shuffle_boxes_50m", "boxes", 50_000_000, "shuffle", True),
        # The fine (21 levels per axis) Morton order of a scan.
        _reorder("morton63_scan_20m", "scan", 20_000_003, "morton63", False),
        # The batched configuration: 8 clouds of 1M to 200M points x 8 views of 256^2 to 2048^2, basic + HQ,
        # replayed as one graph.
        {"name": "batch_8x8", "kind": "batch", "clouds": 8, "smallest": 1_000_000, "largest": 200_000_000,
         "views": 8, "min_size": 256, "max_size": 2048, "flags": 3, "graph": True},
        # A burst of view requests over resident clouds of the served configuration's sizes and resolutions.
        {"name": "serve_burst_16", "kind": "serve", "clouds": 4, "smallest": 1_000_000, "largest": 60_000_000,
         "requests": 16, "streams": 3},
    ]


def draw(rng) -> dict:
    kind = rng.choices(("frame", "hq", "reorder", "batch", "serve"), (3, 3, 4, 2, 1))[0]
    scene = rng.choice(("sphere", "boxes", "scan"))
    if kind in ("frame", "hq"):
        width = _log_int(rng, 64, 3840)
        height = max(48, min(2160, int(width * rng.uniform(0.4, 1.2))))
        frame = rng.choice(("basic", "basic", "rgb") if kind == "frame" else ("hq", "hq", "hq1r"))
        variants = ("atomicMin", "early-z", "dedup", "dedup+early-z")
        if kind == "frame":
            variants += ("reduce", "reduce+early-z")
        return _frame(None, scene, _log_int(rng, 1_000, 200_000_000), rng.choice(("original", *ORDERS)),
                      rng.choice(CAMERAS[scene]), width, height, frame, rng.choice(variants), rng.random() < 0.3)
    if kind == "reorder":
        return _reorder(None, scene, _log_int(rng, 100, 100_000_000), rng.choice(tuple(ORDERS)), rng.random() < 0.5)
    if kind == "batch":
        smallest = _log_int(rng, 1_000, 1_000_000)
        return {"kind": "batch", "clouds": rng.randint(1, 8), "smallest": smallest,
                "largest": _log_int(rng, smallest, 50_000_000), "views": rng.randint(1, 8), "min_size": 64,
                "max_size": _log_int(rng, 128, 2048), "flags": rng.choice((1, 2, 3, 3)), "graph": rng.random() < 0.5}
    smallest = _log_int(rng, 10_000, 1_000_000)
    return {"kind": "serve", "clouds": rng.randint(1, 6), "smallest": smallest,
            "largest": _log_int(rng, smallest, 40_000_000), "requests": rng.randint(1, 16),
            "streams": rng.randint(1, 3)}


CAMERAS = {"sphere": ("front",), "boxes": ("overview", "mid", "inside"), "scan": ("overview", "closeup")}


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _frame(name, scene, n, order, camera, width, height, frame, variant, graph=False) -> dict:
    case = {"kind": "frame", "scene": scene, "n": n, "order": order, "camera": camera, "width": width,
            "height": height, "frame": frame, "variant": variant, "graph": graph}
    return {"name": name, **case} if name else case


def _reorder(name, scene, n, order, perm) -> dict:
    case = {"kind": "reorder", "scene": scene, "n": n, "order": order, "perm": perm}
    return {"name": name, **case} if name else case


def _sizes(case) -> list[int]:
    """Cloud sizes of a batch or a server, log-spaced."""
    k = case["clouds"]
    ratio = case["largest"] / case["smallest"]
    return [int(round(case["smallest"] * ratio ** (i / max(k - 1, 1)))) for i in range(k)]


def _view_sizes(case) -> list[int]:
    k = case["views"]
    span = case["max_size"] - case["min_size"]
    return [case["min_size"] + span * i // max(k - 1, 1) for i in range(k)]


# ---------------------------------------------------------------------------
# prepare
# ---------------------------------------------------------------------------

def _cloud(scene: str, n: int, seed: int) -> torch.Tensor:
    make = {"sphere": scenes.sphere_plane, "boxes": scenes.boxes, "scan": scenes.scan}[scene]
    return make(n, seed=seed, device=DEVICE)


def _context() -> pcr.Context:
    return pcr.Context(0, stream=torch.cuda.current_stream())


def _reordered(ctx, points: torch.Tensor, order: str, seed: int) -> torch.Tensor:
    n = points.shape[0]
    if order != "original" and n > 0:
        ws = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device=DEVICE)
        pcr.pcr_reorder_morton_shuffle128(ctx.handle, points, n, seed, ORDERS[order], ws)
    return points


def _matrix(case, seed: int) -> np.ndarray:
    views = {"sphere": lambda: scenes.sphere_plane_views(), "boxes": lambda: scenes.boxes_views(seed),
             "scan": lambda: scenes.scan_views(case["n"], seed)}[case["scene"]]()
    view = next(v for v in views if v.name == case["camera"])
    return _aspect(view.matrix, view.width, view.height, case["width"], case["height"])


def _aspect(matrix: np.ndarray, width: int, height: int, new_width: int, new_height: int) -> np.ndarray:
    """A camera's matrix for a viewport of another shape (the field of view's height stays)."""
    m = matrix.copy()
    m[0] *= np.float32((width / height) / (new_width / new_height))
    return m


class _Graph:
    """A captured frame or batch, destroyed with its state."""

    def __init__(self, executable: int):
        self.executable = executable

    def __del__(self):
        pcr.pcr_graph_destroy(self.executable)


class _Server:
    """A server handle, destroyed with its state."""

    def __init__(self, handle: int):
        self.handle = handle

    def __del__(self):
        pcr.pcr_server_destroy(self.handle)


def prepare(case: dict, seed: int) -> dict:
    return {"frame": _prepare_frame, "reorder": _prepare_reorder, "batch": _prepare_batch,
            "serve": _prepare_serve}[case["kind"]](case, seed)


def _prepare_frame(case, seed):
    ctx = _context()
    h = ctx.handle
    points = _reordered(ctx, _cloud(case["scene"], case["n"], seed), case["order"], seed)
    fb = pcr.alloc_framebuffer(case["width"], case["height"], DEVICE)
    pcr.pcr_upload_points(h, points, case["n"])
    pcr.pcr_set_matrix(h, _matrix(case, seed))
    pcr.pcr_set_viewport(h, case["width"], case["height"])
    pcr.pcr_set_framebuffer(h, fb["keys"], fb["hq_depth"], fb["hq_rg"], fb["hq_ba"])
    pcr.pcr_set_hq1r_buffer(h, fb["hq1r_primary"])
    state = {"case": case, "ctx": ctx, "points": points, "fb": fb, "variant": VARIANTS[case["variant"]]}
    if case["graph"]:
        pcr.pcr_capture_begin(h)
        _launch_frame(state)
        state["graph"] = _Graph(pcr.pcr_capture_end(h))
    return state


def _prepare_reorder(case, seed):
    n = case["n"]
    ctx = _context()
    return {"case": case, "ctx": ctx, "seed": seed, "source": _cloud(case["scene"], n, seed),
            "points": torch.empty((n, 4), dtype=torch.int32, device=DEVICE),
            "workspace": torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device=DEVICE),
            "perm": torch.empty(n, dtype=torch.int32, device=DEVICE) if case["perm"] else None}


def _prepare_batch(case, seed):
    ctx = _context()
    h = ctx.handle
    clouds = [_reordered(ctx, _cloud("boxes", n, 8 * seed + c), "morton_shuffle128", seed)
              for c, n in enumerate(_sizes(case))]
    sizes = _view_sizes(case)
    jobs = scenes.batch_views(len(clouds), sizes)
    # one tensor per kind of buffer; each view's part starts on a multiple of 64 pixels
    starts, total = [], 0
    for _, v in jobs:
        starts.append(total)
        total += (v.width * v.height + 63) // 64 * 64
    words = {"keys": torch.int64, "image": torch.int32, "hq_depth": torch.int32, "hq_rg": torch.int64,
             "hq_ba": torch.int64, "hq_image": torch.int32}
    used = [k for k in words if case["flags"] & (pcr.PCR_BATCH_BASIC if k in ("keys", "image") else pcr.PCR_BATCH_HQ)]
    buffers = {k: torch.zeros(total, dtype=words[k], device=DEVICE) for k in used}
    views = [pcr.batch_view(v.matrix, v.width, v.height, c, case["flags"],
                            **{k: b[s:s + v.width * v.height] for k, b in buffers.items()})
             for (c, v), s in zip(jobs, starts)]
    workspace = torch.empty(pcr.pcr_batch_workspace_size(), dtype=torch.uint8, device=DEVICE)
    pcr.pcr_batch_prepare(h, [pcr.batch_cloud(c) for c in clouds], views, FACTOR, 0, workspace)
    state = {"case": case, "ctx": ctx, "clouds": clouds, "buffers": buffers, "workspace": workspace}
    if case["graph"]:
        state["graph"] = _Graph(pcr.pcr_batch_capture(h, workspace, 0))
    return state


def _prepare_serve(case, seed):
    ctx = _context()
    sizes = _sizes(case)
    clouds = [_reordered(ctx, _cloud("boxes", n, 8 * seed + c), "morton_shuffle128", seed)
              for c, n in enumerate(sizes)]
    # the stream's clouds and cameras; the resolutions in turn, and every other frame a high-quality one
    requests = []
    for i, (_, cloud, m, w, h, _) in enumerate(scenes.serve_requests(case["requests"], seed=seed,
                                                                     num_clouds=len(sizes))):
        size = scenes.SERVE_RESOLUTIONS[i % len(scenes.SERVE_RESOLUTIONS)]
        requests.append((cloud, _aspect(m, w, h, *size), *size, pcr.PCR_BATCH_HQ if i % 2 else pcr.PCR_BATCH_BASIC))
    width, height = max(s[0] for s in scenes.SERVE_RESOLUTIONS), max(s[1] for s in scenes.SERVE_RESOLUTIONS)
    arena = torch.empty(case["requests"] * 36 * width * height + (64 << 20), dtype=torch.uint8, device=DEVICE)
    server = _Server(pcr.pcr_server_create(ctx.handle, arena, width, height, case["requests"], max_batch_views=64,
                                           max_inflight=case["streams"], max_batch_clouds=1, depth_factor=FACTOR,
                                           policy=pcr.PCR_SERVE_LARGEST_GROUP))
    for c, points in enumerate(clouds):
        pcr.pcr_server_add_device_cloud(server.handle, c, points)
    torch.cuda.current_stream().synchronize()  # the server's streams read the clouds
    return {"case": case, "server": server, "ctx": ctx, "clouds": clouds, "arena": arena, "requests": requests}


# ---------------------------------------------------------------------------
# run
# ---------------------------------------------------------------------------

def run(state: dict):
    return {"frame": _run_frame, "reorder": _run_reorder, "batch": _run_batch, "serve": _run_serve}[
        state["case"]["kind"]](state)


def _launch_frame(state):
    h, fb, frame, variant = state["ctx"].handle, state["fb"], state["case"]["frame"], state["variant"]
    if frame == "basic":
        pcr.pcr_render_basic(h, variant, True)
        pcr.pcr_resolve(h, pcr.PCR_RESOLVE_BASIC, fb["image"], 0)
    elif frame == "rgb":
        pcr.pcr_render_rgb(h, variant, True)
        pcr.pcr_resolve(h, pcr.PCR_RESOLVE_RGB, fb["image"], 0)
    elif frame == "hq":
        pcr.pcr_render_hq(h, FACTOR, variant, True)
        pcr.pcr_resolve(h, pcr.PCR_RESOLVE_HQ, fb["image"], 0)
    else:
        pcr.pcr_render_hq1r(h, FACTOR, variant, True)
        pcr.pcr_resolve(h, pcr.PCR_RESOLVE_HQ1R, fb["image"], 0)


# Outputs of each frame.  How HQS1R splits a sum between its word and the
# fallback depends on the order of the adds; its image does not.
FRAME_OUTPUTS = {"basic": ("keys", "image"), "rgb": ("keys", "image"), "hq": ("hq_depth", "hq_rg", "hq_ba", "image"),
                 "hq1r": ("hq_depth", "image")}


def _run_frame(state):
    if "graph" in state:
        pcr.pcr_graph_launch(state["ctx"].handle, state["graph"].executable)
    else:
        _launch_frame(state)
    return [state["fb"][k] for k in FRAME_OUTPUTS[state["case"]["frame"]]]


def _run_reorder(state):
    """The order is made in place: on a copy, so that the source stays as it was."""
    points, perm = state["points"], state["perm"]
    points.copy_(state["source"])
    pcr.pcr_reorder_morton_shuffle128(state["ctx"].handle, points, points.shape[0], state["seed"],
                                      ORDERS[state["case"]["order"]], state["workspace"], perm)
    return [points] if perm is None else [points, perm]


def _run_batch(state):
    if "graph" in state:
        pcr.pcr_graph_launch(state["ctx"].handle, state["graph"].executable)
    else:
        pcr.pcr_batch_launch(state["ctx"].handle, state["workspace"], 0)
    return state["buffers"]


def _run_serve(state):
    server, arena = state["server"].handle, state["arena"]
    tickets = [pcr.pcr_server_submit(server, *request) for request in state["requests"]]
    done = 0
    while done < len(tickets):
        done += pcr.pcr_server_step(server)
    base = arena.data_ptr()

    def buffer(address, words, dtype):
        size = 8 if dtype == torch.int64 else 4
        return arena[address - base:address - base + words * size].view(dtype)

    out = []
    for ticket in tickets:
        r = pcr.pcr_server_get_result(server, ticket)
        px = r.width * r.height
        if r.flags & pcr.PCR_BATCH_BASIC:
            out += [buffer(r.keys, px, torch.int64), buffer(r.image, px, torch.int32)]
        else:
            out += [buffer(r.hq_depth, px, torch.int32), buffer(r.hq_rg, px, torch.int64),
                    buffer(r.hq_ba, px, torch.int64), buffer(r.hq_image, px, torch.int32)]
    pcr.pcr_server_poll_completed(server)
    for ticket in tickets:
        pcr.pcr_server_release(server, ticket)
    return out


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------

PROJECT_FLOPS = 28  # per point and view: three matrix rows, two divisions, the screen transform
BASIC_PIXEL, HQ_PIXEL, HQ1R_PIXEL = 8 + 4, 4 + 8 + 8 + 4, 4 + 4  # bytes of the buffers a frame returns


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "frame":
        pixel = {"basic": BASIC_PIXEL, "rgb": BASIC_PIXEL, "hq": HQ_PIXEL, "hq1r": HQ1R_PIXEL}[case["frame"]]
        return {"bytes": POINT * case["n"] + pixel * case["width"] * case["height"],
                "flops": PROJECT_FLOPS * case["n"]}
    if kind == "reorder":
        return {"bytes": (2 * POINT + (4 if case["perm"] else 0)) * case["n"], "flops": 0}
    sizes = _sizes(case)
    if kind == "batch":
        pixel = (BASIC_PIXEL if case["flags"] & 1 else 0) + (HQ_PIXEL if case["flags"] & 2 else 0)
        pixels = len(sizes) * sum(s * s for s in _view_sizes(case))
        return {"bytes": POINT * sum(sizes) + pixel * pixels, "flops": PROJECT_FLOPS * sum(sizes) * case["views"]}
    # half of the requests ask for a basic frame, half for a high-quality one; a mean resolution
    pixels = sum(w * h for w, h in scenes.SERVE_RESOLUTIONS) / len(scenes.SERVE_RESOLUTIONS)
    mean = sum(sizes) / len(sizes)
    return {"bytes": POINT * sum(sizes) + case["requests"] * pixels * (BASIC_PIXEL + HQ_PIXEL) / 2,
            "flops": PROJECT_FLOPS * case["requests"] * mean}


def tolerance(case: dict):
    return "exact"
