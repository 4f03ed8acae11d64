"""The calls that this library is used for, as cases whose time is measured.

A case is a dict of plain values.  Its "kind" names the entry points it goes
through:

  frame   Handle.compute and, with "uv", Handle.uvmap on device images: the
          camera loop of the paper (Sec. 3) with the images already on the GPU
  host    sgm_compute_host: the same from pinned host images to pinned host
          maps, copies included (a served camera frame)
  batch   Batch.run: many pairs of uneven size in one call
  maps    Handle.uvmap and uvmap_postprocess of a disparity map that the
          program already holds (Sec. 3.2)

Handles keep the settings they are created with; nothing is tuned per size.
All outputs are whole numbers.
"""
import random

import torch

from paper_1807_06271_gb300 import sgm

_STREAM4, _FOUR, _EIGHT = sgm.SGM_PATHS_STREAM4, sgm.SGM_PATHS_4, sgm.SGM_PATHS_8
# sizes and disparity counts of the pairs of a batch
_BATCH_SIZES = ((320, 240), (640, 480), (1242, 375), (1280, 720))
_BATCH_D = (64, 128)


def _case(kind, W, H, D, window, mask, P1, P2, median=5, cost="census", uv=True, rect=False, pad=0):
    return {"kind": kind, "W": W, "H": H, "D": D, "census_w": window[0], "census_h": window[1], "mask": mask,
            "P1": P1, "P2": P2, "median": median, "cost": cost, "uv": uv, "rect": rect, "pad": pad}


def listed():
    named = {
        # the smallest pair: a thumbnail for a fast first look; launches and chain latency
        "pair-160x96-d64": _case("frame", 160, 96, 64, (9, 7), _EIGHT, 8, 96, median=3),
        # a small on-board camera, four paths
        "pair-320x240-d64-4path": _case("frame", 320, 240, 64, (5, 5), _FOUR, 4, 24),
        # the paper's own setting (Sec. 4.1), both matching costs: D is no multiple of 8
        "paper-640x360-d60": _case("frame", 640, 360, 60, (5, 5), _STREAM4, 8, 32),
        "paper-640x360-d60-sad": _case("frame", 640, 360, 60, (5, 5), _STREAM4, 200, 800, cost="sad"),
        # a raw camera: odd size, padded rows, rectified through maps, 7x7 window, odd D
        "rectified-641x479-d97": _case("frame", 641, 479, 97, (7, 7), _EIGHT, 8, 64, median=3, rect=True, pad=63),
        # a served VGA camera frame, host buffers in and out
        "host-640x480-d64": _case("host", 640, 480, 64, (5, 5), _FOUR, 4, 24),
        # the KITTI shape with all eight paths: the headline workload
        "kitti-1242x375-d128": _case("frame", 1242, 375, 128, (9, 7), _EIGHT, 8, 96, median=3),
        # the same from a camera mounted on its side: the columns are the long axis
        "portrait-480x752-d128": _case("frame", 480, 752, 128, (9, 7), _EIGHT, 8, 96, median=3, uv=False),
        # HD, four paths, U/V maps
        "hd-1280x720-d128-4path": _case("frame", 1280, 720, 128, (5, 5), _FOUR, 4, 24),
        # full HD at a long range, eight paths: the largest single pair
        "fullhd-1920x1080-d192": _case("frame", 1920, 1080, 192, (9, 7), _EIGHT, 8, 96, median=3),
        # the maps of a HD disparity map alone: the smallest call
        "maps-1280x720-d128": _case("maps", 1280, 720, 128, (5, 5), _FOUR, 4, 24),
        # sixteen recorded pairs of mixed size, processed offline
        "batch-16-mixed": {"kind": "batch", "pairs": 16, "mix": 1810, "census_w": 9, "census_h": 7, "mask": _EIGHT,
                           "P1": 8, "P2": 96, "median": 3, "uv": True},
    }
    return [dict(case, name=name) for name, case in named.items()]


def draw(rng):
    """One more case: sizes spread evenly over the logarithm of the listed range, any parity."""
    most = _estimates(1920, 1080, 192) * 8
    kind = rng.choice(("frame", "frame", "frame", "frame", "frame", "host", "maps", "batch"))
    while kind == "batch":
        case = {"kind": "batch", "pairs": rng.randint(2, 16), "mix": rng.randrange(1 << 20), "census_w": 9,
                "census_h": 7, "mask": _EIGHT, "P1": 8, "P2": 96, "median": 3, "uv": True}
        if sum(_estimates(*shape) for shape in _batch_shapes(case)) * 8 <= 1.5 * most:
            return case
    while True:
        W, H = round(160 * 12 ** rng.random()), round(96 * 11.25 ** rng.random())
        D = rng.choice((32, 48, 60, 64, 64, 96, 97, 128, 128, 160, 192))
        mask = rng.choice((_EIGHT, _EIGHT, _FOUR, _STREAM4))
        if W > D and _estimates(W, H, D) * bin(mask).count("1") <= most:
            break
    if kind == "frame" and rng.random() < 0.2:
        return _case(kind, W, H, D, (5, 5), rng.choice((_FOUR, _STREAM4)), 200, 800, cost="sad",
                     uv=rng.random() < 0.5)
    window = rng.choice(((5, 5), (5, 5), (7, 7), (9, 7), (9, 7)))
    P1, P2 = rng.choice(((4, 24), (8, 32), (8, 64), (8, 96)))
    rect = kind == "frame" and rng.random() < 0.25
    return _case(kind, W, H, D, window, mask, P1, P2, median=rng.choice((0, 3, 3, 5, 5, 7)),
                 uv=kind == "host" or rng.random() < 0.6, rect=rect, pad=rng.choice((0, 0, 7, 64)) if kind == "frame" else 0)


def _estimates(W, H, D):
    return W * H * D


def _batch_shapes(case):
    rng = random.Random(case["mix"])
    return [(*rng.choice(_BATCH_SIZES), rng.choice(_BATCH_D)) for _ in range(case["pairs"])]


# ---- inputs ---------------------------------------------------------------------

def _box(img):
    """3 x 3 box filter with replicated borders."""
    pad = torch.nn.functional.pad(img[None, None], (1, 1, 1, 1), mode="replicate")
    return torch.nn.functional.avg_pool2d(pad, 3, 1)[0, 0]


def _scene(W, H, D, g):
    """(left, right, disparity) of a ground plane with boxes standing on it: blurred texture of two
    grains, sensor noise and pixels without a match, as the camera scenes of the tests have them."""
    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    coarse = torch.nn.functional.interpolate(rand(1, 1, H // 8 + 2, W // 8 + 2), size=(H, W), mode="bilinear")[0, 0]
    left = (_box(rand(H, W)) * 160 + coarse * 95).floor()
    horizon = (2 * H) // 5
    row = torch.arange(H, device="cuda", dtype=torch.float32)
    disp = ((row - horizon).clamp(min=0) * (0.7 * D / max(H - 1 - horizon, 1))).round()[:, None].repeat(1, W)
    for x, y, w, h, d in rand(6, 5).tolist():
        x0, y0 = int(x * W * 0.8), int(y * H * 0.7)
        box = disp[y0:y0 + 4 + int(h * H * 0.4), x0:x0 + 4 + int(w * W * 0.3)]
        box.clamp_(min=float(D // 8 + int(d * (D - D // 8 - 1))))
    col = torch.arange(W, device="cuda", dtype=torch.int64)
    src = col[None, :] + disp.long()
    right = torch.where(src < W, left.gather(1, src.clamp(max=W - 1)), rand(H, W) * 255)
    right = torch.where(rand(H, W) < 0.05, rand(H, W) * 255, right)
    right = (right + 2 * torch.randn(H, W, generator=g, device="cuda")).round().clamp(0, 255)
    return left.to(torch.uint8), right.to(torch.uint8), disp.clamp(max=D - 1).to(torch.uint8)


def _warp(W, H, g):
    """Rectification maps of a slightly rotated, shifted camera (some entries outside the image)."""
    a, b, c = ((torch.rand(3, generator=g, device="cuda") - 0.5) * 6).tolist()
    y, x = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
    mx = (x + a + b * y / H).round().int() & 0xFFFF
    my = (y + c + b * x / W).round().int() & 0xFFFF
    return mx.to(torch.uint16).contiguous(), my.to(torch.uint16).contiguous()


def _params(case):
    cost = sgm.SGM_COST_SAD if case.get("cost") == "sad" else sgm.SGM_COST_CENSUS
    pad = case.get("pad", 0)
    return sgm.SgmParams(census_w=case["census_w"], census_h=case["census_h"], path_mask=case["mask"], P1=case["P1"],
                         P2=case["P2"], lr_tolerance=1, median_k=case["median"],
                         row_pitch=case["W"] + pad if pad else 0, cost=cost)


def _outputs(W, H, D, uv, **where):
    out = {"disp": torch.empty((H, W), dtype=torch.uint8, **where)}
    if uv:
        out["umap"] = torch.empty((D, W), dtype=torch.int16, **where)
        out["vmap"] = torch.empty((H, D), dtype=torch.int16, **where)
    return out


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(case)
        scenes = [_scene(*shape, g) for shape in shapes]
        outs = [_outputs(*shape, case["uv"], device="cuda") for shape in shapes]
        return {"kind": kind, "batch": sgm.Batch(shapes, _params(case)), "left": [s[0] for s in scenes],
                "right": [s[1] for s in scenes], "out": {k: [o[k] for o in outs] for k in outs[0]}}
    W, H, D, pad = case["W"], case["H"], case["D"], case["pad"]
    left, right, disp = _scene(W, H, D, g)
    state = {"kind": kind, "handle": sgm.Handle(W, H, D, _params(case))}
    if kind == "maps":
        # some pixels have no valid match
        bad = torch.rand(H, W, generator=g, device="cuda") < 0.06
        state["disp"] = torch.where(bad, torch.full_like(disp, sgm.SGM_INVALID), disp)
        state["out"] = {k: v for k, v in _outputs(W, H, D, True, device="cuda").items() if k != "disp"}
        state["out"]["upost"] = torch.empty((D, W), dtype=torch.uint8, device="cuda")
        state["out"]["vpost"] = torch.empty((H, D), dtype=torch.uint8, device="cuda")
        return state
    if kind == "host":
        state["left"], state["right"] = left.cpu().pin_memory(), right.cpu().pin_memory()
        state["out"] = _outputs(W, H, D, True, pin_memory=True)
        return state
    if case["rect"]:
        maps = (*_warp(W, H, g), *_warp(W, H, g))
        sgm.sgm_set_rectification(state["handle"], *maps)
    state["left"], state["right"] = (torch.nn.functional.pad(t, (0, pad)).contiguous() for t in (left, right))
    state["out"] = _outputs(W, H, D, case["uv"], device="cuda")
    return state


# ---- one pass ----------------------------------------------------------------------

def run(state):
    out = state["out"]
    if state["kind"] == "batch":
        state["batch"].run(state["left"], state["right"], out["disp"], out.get("umap"), out.get("vmap"))
        return out
    h = state["handle"]
    if state["kind"] == "host":
        sgm.sgm_compute_host(h, state["left"], state["right"], out["disp"], out["umap"], out["vmap"])
    elif state["kind"] == "maps":
        h.uvmap(state["disp"], out["umap"], out["vmap"])
        sgm.uvmap_postprocess(h, out["umap"], out["vmap"], u_threshold=8, v_threshold=8, dilate_r=2,
                              uout=out["upost"], vout=out["vpost"])
    else:
        h.compute(state["left"], state["right"], out["disp"])
        if "umap" in out:
            h.uvmap(out["disp"], out["umap"], out["vmap"])
    return out


def work(case):
    """Images (and rectification maps) in, maps out; per estimate and path 3 minima, 2 sums, a
    difference and the running minimum of Eq. 2, the sum over the paths, 5 operations for the matching
    cost and 4 for the two winners.  Maps alone: one count and some 20 filter operations per cell."""
    if case["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for W, H, D in _batch_shapes(case):
            one = work(dict(case, kind="frame", W=W, H=H, D=D, rect=False))
            total = {k: total[k] + one[k] for k in total}
        return total
    W, H, D = case["W"], case["H"], case["D"]
    maps = 2 * D * (W + H)
    if case["kind"] == "maps":
        return {"bytes": W * H + maps + D * (W + H), "flops": 2 * W * H + 20 * D * (W + H)}
    paths = bin(case["mask"]).count("1")
    return {"bytes": 3 * W * H + (8 * W * H if case["rect"] else 0) + (maps if case["uv"] else 0),
            "flops": _estimates(W, H, D) * (8 * paths + 8)}


def exact(case, seed):
    """No output is a rounded number: all are whole and have to come out the same."""
    return None
