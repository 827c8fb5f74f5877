"""Cases for timing the visibility color map engine through its public entry points.

A case is a dict of plain values: the entry point it goes through (``call``),
the scene and the request's sizes and options.  ``prepare`` draws the scene
and the request's positions from a seed, ``run`` is one pass as a program of
the engine's user makes it, ``work`` the bytes and operations it cannot do
without, ``exact`` its result in float64 where that is quick.

Scenes are city-like box fields (clustered footprints, lognormal heights) or,
in 2D, uniform rectangles.  Every length is an integer number of 2^-10 m.
"""

import math
import random

import numpy as np
import torch

import paper_1310_7297_gb300 as vcm

U = 1024                      # lattice units per metre
NORMALS = (0, 1, 2, 3)        # +x, -x, +y, -y
PATCHES = ((8, 4), (16, 8), (32, 16), (64, 32))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(name, call, dims=3, boxes=5000, half_m=1000, nx=512, ny=512, layers=5, pu=32, pw=16, target_m=20,
          normal=2, flags=0, bits=False, fov=0.0, cell_m=0, levels=16, span_m=0, requests=1, side_max=1024, mix=0):
    """One case.  ``half_m``: half the scene's side; ``span_m``: half the
    viewpoint grid's side (0: all of the scene); ``cell_m``: the index's cell
    (0: the engine picks).  For several requests ``mix`` draws their
    sizes, sides log-uniform from 64 to ``side_max`` viewpoints."""
    c = dict(call=call, dims=dims, boxes=boxes, half_m=half_m, nx=nx, ny=ny, layers=layers, pu=pu, pw=pw,
             target_m=target_m, normal=normal, flags=flags, bits=bits, fov=fov, cell_m=cell_m, levels=levels,
             span_m=span_m, requests=requests, side_max=side_max, mix=mix)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain 2D map: a 10 m segment in a 1 km plane; the smallest call, mostly launches
        _case("segment_2d", "compute", dims=2, boxes=100, half_m=500, nx=128, ny=128, layers=1, pu=64, pw=1,
              target_m=10, levels=8),
        # the smallest request of a served mix, alone against a resident scene of 50,000 boxes
        _case("small_request", "compute", boxes=50000, half_m=5000, nx=64, ny=64, layers=1, pu=8, pw=4,
              target_m=12, normal=1, cell_m=50, span_m=1000),
        # the plain 3D map: five heights over a 2 km quarter
        _case("city", "compute"),
        # the same with its occlusion bits, which later gazes are recoloured from
        _case("city_bits", "compute", bits=True),
        # a sign seen from both faces, with a field of view; odd sizes throughout
        _case("two_sided_fov", "compute", boxes=2000, half_m=400, nx=97, ny=83, layers=3, pu=45, pw=13, normal=0,
              flags=vcm.VCM_TWO_SIDED, fov=120.0),
        # only the places that see the whole target
        _case("strict", "compute", flags=vcm.VCM_STRICT, normal=3),
        # the viewer-centric map: one segment per cell
        _case("viewer", "compute", pu=1, pw=1, target_m=2, flags=vcm.VCM_VIEWER),
        # a new gaze over bits made earlier
        _case("recolor_gaze", "recolor", fov=120.0),
        # scene and map in one call that allocates nothing
        _case("static_scene", "static", boxes=1500, half_m=400, nx=96, ny=96, layers=2, pu=16, pw=8),
        # a served mix of interactive sizes: submitted, polled and read on the host
        _case("serve_mix", "serve", boxes=100000, half_m=5000, cell_m=50, requests=24, side_max=256, mix=1),
        # uneven requests in one launch
        _case("batch", "batch", boxes=50000, half_m=5000, cell_m=50, requests=64, mix=2),
        # a large target over a whole city: 33.5 M viewpoints of 2,048 patches
        _case("large_city", "compute", boxes=100000, half_m=5000, nx=2048, ny=2048, layers=8, pu=64, pw=32,
              target_m=40, cell_m=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("2d", "3d", "3d", "3d", "option", "viewer", "recolor", "static", "batch", "serve", "large"))
    nx, ny, layers = _log_int(rng, 48, 640), _log_int(rng, 48, 640), rng.randint(1, 6)
    pu, pw = rng.choice(PATCHES) if rng.random() < 0.6 else (_log_int(rng, 4, 80), _log_int(rng, 2, 40))
    normal, boxes = rng.choice(NORMALS), _log_int(rng, 200, 20000)
    half = int(1000 * max(0.3, math.sqrt(boxes / 5000.0)))
    target, levels = rng.randint(2, 50), rng.choice((8, 16, 64, 256))
    one = dict(boxes=boxes, half_m=half, nx=nx, ny=ny, layers=layers, pu=pu, pw=pw, target_m=target, normal=normal,
               levels=levels)
    if kind == "2d":
        n = _log_int(rng, 64, 512)
        return _case(None, "compute", dims=2, boxes=_log_int(rng, 40, 800), half_m=500, nx=n, ny=n + rng.randint(0, 9),
                     layers=1, pu=_log_int(rng, 8, 200), pw=1, target_m=rng.randint(4, 40), normal=normal, levels=8)
    if kind == "3d":
        return _case(None, "compute", bits=rng.random() < 0.3, **one)
    if kind == "option":
        flags = rng.choice((0, vcm.VCM_STRICT, vcm.VCM_TWO_SIDED, vcm.VCM_STRICT | vcm.VCM_TWO_SIDED))
        return _case(None, "compute", flags=flags, fov=rng.choice((0.0, 60.0, 120.0, 200.0)),
                     bits=rng.random() < 0.3, **one)
    if kind == "viewer":
        return _case(None, "compute", **dict(one, pu=1, pw=1, target_m=rng.randint(1, 5), flags=vcm.VCM_VIEWER))
    if kind == "recolor":
        return _case(None, "recolor", fov=rng.choice((0.0, 60.0, 120.0)),
                     flags=rng.choice((0, vcm.VCM_STRICT, vcm.VCM_TWO_SIDED)), **one)
    if kind == "static":
        return _case(None, "static", **dict(one, boxes=_log_int(rng, 50, 4000), half_m=500, nx=_log_int(rng, 32, 256),
                                            ny=_log_int(rng, 32, 256), layers=rng.randint(1, 3)))
    if kind == "batch":
        return _case(None, "batch", boxes=50000, half_m=5000, cell_m=50, requests=rng.randint(2, 24),
                     side_max=rng.choice((256, 512, 1024)), mix=rng.randint(10, 10 ** 6))
    if kind == "serve":
        return _case(None, "serve", boxes=100000, half_m=5000, cell_m=50, requests=rng.randint(2, 24), side_max=256,
                     mix=rng.randint(10, 10 ** 6))
    return _case(None, "compute", boxes=100000, half_m=5000, nx=_log_int(rng, 512, 2048), ny=_log_int(rng, 512, 2048),
                 layers=rng.randint(1, 6), pu=64, pw=32, target_m=rng.randint(20, 50), normal=normal, cell_m=50,
                 span_m=rng.choice((0, 1000)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _units(x_m):
    return np.floor(np.asarray(x_m) * U + 0.5).astype(np.int64)


def _hits(lo, hi, a, b, dims):
    return np.all((lo[:, :dims] <= b[:dims]) & (a[:dims] <= hi[:, :dims]), axis=1)


def _target_extent(r):
    """The target's box plus a metre each way."""
    half = np.full(3, U, np.int64)
    half[r["axis_u"] >> 1] += r["width"] // 2 + 1
    if r["dims"] == 3:
        half[r["axis_w"] >> 1] += r["height"] // 2 + 1
    c = np.array(r["center"], np.int64)
    return c - half, c + half


def _scene(case, rng, keep_out):
    """Box corners in lattice units, none of them on the target."""
    n, half, dims = case["boxes"], case["half_m"], case["dims"]
    comps = 64 if half >= 3000 else 16
    means = rng.uniform(-half, half, (comps, 2))
    sigma = rng.uniform(0.05, 0.25, comps) * min(half, 1000) * (1.0 if half < 3000 else 2.4)
    los, his, got = [], [], 0
    while got < n:
        m = n + n // 2 + 16
        if dims == 2:
            ctr, size = rng.uniform(-half, half, (m, 2)), rng.uniform(5, 30, (m, 2))
            top = np.zeros(m)
        else:
            k = rng.integers(0, comps, m)
            ctr = means[k] + rng.normal(size=(m, 2)) * sigma[k][:, None]
            size = rng.uniform(10, 60, (m, 2))
            top = np.exp(math.log(20.0) + 0.6 * rng.normal(size=m))
        lo = np.zeros((m, 3), np.int64)
        hi = np.zeros((m, 3), np.int64)
        lo[:, :2], hi[:, :2] = _units(ctr - size / 2), _units(ctr + size / 2)
        if dims == 3:
            hi[:, 2] = np.maximum(1, _units(top))
        ok = (np.abs(lo[:, :2]).max(axis=1) <= half * U) & (np.abs(hi[:, :2]).max(axis=1) <= half * U)
        if keep_out is not None:
            ok &= ~_hits(lo, hi, keep_out[0], keep_out[1], dims)
        los.append(lo[ok])
        his.append(hi[ok])
        got += int(ok.sum())
    return np.concatenate(los)[:n], np.concatenate(his)[:n]


def _request(case, rng):
    """The case's single request: the target near the middle of the scene,
    the viewpoint grid centred on it."""
    half, dims = case["span_m"] or case["half_m"], case["dims"]
    jitter = rng.integers(-4 * U, 4 * U + 1, 2)
    step = [max(1, 2 * half * U // case["nx"]), max(1, 2 * half * U // case["ny"])]
    horizontal = 0 if (case["normal"] >> 1) == 1 else 2
    gaze = rng.uniform(-0.5, 0.5, 3)
    gaze[case["normal"] >> 1] += -1.0 if case["normal"] & 1 else 1.0
    return {
        "dims": dims, "center": [int(jitter[0]), int(jitter[1]), 30 * U if dims == 3 else 0], "axis_u": horizontal,
        "axis_w": 4, "normal": case["normal"], "width": case["target_m"] * U,
        "height": case["target_m"] * U // 2 if dims == 3 else 0, "patches_u": case["pu"], "patches_w": case["pw"],
        "grid_origin": [-half * U, -half * U], "grid_step": [int(s) for s in step], "grid_nx": case["nx"],
        "grid_ny": case["ny"], "layer_z": [1741 + 10 * U * k for k in range(case["layers"])] if dims == 3 else [0],
        "color_levels": case["levels"], "v_ref": 0.0, "flags": case["flags"], "fov_deg": case["fov"],
        "gaze": tuple(float(np.float32(g)) for g in gaze) if case["fov"] > 0 else (0.0, 0.0, 0.0),
    }


def _mix_sizes(case):
    """(side, layers, patches_u, patches_w, target metres) of each request of a mix."""
    rng = random.Random(case["mix"])
    return [(_log_int(rng, 64, case["side_max"]), rng.randint(1, 8)) + rng.choice(PATCHES) + (rng.randint(2, 50),)
            for _ in range(case["requests"])]


def _mix_requests(case, rng, lo, hi):
    """Targets anywhere in the scene, each with a 2 km square of viewpoints around it."""
    half = case["half_m"]
    out = []
    for side, layers, pu, pw, width in _mix_sizes(case):
        step = 2000 * U // side
        while True:
            normal = int(rng.integers(0, 4))
            c = _units(np.append(rng.uniform(-half + 100, half - 100, 2), rng.uniform(10, 60)))
            o = np.clip(c[:2] - step * side // 2, -half * U, half * U - step * side)
            r = {"dims": 3, "center": [int(x) for x in c], "axis_u": 2 if normal < 2 else 0, "axis_w": 4,
                 "normal": normal, "width": width * U, "height": width * U // 2, "patches_u": pu, "patches_w": pw,
                 "grid_origin": [int(o[0]), int(o[1])], "grid_step": [step, step], "grid_nx": side, "grid_ny": side,
                 "layer_z": [1741 + 10 * U * k for k in range(layers)], "color_levels": 16, "v_ref": 0.0, "flags": 0}
            if not _hits(lo, hi, *_target_extent(r), 3).any():
                break
        out.append(r)
    return out


def _inputs(case, seed):
    """Scene corners (lattice units) and the requests of a seed."""
    rng = np.random.default_rng(int(seed))
    if case["requests"] > 1:
        lo, hi = _scene(case, rng, None)
        return lo, hi, _mix_requests(case, rng, lo, hi)
    req = _request(case, rng)
    lo, hi = _scene(case, rng, _target_extent(req))
    return lo, hi, [req]


def prepare(case, seed):
    lo, hi, reqs = _inputs(case, seed)
    lo, hi = (lo / U).astype(np.float32), (hi / U).astype(np.float32)
    state = {"case": case, "reqs": reqs, "req": reqs[0]}
    if case["call"] == "static":
        # the caller's own buffers: this entry point allocates nothing
        n = vcm.n_viewpoints(reqs[0])
        state.update(lo=lo, hi=hi, v=torch.empty(n, dtype=torch.float32, device="cuda"),
                     color=torch.empty(n, dtype=torch.uint8, device="cuda"),
                     stats=torch.empty(vcm.vcm.STATS_BYTES, dtype=torch.uint8, device="cuda"))
        return state
    ctx = state["ctx"] = vcm.Context(0)
    ctx.vcm_scene_load_mem(lo, hi, case["dims"])
    ctx.vcm_build(case["cell_m"])
    if case["call"] == "recolor":
        plain = dict(reqs[0], flags=0, fov_deg=0.0, gaze=(0.0, 0.0, 0.0))
        state["bits"] = ctx.compute(plain, emit_bits=True)[2]
    if case["call"] == "batch":
        # one buffer for all values and one for all colors, a 256-byte aligned part for each request
        at, total = [], 0
        for r in reqs:
            at.append(total)
            total += -(-vcm.n_viewpoints(r) // 256) * 256
        state["v"] = torch.zeros(total, dtype=torch.float32, device="cuda")
        state["color"] = torch.zeros(total, dtype=torch.uint8, device="cuda")
        state["stats"] = torch.zeros(vcm.vcm.STATS_BYTES * len(reqs), dtype=torch.uint8, device="cuda")
        state["d_v"] = [state["v"].data_ptr() + 4 * a for a in at]
        state["d_color"] = [state["color"].data_ptr() + a for a in at]
    return state


def run(state):
    case, req = state["case"], state["req"]
    call = case["call"]
    if call == "compute":
        v, color, bits, _ = state["ctx"].compute(req, emit_bits=case["bits"])
        return {"v": v, "color": color, "bits": bits} if case["bits"] else {"v": v, "color": color}
    if call == "recolor":
        v, color, _ = state["ctx"].recolor(req, state["bits"])
        return {"v": v, "color": color}
    stream = torch.cuda.current_stream().cuda_stream
    if call == "static":
        vcm.vcm.vcm_compute_static(state["lo"], state["hi"], case["dims"], req, state["v"].data_ptr(),
                                   state["color"].data_ptr(), None, state["stats"].data_ptr(), stream)
        return {"v": state["v"], "color": state["color"]}
    if call == "batch":
        state["ctx"].vcm_compute_batch(state["reqs"], state["d_v"], state["d_color"], [None] * len(state["reqs"]),
                                       state["stats"].data_ptr(), stream)
        return {"v": state["v"], "color": state["color"]}
    ctx, out = state["ctx"], []
    for t in [ctx.vcm_submit(r) for r in state["reqs"]]:
        ctx.vcm_poll(t, -1)
        v, color, _, _ = ctx.vcm_result_get(t)
        ctx.vcm_result_release(t)
        out.append({"v": v, "color": color})
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the boxes (six or four floats each) and the bits of a recolour
    read once, values, colors and bits written once.  Operations: one slab
    test (19 float operations, 13 in 2D) per viewpoint, the least that shows
    a viewpoint blocked; a recolour's 12 of the side and cone test."""
    if case["requests"] > 1:
        vp = sum(side * side * layers for side, layers, _, _, _ in _mix_sizes(case))
    else:
        vp = case["nx"] * case["ny"] * (case["layers"] if case["dims"] == 3 else 1)
    words = 1 if case["flags"] & vcm.VCM_VIEWER else -(-case["pu"] * case["pw"] // 32)
    bits = 4 * words * vp if case["bits"] or case["call"] == "recolor" else 0
    scene = 0 if case["call"] == "recolor" else case["boxes"] * 8 * case["dims"]
    per_vp = 12 if case["call"] == "recolor" else 19 if case["dims"] == 3 else 13
    return {"bytes": scene + bits + 5 * vp, "flops": per_vp * vp}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------

def _rounded(num, den):
    """num / den of integers, halves away from zero."""
    return np.sign(num) * ((2 * np.abs(num) + den) // (2 * den))


def exact(case, seed):
    """Values (and bits) by testing every segment against every box in
    float64; None where that would take long, or for the mixes."""
    if case["requests"] > 1 or case["call"] == "recolor":
        return None
    viewer = bool(case["flags"] & vcm.VCM_VIEWER)
    P = 1 if viewer else case["pu"] * case["pw"]
    n_vp = case["nx"] * case["ny"] * case["layers"]
    if float(n_vp) * P * case["boxes"] > 4e10:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    lo, hi, (r,) = _inputs(case, seed)
    dims = case["dims"]

    def t64(x):
        return torch.as_tensor(np.asarray(x, np.float64) / U, device=dev)

    # viewpoints in output order
    axis = [t64(_rounded(2 * r["grid_origin"][k] + (2 * np.arange(n) + 1) * r["grid_step"][k], 2))
            for k, n in ((0, case["nx"]), (1, case["ny"]))]
    z, y, x = torch.meshgrid(t64(r["layer_z"]), axis[1], axis[0], indexing="ij")
    q = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1) * (1.0 if dims == 3 else 0.0)], 1)
    # patch centres, columns fastest
    if viewer:
        p = t64([r["center"]])
    else:
        pts = np.tile(np.array(r["center"], np.int64), (P, 1))
        for code, count, extent, index in ((r["axis_u"], case["pu"], r["width"], np.arange(P) % case["pu"]),
                                           (r["axis_w"], case["pw"], r["height"], np.arange(P) // case["pu"])):
            if extent:
                a, sign = code >> 1, -1 if code & 1 else 1
                pts[:, a] = _rounded(2 * count * pts[:, a] + sign * (2 * index + 1 - count) * extent, 2 * count)
        p = t64(pts)
    blo, bhi = t64(lo), t64(hi)
    plo, phi = p.min(0).values, p.max(0).values
    blocked = torch.zeros(n_vp, P, dtype=torch.bool, device=dev)
    axes = list(range(dims))
    per_box = max(1, int(2e7 // P))
    rows = 2048
    for a in range(0, n_vp, rows):
        qs = q[a:a + rows]
        # boxes that meet the bounds of these viewpoints and the target
        mlo, mhi = torch.minimum(qs.min(0).values, plo), torch.maximum(qs.max(0).values, phi)
        near = ((blo <= mhi) & (bhi >= mlo))[:, :dims].all(1).nonzero()[:, 0]
        k = max(1, per_box // qs.shape[0])
        for b in range(0, near.numel(), k):
            l, h = blo[near[b:b + k]], bhi[near[b:b + k]]
            enter = torch.zeros((), dtype=torch.float64, device=dev)
            leave = torch.ones((), dtype=torch.float64, device=dev)
            for ax in axes:
                d = (p[None, :, ax] - qs[:, None, ax])[:, :, None]
                t0 = (l[None, :, ax] - qs[:, None, ax])[:, None, :] / d
                t1 = (h[None, :, ax] - qs[:, None, ax])[:, None, :] / d
                # a zero direction inside the slab (infinities of both signs, or 0 / 0) does not constrain
                inside = (l[None, :, ax] <= qs[:, None, ax]) & (qs[:, None, ax] <= h[None, :, ax])
                free = (d == 0) & inside[:, None, :]
                first = torch.where(free, -torch.inf, torch.minimum(t0, t1))
                last = torch.where(free, torch.inf, torch.maximum(t0, t1))
                enter, leave = torch.maximum(enter, first), torch.minimum(leave, last)
            blocked[a:a + rows] |= (enter <= leave).any(2)
    # the measure
    v = torch.zeros(n_vp, dtype=torch.float64, device=dev)
    if viewer:
        D = (q - p).square().sum(1).sqrt()
        S = r["width"] / U
        see = ~blocked[:, 0] & (D > 0)
        v[see] = 4 * torch.asin(S * S / (4 * D[see] ** 2 + S * S)) if dims == 3 else 2 * torch.atan(S / (2 * D[see]))
    else:
        na = r["normal"] >> 1
        sign = -1.0 if r["normal"] & 1 else 1.0
        two = bool(case["flags"] & vcm.VCM_TWO_SIDED)
        area = r["width"] / U / case["pu"] * (r["height"] / U / case["pw"] if dims == 3 else 1.0)
        g = np.array(r["gaze"][:dims] + (0.0,) * (3 - dims), np.float64)
        if not g.any():
            g[na] = sign
        g = torch.as_tensor(g / np.linalg.norm(g), device=dev)
        for a in range(0, n_vp, rows):
            d = q[a:a + rows, None, :] - p[None, :, :]
            s = d[:, :, na] * sign
            s = s.abs() if two else s
            dist = d.square().sum(2).sqrt()
            term = area * s / (dist ** 3 if dims == 3 else dist ** 2)
            ok = ~blocked[a:a + rows] & (s > 0)
            if 0 < case["fov"] < 360:
                along = (d * g).sum(2)
                along = along.abs() if two else along
                ok &= along >= math.cos(case["fov"] * math.pi / 360) * dist
            v[a:a + rows] = torch.where(ok, term, 0.0).sum(1)
        if case["flags"] & vcm.VCM_STRICT:
            v[blocked.any(1)] = 0.0
    out = {"v": v, "color": None}
    if case["bits"]:
        words = -(-P // 32)
        full = torch.zeros(n_vp, words * 32, dtype=torch.int64, device=dev)
        full[:, :P] = blocked
        w = (full.reshape(n_vp, words, 32) << torch.arange(32, device=dev)).sum(2)
        out["bits"] = torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32).reshape(-1)
    return out
