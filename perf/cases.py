"""The calls a user of this framework spends time in, as measurable cases.

A case is one call (or the short sequence of calls a program makes per optimisation step) on a
synthetic collage: the optimisation step in its forms (device-resident, host buffers, loss and
gradient for the caller's own step, autograd), the coarse-to-fine schedule, the outline fitting,
the render, the quality metrics and the skeleton-based initialisation.  Sizes follow the
repository's workloads and the resolutions and element counts of the paper's tables (100 elements
of 20 cubics at up to 1200 px); ``draw`` spreads over the same ranges, ragged sizes included.

``exact`` restates each call in 64-bit torch from the definitions alone: coverage from the signed
distance of every (element, pixel) pair, the losses of Eqs. 5-8, the closed-form adjoint and Adam.
"""
from __future__ import annotations

import math

import numpy as np
import torch

# ------------------------------------------------------------------------------------------------
# Cases
# ------------------------------------------------------------------------------------------------
_DEFAULTS = dict(op="step", mix="mixed", cubics=8, container="annulus", n=100, fill=0.75,
                 spread=0.5, res=512, batch=1, pad=0.0, uniform=True, force=0.0, tile=8,
                 deterministic=False, iters=4, maps=False)


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest collage: a few disks on a coarse grid, several iterations per call (launches
        # and the call's own latency count), library defaults
        _case("disks16_128_step", mix="disks", container="disk", n=16, fill=0.28, spread=0.33,
              res=128, uniform=False, tile=16, iters=10),
        # an interactive program's own optimiser around the autograd function, small ragged grid
        _case("mixed120_200_autograd", op="autograd", n=120, res=200, pad=2.0, tile=16),
        # a mid-size crowded collage, the plain optimisation loop
        _case("blobs200_512_step", mix="blobs", container="star", n=200, fill=2.9, res=512),
        # the paper's workload (100 closed paths of 20 cubics, Table 1) at 1000 px: loss and gradient
        # for a program that steps by itself
        _case("outlines100_1000_gradient", op="gradient", mix="blobs", cubics=20, container="star",
              n=100, fill=0.9, spread=0.3, res=1000, tile=16),
        # the headline level end to end: params in host memory in and out at every iteration
        _case("mixed1000_1024_host", op="host", n=1000, res=1024, pad=2.0),
        # the coarse-to-fine run of a whole collage (a tenth of the usual iterations per level)
        _case("mixed1000_schedule", op="schedule", n=1000, res=1024, pad=2.0, iters=5),
        # many independent collages of uneven size in one handle
        _case("batch64_step", mix="disks_blobs", container="any", n=410, fill=0.5, spread=0.3,
              res=1024, batch=64, iters=2),
        # the largest collage: open packing with reproducible gradients
        _case("open5000_2048_step_det", container="rect", n=5000, fill=2.9, spread=0.6, res=2048,
              pad=1.0, force=1e3, deterministic=True, iters=2),
        # the picture of that collage (previews, export)
        _case("open5000_2048_render", op="render", container="rect", n=5000, fill=2.9, spread=0.6,
              res=2048, pad=1.0),
        # the quality report after a run
        _case("mixed1000_1024_metrics", op="metrics", n=1000, res=1024),
        # the skeleton-based initialisation before a run, with its maps
        _case("mixed1000_1024_mat_init", op="mat_init", n=1000, res=1024, maps=True),
        # items traced from silhouettes: gradient of the outline points, a batch of outlines
        _case("fit64_256_gradient", op="fit", mix="blobs", cubics=20, container="star", n=1, res=256,
              batch=64, uniform=False),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["step"] * 6 + ["gradient"] * 3 + ["host"] * 2 + ["render"] * 2 +
                    ["autograd", "schedule", "metrics", "mat_init", "fit"])
    c = _case(op=op, mix=rng.choice(["disks", "blobs", "mixed", "mixed", "disks_blobs"]),
              cubics=rng.choice([4, 8, 8, 20]), container=rng.choice(["disk", "annulus", "star", "rect"]),
              fill=round(math.exp(rng.uniform(math.log(0.25), math.log(3.0))), 3),
              spread=round(rng.uniform(0.1, 0.6), 3), res=logint(64, 2048),
              pad=rng.choice([0.0, 0.0, 1.0, 2.0]), uniform=rng.random() < 0.8,
              force=rng.choice([0.0, 0.0, 1e3]), tile=rng.choice([8, 8, 16]),
              deterministic=rng.random() < 0.3, iters=rng.randint(1, 8))
    if op == "fit":
        return dict(c, mix="blobs", cubics=rng.choice([8, 12, 20]), container="star", n=1, pad=0.0,
                    res=logint(96, 384), batch=logint(1, 64), uniform=False, force=0.0)
    if op == "schedule":
        c.update(res=8 * logint(16, 128), iters=rng.randint(1, 5))
    if op in ("metrics", "mat_init"):
        c.update(res=logint(64, 1200), maps=rng.random() < 0.5)
    if op == "step" and rng.random() < 0.25:  # a batch: grids of a quarter, a half and the whole of res
        c.update(res=4 * logint(32, 256), batch=logint(2, 48), mix="disks_blobs", container="any",
                 fill=min(c["fill"], 0.7), iters=rng.randint(1, 2))
    # mean radius of at least 4 px, at most 5000 elements (1000 where every level runs or each is placed)
    most = c["fill"] * 0.6 * c["res"] ** 2 / (16 * math.pi)
    if c["batch"] > 1:
        most /= 16
    c["n"] = logint(4, max(5, min(1000 if op in ("schedule", "mat_init") or c["batch"] > 1 else 5000, most)))
    if c["batch"] > 1:
        c["n"] = max(12, min(c["n"], 410))
    return c


# ------------------------------------------------------------------------------------------------
# Inputs: element outlines, containers and initial transforms, from the seed alone
# ------------------------------------------------------------------------------------------------
def _ring(r, m, phase=0.0):
    a = phase + 2.0 * np.pi * np.arange(m) / m
    return 0.5 + np.stack([r * np.cos(a), r * np.sin(a)], 1)


def _container(kind, rng, n):
    """(rings, area, n positions inside)"""
    def polar(r0, r1):
        rad = np.sqrt(rng.uniform(r0 * r0, r1 * r1, n))
        a = rng.uniform(0.0, 2.0 * np.pi, n)
        return 0.5 + np.stack([rad * np.cos(a), rad * np.sin(a)], 1)

    if kind == "disk":
        return [_ring(0.45, 256)], math.pi * 0.45 ** 2, polar(0.0, 0.4)
    if kind == "annulus":
        return [_ring(0.48, 256), _ring(0.2, 256)[::-1]], math.pi * (0.48 ** 2 - 0.2 ** 2), polar(0.2, 0.48)
    if kind == "star":
        a = rng.uniform(0.0, 2.0 * np.pi) + 2.0 * np.pi * np.arange(24) / 24
        rad = np.where(np.arange(24) % 2 == 0, 0.45, 0.25)
        ring = 0.5 + np.stack([rad * np.cos(a), rad * np.sin(a)], 1)
        return [ring], 12 * 0.25 * 0.45 * math.sin(math.pi / 12), polar(0.0, 0.27)
    ring = np.array([(0.05, -0.1), (0.95, -0.1), (0.95, 0.95), (0.05, 0.95)])
    return [ring], 0.9 * 0.95, np.stack([rng.uniform(0.05, 0.95, n), rng.uniform(0.0, 0.95, n)], 1)


def _outline(kind, r, rng, cubics):
    """(library kind, points, stroke half-width) of one element of radius r"""
    if kind == "disk":
        return 1, _ring(r, 32) - 0.5, 0.0
    if kind == "blob":
        m = 3 * cubics
        a = 2.0 * np.pi * np.arange(m) / m
        rad = rng.uniform(0.6, 1.0, m) * r
        return 0, np.stack([rad * np.cos(a), rad * np.sin(a)], 1), 0.0
    if kind == "polygon":
        a = np.sort(rng.uniform(0.0, 2.0 * np.pi, rng.integers(5, 13)))
        return 1, np.stack([r * np.cos(a), r * np.sin(a)], 1), 0.0
    m = int(rng.integers(4, 11))
    return 2, np.stack([np.linspace(-r, r, m), r * rng.uniform(-0.5, 0.5, m)], 1), 0.002


def _kinds(mix, n, rng):
    if mix == "disks":
        return ["disk"] * n
    if mix == "blobs":
        return ["blob"] * n
    u = rng.random(n)
    if mix == "disks_blobs":
        return ["disk" if x < 0.5 else "blob" for x in u]
    return ["blob" if x < 0.6 else "polygon" if x < 0.9 else "stroke" for x in u]


def _problem(case, rng, sizes):
    n, grid, container = case["n"], case["res"], case["container"]
    if case["op"] == "fit":
        # a rough closed path about the centre, fitted to a 12-point star silhouette
        r = rng.uniform(0.25, 0.33)
        rings, _, _ = _container("star", rng, 1)
        m = 3 * case["cubics"]
        a = 2.0 * np.pi * np.arange(m) / m
        rad = r * rng.uniform(0.97, 1.03, m)
        outlines = [(0, np.stack([rad * np.cos(a), rad * np.sin(a)], 1), 0.0)]
        params = np.array([[0.5 + rng.uniform(-0.01, 0.01), 0.5 + rng.uniform(-0.01, 0.01),
                            rng.uniform(0.01, 0.1), 1.0]])
    else:
        if case["batch"] > 1:
            n = int(sizes.integers(min(20, n), max(2 * n - 20, n) + 1))
            grid = grid // int(sizes.choice([1, 2, 4]))
            n = max(4, min(n, int(0.01 * grid * grid)))
        if container == "any":
            container = str(rng.choice(["star", "annulus"]))
        rings, area, pos = _container(container, rng, n)
        radius = math.sqrt(case["fill"] * area / (n * math.pi)) * rng.uniform(1 - case["spread"], 1 + case["spread"], n)
        outlines = [_outline(k, r, rng, case["cubics"]) for k, r in zip(_kinds(case["mix"], n, rng), radius)]
        params = np.stack([pos[:, 0], pos[:, 1], rng.uniform(0.0, 2.0 * np.pi, n), rng.uniform(0.9, 1.1, n)], 1)
    return {
        "kind": np.array([o[0] for o in outlines], np.int32),
        "pt_off": np.cumsum([0] + [len(o[1]) for o in outlines]).astype(np.int32),
        "pts": np.concatenate([o[1] for o in outlines]).astype(np.float32).reshape(-1),
        "hw": np.array([o[2] for o in outlines], np.float32),
        "params0": params.astype(np.float32).reshape(-1),
        "ring_off": np.cumsum([0] + [len(r) for r in rings]).astype(np.int32),
        "ring_pts": np.concatenate(rings).astype(np.float32).reshape(-1),
        "grid": int(grid),
    }


def _inputs(case, seed):
    """The problems, and the optimiser's moments after a while of optimising (float32)."""
    rng = np.random.default_rng([20240604, int(seed)])
    sizes = np.random.default_rng([case["n"], case["res"], case["batch"]])  # a batch's counts and grids: the case's
    problems = [_problem(case, rng, sizes) for _ in range(case["batch"])]
    r = np.concatenate([np.maximum.reduceat(np.hypot(*p["pts"].reshape(-1, 2).T), p["pt_off"][:-1]) for p in problems])
    # gradients grow with the outline's length; those of theta and s with the radius as well
    scale = 3e5 * r[:, None] * np.stack([np.ones_like(r), np.ones_like(r), r, r], 1)
    m = (0.1 * scale * rng.standard_normal(scale.shape)).astype(np.float32)
    v = (scale * scale * rng.uniform(0.5, 2.0, scale.shape)).astype(np.float32)
    return problems, m, v


_ADAM_STEP = 200  # iterations the optimiser has behind it


def _options(case):
    o = dict(pad_px=case["pad"], delta_down=case["force"], tile=case["tile"],
             deterministic=int(case["deterministic"]), level_res=[case["res"]], level_iters=[case["iters"]])
    if not case["uniform"]:
        o["gamma"] = 0.0
    if case["op"] == "schedule":
        o.update(level_res=[case["res"] // k for k in (8, 4, 2, 1)], level_iters=[case["iters"] * k for k in (6, 4, 2, 1)],
                 n_levels=4)
    if case["op"] == "fit":
        o.update(alpha=1.0, beta=0.0, gamma=0.0, delta_down=0.0, w_in=1.0, w_out=1.0, fit_controls=1)
    return o


def prepare(case, seed):
    from paper_2406_04008_gb300.collage import Collage

    problems, m, v = _inputs(case, seed)
    params = np.concatenate([p["params0"] for p in problems]).reshape(-1, 4)
    state = {"op": case["op"], "iters": case["iters"], "maps": case["maps"],
             "col": Collage(problems, **_options(case)),
             "params": torch.from_numpy(params.copy()).cuda(), "host_params": params.reshape(-1).copy()}
    if case["op"] in ("step", "host", "schedule"):
        moments = torch.from_numpy(np.concatenate([params.reshape(-1), m.reshape(-1), v.reshape(-1)])).cuda()
        state["col"].set_state(moments, _ADAM_STEP, 0)
    if case["op"] == "fit":
        state["points"] = torch.from_numpy(np.concatenate([p["pts"] for p in problems])).cuda()
    return state


def run(state):
    from paper_2406_04008_gb300.collage import collage_loss

    col, op = state["col"], state["op"]
    if op == "step":  # the params a program holds, some iterations, the new params and the loss
        col.set_params(state["params"])
        col.step(state["iters"])
        return col.get_params(), col.loss()
    if op == "host":  # one iteration on host buffers
        params, loss = col.step_host(1, state["host_params"])
        return params, loss
    if op == "autograd":  # the program's own optimiser
        params = state["params"].detach().requires_grad_()
        loss = collage_loss(params, col)
        loss.backward()
        return loss.detach(), params.grad
    if op == "gradient":
        col.set_params(state["params"])
        return col.loss_backward()
    if op == "schedule":
        col.set_level(0)
        col.set_params(state["params"])
        col.run_schedule()
        return col.get_params(), col.loss()
    if op == "render":
        col.set_params(state["params"])
        return col.render()
    if op == "metrics":
        col.set_params(state["params"])
        return col.metrics()
    if op == "mat_init":
        axis, width = col.mat_init(want_maps=state["maps"])
        return [col.get_params()] + ([axis, width] if state["maps"] else [])
    col.set_controls(state["points"])  # fit
    terms, _ = col.loss_backward()
    return terms, col.control_grad()


def work(case):
    problems, _, _ = _inputs(case, 0)
    passes = case["iters"] if case["op"] == "step" else 1
    if case["op"] == "schedule":  # 6, 4, 2 and 1 parts of the iterations, a quarter of the pixels per coarser level
        passes = case["iters"] * (1 + 2 / 4 + 4 / 16 + 6 / 64)
    data = pairs = pixels = 0.0
    for p in problems:
        n, res = len(p["kind"]), p["grid"]
        m = 1.0 + case["pad"]
        off = p["pt_off"]
        r = np.maximum.reduceat(np.hypot(*p["pts"].reshape(-1, 2).T), off[:-1])
        segs = np.where(p["kind"] == 0, np.diff(off) // 3 * 16, np.diff(off))
        side = np.minimum(2 * (0.9 * r * res + m + p["hw"] * res), res)
        pairs += float((segs * side * side).sum())
        pixels += float(res) * res
        data += 8.0 * off[-1] + 4.0 * res * res  # outlines and the container raster
        data += {"step": 96.0, "host": 96.0, "schedule": 96.0}.get(case["op"], 32.0) * n
        data += {"render": 8.0, "mat_init": 8.0 if case["maps"] else 0.0}.get(case["op"], 0.0) * res * res
    if case["op"] == "mat_init":
        flops = 20.0 * pixels + 8.0 * sum(len(p["kind"]) * 3.0 * p["grid"] for p in problems)
    else:
        # 14 per pixel-segment pair of the outlines' boxes; composite, losses, distribution term
        flops = passes * (14.0 * pairs + (80.0 if case["uniform"] else 30.0) * pixels)
    return {"bytes": float(data), "flops": float(flops)}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------------
_CHUNK = 1 << 24  # pixel-segment pairs handled at once
_RHO = 1.0
_TAU = 0.5


def _smooth(x):
    x = x.clamp(-1.0, 1.0)
    return 0.25 * (1.0 + x) ** 2 * (2.0 - x)


def _dsmooth(x):
    x = x.clamp(-1.0, 1.0)
    return 0.75 * (1.0 - x * x)


def _f64(a):
    return torch.as_tensor(np.asarray(a, np.float64), device="cuda")


def _bernstein():
    t = torch.arange(16, device="cuda", dtype=torch.float64) / 16.0
    u = 1.0 - t
    return torch.stack([u ** 3, 3 * u * u * t, 3 * u * t * t, t ** 3], 1)  # [sample, point]


def _groups(prob):
    """Elements of like segment counts: (element ids, start points, end points, valid, closed)."""
    pts, off = prob["pts"].astype(np.float64).reshape(-1, 2), prob["pt_off"]
    b = _bernstein().cpu().numpy()
    verts = []
    for e, kind in enumerate(prob["kind"]):
        p = pts[off[e]:off[e + 1]]
        if kind == 0:
            c = np.arange(0, len(p), 3)
            four = np.stack([p[(c + i) % len(p)] for i in range(4)], 1)  # [curve, 4, 2]
            p = np.einsum("jr,crk->cjk", b, four).reshape(-1, 2)
        verts.append(p)
    segs = [len(v) - (1 if k == 2 else 0) for v, k in zip(verts, prob["kind"])]
    out, lo = [], 0
    for hi in (16, 64, 128, 256, 1024):
        ids = [e for e in range(len(verts)) if lo < segs[e] <= hi]
        lo = hi
        if not ids:
            continue
        s = max(segs[e] for e in ids)
        a, z, ok = np.zeros((len(ids), s, 2)), np.zeros((len(ids), s, 2)), np.zeros((len(ids), s), bool)
        for i, e in enumerate(ids):
            a[i, :segs[e]] = verts[e][:segs[e]]
            z[i, :segs[e]] = np.roll(verts[e], -1, 0)[:segs[e]]
            a[i, segs[e]:] = z[i, segs[e]:] = a[i, 0]
            ok[i, :segs[e]] = True
        out.append((torch.tensor(ids, device="cuda"), _f64(a), _f64(z), torch.tensor(ok, device="cuda"),
                    torch.tensor(prob["kind"][ids] != 2, device="cuda")))
    return out


def _nearest(dx, dy, ax, ay, bx, by):
    """Squared distance to the nearest of each row's segments, its index, and the winding number."""
    ex, ey = bx - ax, by - ay
    wx, wy = dx[:, None] - ax, dy[:, None] - ay
    ee = ex * ex + ey * ey
    t = torch.where(ee > 0, (wx * ex + wy * ey) / ee.clamp_min(1e-300), torch.zeros_like(ee)).clamp(0.0, 1.0)
    d2, idx = ((wx - t * ex) ** 2 + (wy - t * ey) ** 2).min(1)
    cross = ex * wy - ey * wx
    a_le, b_le = wy >= 0, dy[:, None] >= by
    wind = (a_le & ~b_le & (cross > 0)).sum(1) - (~a_le & b_le & (cross < 0)).sum(1)
    return d2, idx, wind


def _coverage(prob, res):
    ring, off = prob["ring_pts"].astype(np.float64).reshape(-1, 2) * res, prob["ring_off"]
    a = _f64(ring)
    b = _f64(np.concatenate([np.roll(ring[off[i]:off[i + 1]], -1, 0) for i in range(len(off) - 1)]))
    sd, step = [], max(1, _CHUNK // len(ring))
    for i in range(0, res * res, step):
        pix = torch.arange(i, min(i + step, res * res), device="cuda")
        d2, _, wind = _nearest(pix % res + 0.5, torch.div(pix, res, rounding_mode="floor") + 0.5,
                               a[None, :, 0], a[None, :, 1], b[None, :, 0], b[None, :, 1])
        sd.append(torch.where(wind != 0, d2.sqrt(), -d2.sqrt()))
    return _smooth(torch.cat(sd) / _RHO)


def _pairs(prob, groups, q, res, pad):
    """Every (element, pixel) pair within the coverage margin or inside: element, pixel, signed
    distance, position about the element's centre, closest segment (start, end, index)."""
    found = []
    hw = _f64(prob["hw"]) * res
    for ids, a, z, ok, closed in groups:
        t = q[ids]
        c, s, k = torch.cos(t[:, 2, None]), torch.sin(t[:, 2, None]), t[:, 3, None] * res
        turn = lambda v: torch.stack([k * (c * v[..., 0] - s * v[..., 1]), k * (s * v[..., 0] + c * v[..., 1])], -1)  # noqa: E731,B023
        a, z = turn(a), turn(z)
        centre = t[:, :2] * res
        width = torch.where(closed, torch.zeros_like(hw[ids]), hw[ids])
        margin = _RHO + pad + width
        both = torch.cat([a, z], 1)
        low = ((centre + both.amin(1) - margin[:, None] - 0.5).floor()).clamp(0, res).long()
        high = ((centre + both.amax(1) + margin[:, None] - 0.5).ceil()).clamp(-1, res - 1).long()
        wh = (high - low + 1).clamp_min(0)
        end = (wh[:, 0] * wh[:, 1]).cumsum(0)
        total, step = int(end[-1]), max(1, _CHUNK // a.shape[1])
        for i in range(0, total, step):
            at = torch.arange(i, min(i + step, total), device="cuda")
            e = torch.searchsorted(end, at, right=True)
            at = at - (end[e] - wh[e, 0] * wh[e, 1])
            x, y = low[e, 0] + at % wh[e, 0], low[e, 1] + torch.div(at, wh[e, 0], rounding_mode="floor")
            dx, dy = x + 0.5 - centre[e, 0], y + 0.5 - centre[e, 1]
            d2, j, wind = _nearest(dx, dy, a[e, :, 0], a[e, :, 1], z[e, :, 0], z[e, :, 1])
            dist = d2.sqrt()
            sd = torch.where(closed[e], torch.where(wind != 0, dist, -dist), width[e] - dist)
            keep = sd > -(_RHO + pad)
            e, j = e[keep], j[keep]
            found.append((ids[e], (y * res + x)[keep], sd[keep], dx[keep], dy[keep], a[e, j], z[e, j], j, closed[e]))
    return [torch.cat(f) for f in zip(*found)]


def _box(image, res, r):
    """Zero-padded box sums of side 2r + 1 from an integral image (exact for integers)."""
    ii = torch.zeros(res + 2 * r + 1, res + 2 * r + 1, dtype=image.dtype, device="cuda")
    ii[r + 1:r + 1 + res, r + 1:r + 1 + res] = image.view(res, res)
    ii = ii.cumsum(0).cumsum(1)
    w = 2 * r + 1
    return (ii[w:, w:] - ii[:-w, w:] - ii[w:, :-w] + ii[:-w, :-w]).reshape(-1)


def _uniform_term(occ, cov, res):
    loss, grad = torch.zeros((), dtype=torch.float64, device="cuda"), torch.zeros_like(occ)
    for k in range(4):
        r = 2 + 3 * k
        box = _box((occ * 2.0 ** 40).round().long(), res, r).double() * 2.0 ** -40
        rest = 1.0 - box.clamp_max(1.0)
        free = cov * (1.0 - occ)
        loss = loss + (k + 1) * (free * rest).sum()
        grad -= (k + 1) * (cov * rest + _box(torch.where(box < 1.0, free, torch.zeros_like(free)), res, r))
    return loss, grad


def _evaluate(prob, groups, q, res, o, cov):
    """Images, loss terms and gradient of one collage at the params q."""
    pad, n, npx = o["pad_px"], len(prob["kind"]), res * res
    e, pix, sd, dx, dy, a, z, seg, closed = _pairs(prob, groups, q, res, pad)
    ones = torch.ones(npx, dtype=torch.float64, device="cuda")
    keep = _smooth(-sd / _RHO)
    over = 1.0 - _TAU * _smooth((sd + pad) / _RHO)
    ihat = ones.scatter_reduce(0, pix, keep, "prod")
    prod = ones.scatter_reduce(0, pix, over, "prod")
    w = torch.where(cov >= 0.5, o["w_in"] * ones, o["w_out"] * ones)
    excess = 1.0 - prod - _TAU
    phi = 1.0 - (torch.div(torch.arange(npx, device="cuda"), res, rounding_mode="floor") + 0.5) / res
    diff = ihat - (1.0 - cov)
    terms = [(w * diff * diff).sum() / npx, excess.clamp_min(0.0).sum() / npx, 0.0 * diff[0],
             ((1.0 - ihat) * phi).sum() / npx]
    g_ihat = o["alpha"] / npx * 2.0 * w * diff - o["delta_down"] / npx * phi
    if o["gamma"] != 0.0:
        terms[2], g_occ = _uniform_term(1.0 - ihat, cov, res)
        g_ihat = g_ihat - o["gamma"] * g_occ
    terms.append(o["alpha"] * terms[0] + o["beta"] * terms[1] + o["gamma"] * terms[2] + o["delta_down"] * terms[3])
    # adjoint: coverage -> signed distance -> closest point -> transform
    g_over = torch.where(excess > 0, o["beta"] / npx * ones, 0.0 * ones)[pix]
    g_c = torch.where(keep > 0, -g_ihat[pix] * ihat[pix] / keep.clamp_min(1e-300), torch.zeros_like(keep))
    g_sd = (g_c * _dsmooth(sd / _RHO) + g_over * _TAU * prod[pix] / over * _dsmooth((sd + pad) / _RHO)) / _RHO
    d = z - a
    ee = (d * d).sum(1)
    u = torch.where(ee > 0, ((dx - a[:, 0]) * d[:, 0] + (dy - a[:, 1]) * d[:, 1]) / ee.clamp_min(1e-300), 0.0 * ee).clamp(0.0, 1.0)
    near = a + u[:, None] * d
    out = torch.stack([dx, dy], 1) - near
    dist = out.norm(dim=1)
    side = torch.where(d[:, 0] * (dy - a[:, 1]) - d[:, 1] * (dx - a[:, 0]) >= 0, 1.0, -1.0) / ee.clamp_min(1e-300).sqrt()
    inner = ((u > 0) & (u < 1))[:, None]
    normal = torch.where(inner, torch.stack([-d[:, 1] * side, d[:, 0] * side], 1), out / dist.clamp_min(1e-300)[:, None])
    g = -torch.where(closed & (sd > 0), 1.0, -1.0) * g_sd
    rows = torch.stack([g * normal[:, 0] * res, g * normal[:, 1] * res,
                        g * (normal[:, 1] * near[:, 0] - normal[:, 0] * near[:, 1]),
                        g * (normal * near).sum(1) / q[e, 3]], 1)
    grad = torch.zeros(n, 4, dtype=torch.float64, device="cuda").index_add(0, e, rows)
    return {"ihat": ihat, "atau": 1.0 - prod, "terms": torch.stack(terms), "grad": grad,
            "pairs": (e, pix, sd), "outline": (g[:, None] * normal, u, seg)}


def _point_gradient(prob, q, res, outline):
    """The gradient of the control points of a single closed cubic path (segment j ends at sample
    j + 1; a closest point moves with its segment's end points)."""
    push, u, seg = outline
    c, s, k = torch.cos(q[0, 2]), torch.sin(q[0, 2]), q[0, 3] * res
    local = k * torch.stack([c * push[:, 0] + s * push[:, 1], c * push[:, 1] - s * push[:, 0]], 1)
    nv = len(prob["pts"]) // 6 * 16
    verts = torch.zeros(nv, 2, dtype=torch.float64, device="cuda")
    verts = verts.index_add(0, seg, local * (1.0 - u)[:, None]).index_add(0, (seg + 1) % nv, local * u[:, None])
    each = torch.einsum("jr,cjk->crk", _bernstein(), verts.view(-1, 16, 2))  # [curve, 4, 2]
    out = each[:, :3].clone()
    out[:, 0] += each[:, 3].roll(1, 0)
    return out.reshape(-1, 2)


def _adam(q, m, v, g, t):
    m = 0.9 * m + 0.1 * g
    v = 0.999 * v + 0.001 * g * g
    q = q - 1e-2 / (1 - 0.9 ** t) * m / (v.sqrt() / math.sqrt(1 - 0.999 ** t) + 1e-8)
    return torch.cat([q[:, :3], q[:, 3:].clamp(0.05, 20.0)], 1), m, v


def _distance2(wall, border):
    """Exact squared distance of every pixel to the nearest wall pixel (with the border beyond the
    image a wall too, if asked); 2^40 where there is none."""
    res = wall.shape[0]
    far = 1 << 20
    rows = torch.arange(res, device="cuda")[:, None].expand(res, res)
    up = torch.where(wall, rows, torch.full_like(rows, -1 if border else -far)).cummax(0).values
    down = torch.where(wall, rows, torch.full_like(rows, res if border else far + res)).flip(0).cummin(0).values.flip(0)
    g = torch.minimum(rows - up, down - rows).clamp_max(far)
    cols = torch.arange(res, device="cuda")
    if border:
        g = torch.nn.functional.pad(g, (1, 1))
        cols = torch.arange(-1, res + 1, device="cuda")
    step2 = (torch.arange(res, device="cuda")[:, None] - cols[None]) ** 2
    g2 = g * g
    chunk = max(1, (_CHUNK * 2) // (res * res))
    return torch.cat([(step2[None] + g2[i:i + chunk, None]).amin(2) for i in range(0, res, chunk)])


def _metrics(prob, r, res, cov):
    e, pix, sd = r["pairs"]
    obj, shape = r["ihat"] <= 0.5, cov >= 0.5
    count = torch.zeros(res * res, dtype=torch.float64, device="cuda").index_add(0, pix, (sd >= 0).double())
    inside, total = int((obj & shape).sum()), int(shape.sum())
    over, outside = int((count >= 2).sum()), int((obj & ~shape).sum())
    d2 = _distance2(obj.view(res, res), False).reshape(-1)
    empty = shape & ~obj
    ratio = (lambda x: x / total) if total else (lambda x: 0.0)
    spread = float(d2[empty].sum()) / int(empty.sum()) / res ** 2 if int(obj.sum()) and int(empty.sum()) else 0.0
    return [inside, total, over, outside, ratio(inside), ratio(over), ratio(outside), spread]


def _axis(prob, res, cov):
    inside = (cov >= 0.5).view(res, res)
    d2 = _distance2(~inside, True)
    wide = torch.nn.functional.pad(d2, (1, 1, 1, 1))
    axis = torch.zeros_like(inside)
    for x, y in ((1, 0), (0, 1), (1, 1), (1, -1)):
        u = wide[1 + y:1 + y + res, 1 + x:1 + x + res]
        v = wide[1 - y:1 - y + res, 1 - x:1 - x + res]
        axis |= (d2 >= u) & (d2 >= v) & ((d2 > u) | (d2 > v))
    return (axis & inside).int().reshape(-1), d2.double().sqrt().reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op == "schedule":  # dozens of iterations: rounding grows along the way
        return None
    problems, m, v = _inputs(case, seed)
    o = dict(alpha=3e3, beta=8e4, gamma=5e-4, delta_down=0.0, w_in=1.0, w_out=100.0, pad_px=0.0)
    o.update({k: x for k, x in _options(case).items() if k in o})
    m, v = _f64(m), _f64(v)
    got, e0 = [], 0
    for prob in problems:
        n, res = len(prob["kind"]), prob["grid"]
        cov = _coverage(prob, res)
        if op == "mat_init":
            got.append(_axis(prob, res, cov))
            continue
        groups = _groups(prob)
        q = _f64(prob["params0"]).view(-1, 4)
        if op in ("step", "host"):
            mm, vv = m[e0:e0 + n], v[e0:e0 + n]
            for i in range(case["iters"] if op == "step" else 1):
                r = _evaluate(prob, groups, q, res, o, cov)
                q, mm, vv = _adam(q, mm, vv, r["grad"], _ADAM_STEP + 1 + i)
            got.append((q, r["terms"]))
        else:
            r = _evaluate(prob, groups, q, res, o, cov)
            if op == "metrics":
                got.append(_metrics(prob, r, res, cov))
            elif op == "fit":
                got.append((r["terms"], _point_gradient(prob, q, res, r["outline"])))
            elif op in ("autograd", "gradient"):
                got.append((r["terms"][4:] if op == "autograd" else r["terms"], r["grad"]))
            else:
                got.append((r["ihat"], r["atau"]))
        e0 += n
    if op == "metrics":
        return np.array(got, np.float64)
    first, second = torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    if op == "mat_init":
        return [None, first, second] if case["maps"] else [None]
    if op == "step":
        return first, second.view(-1, 5)
    if op == "host":
        return first.reshape(-1), second
    if op == "autograd":
        return first.sum(), second
    if op in ("fit", "gradient"):
        return first.view(-1, 5), second
    return first, second
