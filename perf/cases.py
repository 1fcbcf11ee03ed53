"""Performance cases of the sonar framework: what its users have it do.

A case is a dict of plain values.  `listed()` names a dozen that stand for the
work of a simulation, a survey rendering job, a parameter fit and the other
sensors of a vehicle; `draw(rng)` gives more of the same ranges.  `prepare`
makes what a program has in hand before the call, `run` is one pass through
the public entry points, `work` counts what the pass cannot do without, and
`exact` restates the method in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_01074_gb300 import scenes as S
from paper_2503_01074_gb300.autograd import sonar_render
from paper_2503_01074_gb300.sonar import DvlParams, RenderParams, Sonar

DEV = "cuda:0"
ALPHA, GAIN = 0.04, 1.5
DT = 0.05


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    seabed = {"cells": 1024, "extent": 100.0, "mats": 16, "piles": 48, "boxes": 24}
    sonar = {"beams": 512, "elev": 64, "bins": 1000, "az": 512, "hfov": 130.0, "vfov": 20.0, "r_max": 20.0,
             "fan_w": 1024, "fan_h": 576, "normalise": 1}
    return [
        # one tick of a small real-time simulation: a coarse sonar over a plane and
        # a sphere; the time is launches and latency
        {"name": "frame_tiny", "kind": "frame", "scene": "tiny", "beams": 128, "elev": 8, "bins": 256, "az": 128,
         "hfov": 60.0, "vfov": 12.0, "r_max": 10.0, "fan_w": 400, "fan_h": 300, "normalise": 1, "hits": False},
        # one tick of a full imaging sonar over a two-million-triangle seabed,
        # with the display fan and the hit records
        {"name": "frame_seabed", "kind": "frame", "scene": "seabed", **seabed, **sonar, "hits": True},
        # the paper's dense-ray render: 3000 x 460 rays into 350 x 220 bins
        {"name": "frame_dense", "kind": "frame", "scene": "seabed", **seabed, **sonar, "beams": 3000, "elev": 460,
         "bins": 350, "az": 220, "fan_w": 440, "fan_h": 248, "hits": False},
        # odd counts everywhere and whole-image normalisation: a sensor that nobody tuned for
        {"name": "frame_ragged", "kind": "frame", "scene": "seabed", "cells": 517, "extent": 60.0, "mats": 9,
         "piles": 11, "boxes": 7, "beams": 349, "elev": 47, "bins": 777, "az": 233, "hfov": 97.0, "vfov": 17.0,
         "r_max": 27.5, "fan_w": 701, "fan_h": 403, "normalise": 2, "hits": False},
        # one iteration of fitting absorption, gain and 64 reflectivities to a
        # measured image, through autograd
        {"name": "fit_seabed", "kind": "fit", **seabed, **sonar, "mats": 64},
        # rendering a trajectory with the gradient of a given image gradient: a
        # planned batch of 64 poses, forward and adjoint
        {"name": "train_batch", "kind": "batch", **seabed, **sonar, "frames": 64, "fan": True, "hits": True,
         "adjoint": True, "update": False},
        # a fleet of small sonars stepped together: new poses and frame numbers, then the images
        {"name": "fleet_batch", "kind": "batch", **seabed, **sonar, "cells": 512, "beams": 256, "elev": 32,
         "bins": 500, "az": 256, "fan_w": 512, "fan_h": 288, "frames": 32, "fan": True, "hits": False,
         "adjoint": False, "update": True},
        # a dataset job: 128 sensors of three types on four scenes, every geometry its own
        {"name": "mixed_batch", "kind": "mixed", "sensors": 128, "hits": False},
        # a large survey area: 33.6 million triangles, 1024 x 256 rays, 4000 range
        # bins, forward and adjoint with the hit records recomputed rather than kept
        {"name": "train_large", "kind": "batch", "cells": 4096, "extent": 400.0, "mats": 64, "piles": 1000,
         "boxes": 1000, **{**sonar, "beams": 1024, "elev": 256, "bins": 4000, "az": 1024, "r_max": 60.0,
                           "fan_w": 0, "fan_h": 0},
         "frames": 32, "fan": False, "hits": False, "adjoint": True, "update": False},
        # a map that changed: its mesh uploaded, one frame rendered, the mesh released
        {"name": "remap_seabed", "kind": "upload", **seabed, **{**sonar, "fan_w": 0, "fan_h": 0}},
        # velocity logs: 4096 vehicles x 256 steps of DVL beams and the ping schedule
        {"name": "dvl_log", "kind": "dvl", "cells": 512, "extent": 100.0, "vehicles": 4096, "steps": 256},
        # the underwater look of a short camera clip
        {"name": "camera_clip", "kind": "camera", "frames": 8, "height": 1080, "width": 1920},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_sonar(rng, max_rays, max_bins):
    """A sonar of a drawn size; beams per azimuth column one, fewer or many."""
    while True:
        beams, elev = _log_int(rng, 96, 1500), _log_int(rng, 8, 256)
        bins = _log_int(rng, 200, 4000)
        az = rng.choice([beams, beams, beams, max(48, beams // rng.choice([2, 3])), min(2 * beams, 1024)])
        if beams * elev <= max_rays and bins * az <= max_bins:
            break
    fan_w = rng.choice([2 * beams, _log_int(rng, 300, 1600)])
    return {"beams": beams, "elev": elev, "bins": bins, "az": az, "hfov": rng.uniform(50.0, 140.0),
            "vfov": rng.uniform(10.0, 24.0), "r_max": rng.uniform(8.0, 45.0), "fan_w": fan_w,
            "fan_h": (9 * fan_w) // 16, "normalise": rng.choice([1, 1, 1, 1, 2, 0])}


def _draw_scene(rng):
    return {"cells": _log_int(rng, 200, 1100), "extent": rng.uniform(60.0, 120.0), "mats": rng.choice([4, 16, 64]),
            "piles": rng.randint(0, 60), "boxes": rng.randint(0, 40)}


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "fit", "batch", "batch", "batch", "mixed", "upload", "dvl",
                       "camera"])
    if kind == "frame":
        return {"kind": "frame", "scene": "seabed", **_draw_scene(rng), **_draw_sonar(rng, 300_000, 4_000_000),
                "hits": rng.random() < 0.5}
    if kind == "fit":
        return {"kind": "fit", **_draw_scene(rng), **_draw_sonar(rng, 150_000, 2_000_000)}
    if kind == "batch":
        sonar = _draw_sonar(rng, 100_000, 1_000_000)
        most = min(96, 3_000_000 // (sonar["beams"] * sonar["elev"]), 60_000_000 // (sonar["bins"] * sonar["az"]))
        fan, adjoint = rng.random() < 0.7, rng.random() < 0.6
        return {"kind": "batch", **_draw_scene(rng), **sonar, "frames": _log_int(rng, 2, max(3, most)), "fan": fan,
                "hits": rng.random() < 0.5, "adjoint": adjoint, "update": rng.random() < 0.3}
    if kind == "mixed":
        return {"kind": "mixed", "sensors": _log_int(rng, 12, 128), "hits": rng.random() < 0.3}
    if kind == "upload":
        scene = _draw_scene(rng)
        return {"kind": "upload", **scene, "cells": _log_int(rng, 24, 1024),
                **{**_draw_sonar(rng, 40_000, 600_000), "fan_w": 0, "fan_h": 0}}
    if kind == "dvl":
        return {"kind": "dvl", "cells": _log_int(rng, 200, 1024), "extent": rng.uniform(60.0, 120.0),
                "vehicles": _log_int(rng, 1, 4000), "steps": _log_int(rng, 1, 256)}
    return {"kind": "camera", "frames": _log_int(rng, 1, 16), "height": _log_int(rng, 240, 1200),
            "width": _log_int(rng, 320, 1920)}


# ---------------------------------------------------------------------------
# inputs: scenes, sensors, poses
# ---------------------------------------------------------------------------

class _Terrain:
    """A value-noise fBm seabed over [-extent/2, extent/2]^2, evaluated on the GPU."""

    def __init__(self, extent, amplitude, rng):
        self.extent, self.amplitude = extent, amplitude
        self.lattices = [torch.tensor(rng.uniform(-1.0, 1.0, (4 * 2 ** o + 2, 4 * 2 ** o + 2)), device=DEV)
                         for o in range(6)]

    def __call__(self, x, y):
        x = torch.as_tensor(x, dtype=torch.float64, device=DEV)
        y = torch.as_tensor(y, dtype=torch.float64, device=DEV)
        u, w = x / self.extent + 0.5, y / self.extent + 0.5
        total, norm, amp = 0.0, 0.0, 1.0
        for o, lat in enumerate(self.lattices):
            n = 4 * 2 ** o
            fu, fw = (u * n).clamp(0.0, n - 1e-9), (w * n).clamp(0.0, n - 1e-9)
            iu, iw = fu.floor().long(), fw.floor().long()
            tu, tw = fu - iu, fw - iw
            su, sw = tu * tu * (3.0 - 2.0 * tu), tw * tw * (3.0 - 2.0 * tw)
            total = total + amp * ((lat[iu, iw] * (1 - su) + lat[iu + 1, iw] * su) * (1 - sw)
                                   + (lat[iu, iw + 1] * (1 - su) + lat[iu + 1, iw + 1] * su) * sw)
            norm += amp
            amp *= 0.5
        return self.amplitude * total / norm

    def numpy(self, x, y):
        return self(np.asarray(x, np.float64), np.asarray(y, np.float64)).cpu().numpy()


def _seabed(cells, extent, mats, piles, boxes, rng, amplitude=None):
    """Heightfield plus obstacles: (verts, tris, mat) CUDA tensors and the terrain."""
    terrain = _Terrain(extent, amplitude or (4.0 if extent > 200.0 else 2.0), rng)
    n = cells
    xs = (torch.arange(n + 1, dtype=torch.float64, device=DEV) / n - 0.5) * extent
    X, Y = torch.meshgrid(xs, xs, indexing="ij")
    verts = torch.stack([X, Y, terrain(X, Y)], -1).reshape(-1, 3).float()
    i, j = torch.meshgrid(torch.arange(n, device=DEV), torch.arange(n, device=DEV), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)
    a, b, c, d = i * (n + 1) + j, (i + 1) * (n + 1) + j, (i + 1) * (n + 1) + j + 1, i * (n + 1) + j + 1
    tris = torch.stack([a, b, c, a, c, d], -1).reshape(-1, 3).int()
    side = max(1, int(math.isqrt(mats)))
    mat = ((i * side // n) * side + j * side // n).int().repeat_interleave(2)
    if piles + boxes:
        half = extent / 2.0 - 5.0
        xy = rng.uniform(-half, half, (piles + boxes, 2))
        near = np.hypot(xy[:, 0], xy[:, 1]) < 6.0
        xy[near] += 12.0
        z = terrain.numpy(xy[:, 0], xy[:, 1])
        parts = [S.cylinder(tuple(xy[k]), float(z[k]) - 0.5, rng.uniform(0.3, 1.0), rng.uniform(3.0, 8.0), 16,
                            int(rng.integers(0, mats))) for k in range(piles)]
        parts += [S.box(tuple(xy[k]), float(z[k]) - 0.3, rng.uniform(0.5, 4.0, 3), rng.uniform(0, math.pi),
                        int(rng.integers(0, mats))) for k in range(piles, piles + boxes)]
        m = S.merge(parts)
        tris = torch.cat([tris, torch.tensor(m.tris, device=DEV) + verts.shape[0]])
        verts = torch.cat([verts, torch.tensor(m.verts, device=DEV)])
        mat = torch.cat([mat, torch.tensor(m.mat, device=DEV)])
    return (verts.contiguous(), tris.contiguous(), mat.contiguous()), terrain


def _scene(case, rng):
    """The case's mesh, reflectivities and terrain height."""
    if case.get("scene") == "tiny":
        mesh, mu = S.tiny_scene()
        t = tuple(torch.tensor(x, device=DEV) for x in (mesh.verts, mesh.tris, mesh.mat))
        return t, (mu * rng.uniform(0.8, 1.2, mu.shape)).astype(np.float32), None
    mesh, terrain = _seabed(case["cells"], case["extent"], case["mats"], case["piles"], case["boxes"], rng)
    return mesh, rng.uniform(0.1, 0.9, case["mats"]).astype(np.float32), terrain


def _sensors(case, terrain, rng, n):
    """n poses of the case's sonar: above the seabed, pitched down at it."""
    if terrain is None:
        xy, z, lo, hi = np.zeros((n, 2)), np.zeros(n), 35.0, 45.0
    else:
        r = rng.uniform(0.0, 0.3 * case["extent"], n) if n < 16 else np.full(n, 0.2 * case["extent"])
        a = rng.uniform(0.0, 2 * math.pi) + 2 * math.pi * np.arange(n) / n
        xy = np.stack([r * np.cos(a), r * np.sin(a)], -1)
        z = terrain.numpy(xy[:, 0], xy[:, 1]) + rng.uniform(3.0, 5.0)
        lo, hi = 22.0, 28.0
    out = []
    for k in range(n):
        yaw = rng.uniform(-0.05, 0.05) if terrain is None else 2 * math.pi * k / n + rng.uniform(-0.2, 0.2)
        out.append(S.SensorSpec(np.array([xy[k, 0], xy[k, 1], z[k]], np.float32),
                                S.pose_matrix(yaw, math.radians(rng.uniform(lo, hi))), case["beams"], case["elev"],
                                case["bins"], case["az"], math.radians(case["hfov"]), math.radians(case["vfov"]),
                                0.1, case["r_max"], case["fan_w"], case["fan_h"]))
    return out


def _mixed(case, rng):
    """Four seabeds and sensors of the three types in turn, on random poses with random fields of view."""
    scenes = [_seabed(g, 100.0, 16, 48, 24, rng) for g in (512, 640, 768, 1024)]
    items = []
    for k in range(case["sensors"]):
        si = int(rng.integers(0, 4))
        nb, ne, nr = S.SENSOR_TYPES[k % 3]
        x, y = rng.uniform(-35.0, 35.0, 2)
        z = float(scenes[si][1].numpy(x, y)) + rng.uniform(2.0, 6.0)
        spec = S.SensorSpec(np.array([x, y, z], np.float32),
                            S.pose_matrix(rng.uniform(0, 2 * math.pi), math.radians(rng.uniform(15.0, 35.0))),
                            nb, ne, nr, nb, math.radians(rng.uniform(60.0, 130.0)),
                            math.radians(rng.uniform(12.0, 20.0)), 0.1, rng.uniform(10.0, 40.0), 2 * nb,
                            (9 * 2 * nb) // 16)
        items.append((si, spec, int(rng.integers(0, 2 ** 31)), k))
    mu = rng.uniform(0.1, 0.9, 16).astype(np.float32)
    return [s[0] for s in scenes], mu, items


def _dvl_inputs(case, rng):
    mesh, terrain = _seabed(case["cells"], case["extent"], 16, 0, 0, rng)
    poses, vels = S.dvl_trajectories(terrain.numpy, case["vehicles"], case["steps"], DT, int(rng.integers(0, 2 ** 31)),
                                     extent=case["extent"])
    flat = [torch.tensor(x.reshape(-1, x.shape[-1]), device=DEV) for x in (poses, vels)]
    return mesh, flat[0], flat[1], int(rng.integers(0, 2 ** 31))


def _camera_inputs(case, rng):
    shape = (case["frames"], case["height"], case["width"])
    g = torch.Generator(device=DEV).manual_seed(int(rng.integers(0, 2 ** 31)))
    J = torch.rand((*shape, 3), generator=g, device=DEV)
    depth = 0.5 + 20.0 * torch.rand(shape, generator=g, device=DEV) ** 2
    sky = max(1, case["height"] // 12)
    depth[:, :sky] = math.inf   # rows above the horizon see no bottom
    coef = np.concatenate([rng.uniform(0.05, 0.6, 6), rng.uniform(0.0, 0.6, 3)])
    return J, depth, [float(np.float32(x)) for x in coef]


def _params(case):
    return RenderParams(normalise=case.get("normalise", 1))


def _frame_inputs(case, seed):
    """Mesh, reflectivities, the poses and their noise seeds, and a generator for what follows."""
    rng = np.random.default_rng(seed)
    mesh, mu, terrain = _scene(case, rng)
    specs = _sensors(case, terrain, rng, case.get("frames", 1))
    noise = int(rng.integers(0, 2 ** 31))
    g = torch.Generator(device=DEV).manual_seed(int(rng.integers(0, 2 ** 31)))
    return mesh, mu, specs, noise, g


def _grad_image(n, g):
    return torch.randn(n, generator=g, device=DEV) * 1e-3


def _target(case, g):
    return torch.rand((case["bins"], case["az"]), generator=g, device=DEV)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    son = Sonar(0)
    st = {"case": case, "son": son}
    if kind == "camera":
        st["J"], st["depth"], st["coef"] = _camera_inputs(case, np.random.default_rng(seed))
        return st
    if kind == "dvl":
        mesh, st["poses"], st["vel"], st["seed"] = _dvl_inputs(case, np.random.default_rng(seed))
        st["sid"] = son.upload(*mesh)
        st["params"] = DvlParams()
        return st
    st["params"] = _params(case)
    if kind == "mixed":
        meshes, mu, items = _mixed(case, np.random.default_rng(seed))
        sids = [son.upload(*m) for m in meshes]
        st["batch"] = son.batch([(sids[si], spec, s, f) for si, spec, s, f in items])
        st["theta"] = son.theta(ALPHA, GAIN, mu)
        return st
    mesh, mu, specs, noise, g = _frame_inputs(case, seed)
    st["theta"] = son.theta(ALPHA, GAIN, mu)
    st["seed"] = noise
    if kind == "upload":
        st["mesh"], st["spec"] = mesh, specs[0]
        return st
    st["sid"] = son.upload(*mesh)
    if kind == "batch":
        items = [(st["sid"], spec, noise, k) for k, spec in enumerate(specs)]
        if case["update"]:   # planned at an earlier tick; the pass brings the new poses
            st["items"] = items
            items = [(sid, spec.replace_pose(spec.pos + np.float32(0.05), spec.rot), s, f + 1000)
                     for sid, spec, s, f in items]
        st["batch"] = son.batch(items)
        if case["adjoint"]:
            st["grad"] = _grad_image(st["batch"].n_polar, g)
        return st
    st["spec"] = specs[0]
    if kind == "fit":
        st["target"] = _target(case, g)
        st["theta"].requires_grad_(True)
    return st


def run(st):
    case, son = st["case"], st["son"]
    kind = case["kind"]
    if kind == "frame":
        return son.render(st["sid"], st["spec"], st["theta"], st["params"], st["seed"], 7, hits=case["hits"])
    if kind == "fit":
        image = sonar_render(st["theta"], son, st["sid"], st["spec"], st["params"], st["seed"], 7)
        loss = torch.mean((image - st["target"]) ** 2)
        grad, = torch.autograd.grad(loss, st["theta"])
        return {"polar": image.detach(), "loss": loss.detach(), "dtheta": grad}
    if kind in ("batch", "mixed"):
        b = st["batch"]
        if case.get("update"):
            b.update(st["items"])
        fan = case.get("fan", True)
        b.render(st["theta"], st["params"], hits=case["hits"], fan=fan)
        out = {"polar": b.polar, "noised": b.noised}
        if case["hits"]:
            out["hits"] = b.hits
        if fan:
            out["fan"] = b.fan
        if case.get("adjoint"):
            out["dtheta"] = b.backward(st["theta"], st["params"], st["grad"], hits=case["hits"])
        return out
    if kind == "upload":
        sid = son.upload(*st["mesh"])
        out = son.render(sid, st["spec"], st["theta"], st["params"], st["seed"], 7)
        son.release(sid)
        return out
    if kind == "dvl":
        out = son.dvl(st["sid"], st["poses"], st["vel"], st["params"], st["seed"])
        out["emit"] = son.dvl_schedule(out["period"].view(case["vehicles"], case["steps"]), DT)
        return out
    return son.uw_image(st["J"], st["depth"], st["coef"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

# one closest-hit query of a ray: four box tests (24 operations) a level of a
# 4-wide hierarchy and one triangle test
def _ray_flops(tris):
    return 96.0 * max(1.0, math.log(max(tris, 4), 4)) + 60.0


def _tri_count(case):
    if case.get("scene") == "tiny":
        return 1282
    return 2 * case["cells"] ** 2 + 64 * case.get("piles", 0) + 12 * case.get("boxes", 0)


def _render_work(rays, bins, pixels, tris, hits):
    # noised and normalised image, fan, hit records, and a triangle for every ray (once each);
    # per bin a quarter of a 40-multiply random block, a logarithm and a root; per pixel the
    # polar coordinates and four taps
    return {"bytes": 8 * bins + 4 * pixels + (16 * rays if hits else 0) + 48 * min(rays, tris),
            "flops": rays * _ray_flops(tris) + 50 * bins + 60 * pixels}


def work(case):
    kind = case["kind"]
    if kind == "camera":
        n = case["frames"] * case["height"] * case["width"]
        return {"bytes": 28 * n, "flops": 30 * n}
    tris = 2_100_000 if kind == "mixed" else _tri_count(case)
    if kind == "dvl":
        n = case["vehicles"] * case["steps"]
        return {"bytes": (60 + 36 + 4) * n + 48 * min(4 * n, tris), "flops": 4 * n * _ray_flops(tris) + 300 * n}
    if kind == "mixed":   # the mean of the three sensor types
        n = case["sensors"]
        rays, bins = n * 57_344, n * 896_000
        return _render_work(rays, bins, n * 1_032_192, 4 * tris, case["hits"])
    n = case.get("frames", 1)
    rays, bins = n * case["beams"] * case["elev"], n * case["bins"] * case["az"]
    fan = case["fan_w"] * case["fan_h"] if kind == "frame" or (kind == "batch" and case["fan"]) else 0
    w = _render_work(rays, bins, n * fan, tris, case.get("hits", False))
    if kind == "fit" or case.get("adjoint"):
        # the gradient image, and the gradient of every ray's score
        w = {"bytes": w["bytes"] + 4 * bins, "flops": w["flops"] + 4 * bins + 150 * rays}
    if kind == "upload":
        # vertices, indices and materials read; triangles and a box for every second one written
        w = {"bytes": w["bytes"] + (6 + 12 + 4) * tris + (52 + 16) * tris, "flops": w["flops"] + 100 * tris}
    return w


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------

class _Grid:
    """Triangles binned by their (x, y) boxes into square cells, for exact ray queries."""

    def __init__(self, mesh):
        verts, tris, mat = mesh
        v = verts.double()[tris.long()]
        self.v0, self.e1, self.e2 = v[:, 0], v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
        self.n = torch.linalg.cross(self.e1, self.e2)
        self.mat = mat.long()
        lo, hi = v.amin(1)[:, :2], v.amax(1)[:, :2]
        self.org = lo.amin(0)
        size = float((hi.amax(0) - self.org).amax())
        self.m = m = max(8, min(4096, int(math.isqrt(max(1, tris.shape[0] // 2)))))
        self.h = size / m
        pad = 1e-7 * size
        c0 = ((lo - self.org - pad) / self.h).floor().long().clamp(0, m - 1)
        c1 = ((hi - self.org + pad) / self.h).floor().long().clamp(0, m - 1)
        cnt = (c1 - c0 + 1).prod(1)
        tri = torch.repeat_interleave(torch.arange(len(cnt), device=DEV), cnt)
        k = torch.arange(len(tri), device=DEV) - (cnt.cumsum(0) - cnt)[tri]
        w = (c1 - c0 + 1)[tri, 1]
        cell = (c0[tri, 0] + k // w) * m + c0[tri, 1] + k % w
        order = cell.argsort()
        self.tri = tri[order]
        self.count = torch.bincount(cell, minlength=m * m)
        self.start = self.count.cumsum(0) - self.count

    def _test(self, f, o, d):
        p = torch.linalg.cross(d, self.e2[f])
        det = (self.e1[f] * p).sum(1)
        s = o - self.v0[f]
        q = torch.linalg.cross(s, self.e1[f])
        u, v, t = (s * p).sum(1) / det, (d * q).sum(1) / det, (self.e2[f] * q).sum(1) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        return torch.where(ok, t, math.inf)

    def closest(self, o, d, tmax):
        """Nearest hit of each ray nearer than tmax: (t, triangle or -1)."""
        parts = [self._march(o[k:k + 2_000_000], d[k:k + 2_000_000], tmax[k:k + 2_000_000])
                 for k in range(0, len(o), 2_000_000)]
        return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])

    def _march(self, o, d, tmax):
        best = tmax.clone()
        hit = torch.full((len(o),), -1, dtype=torch.long, device=DEV)
        dxy = torch.where(d[:, :2].abs() < 1e-300, 1e-300, d[:, :2])
        inv = 1.0 / dxy
        ta, tb = (self.org - o[:, :2]) * inv, (self.org + self.m * self.h - o[:, :2]) * inv
        t_in = torch.minimum(ta, tb).amax(1).clamp(min=0.0)
        t_out = torch.maximum(ta, tb).amin(1)
        ray = torch.nonzero(t_in <= t_out)[:, 0]
        at = o[ray, :2] + t_in[ray, None] * d[ray, :2]
        c = ((at - self.org) / self.h).floor().long().clamp(0, self.m - 1)
        step = torch.where(dxy > 0, 1, -1)[ray]
        edge = self.org + (c + (step > 0)) * self.h
        tn = (edge - o[ray, :2]) * inv[ray]
        dt = (self.h * inv.abs())[ray]
        while len(ray):
            cell = c[:, 0] * self.m + c[:, 1]
            cnt, first = self.count[cell], self.start[cell]
            k = 0
            live = torch.nonzero(cnt > 0)[:, 0]
            while len(live):
                r, f = ray[live], self.tri[first[live] + k]
                t = self._test(f, o[r], d[r])
                near = t < best[r]
                best[r] = torch.where(near, t, best[r])
                hit[r] = torch.where(near, f, hit[r])
                k += 1
                live = live[cnt[live] > k]
            nxt = tn.amin(1)
            ax = (tn[:, 1] < tn[:, 0]).long()
            ar = torch.arange(len(ray), device=DEV)
            c[ar, ax] += step[ar, ax]
            tn[ar, ax] += dt[ar, ax]
            keep = (best[ray] > nxt) & (c >= 0).all(1) & (c < self.m).all(1)
            ray, c, step, tn, dt = ray[keep], c[keep], step[keep], tn[keep], dt[keep]
        return best, hit


def _philox(c, key):
    """Philox4x32-10 of int64 counter words c[0..3] under a 64-bit key."""
    m = 0xFFFFFFFF
    k0, k1 = key & m, key >> 32
    x = [torch.as_tensor(w, dtype=torch.int64, device=DEV) for w in c]
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((p1 >> 32) & m) ^ x[1] ^ k0, p1 & m, ((p0 >> 32) & m) ^ x[3] ^ k1, p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return x


def _uniform(w):
    return (w.double() + 1.0) / 2.0 ** 32


def _f32(x):
    return float(np.float32(x))


def _rays(spec):
    h, v = _f32(spec.hfov), _f32(spec.vfov)
    phi = -h / 2 + (torch.arange(spec.n_beams, dtype=torch.float64, device=DEV) + 0.5) * h / spec.n_beams
    th = -v / 2 + (torch.arange(spec.n_elev, dtype=torch.float64, device=DEV) + 0.5) * v / spec.n_elev
    phi, th = torch.meshgrid(phi, th, indexing="ij")
    ds = torch.stack([phi.sin() * th.cos(), phi.cos() * th.cos(), th.sin()], -1).reshape(-1, 3)
    d = ds @ torch.tensor(np.asarray(spec.rot, np.float64), device=DEV).T
    d = d / d.norm(dim=1, keepdim=True)
    return torch.tensor(np.asarray(spec.pos, np.float64), device=DEV).expand_as(d), d


def _image(spec, grid, d, t, hit, theta, normalise, seed, frame, prm):
    """(noised, normalised) image of one frame from its hits, differentiable in theta."""
    nr, naz = spec.n_range_bins, spec.n_az_bins
    rmin, rmax, hf = _f32(spec.r_min), _f32(spec.r_max), _f32(spec.hfov)
    ok = torch.nonzero((hit >= 0) & (t >= rmin) & (t < rmax))[:, 0]
    f, r = hit[ok], t[ok]
    cos = ((d[ok] * grid.n[f]).sum(1) / grid.n[f].norm(dim=1)).abs()
    score = theta[2 + grid.mat[f]] * cos * torch.exp(-2.0 * theta[0] * r) * theta[1]
    row = ((r - rmin) * (nr / (rmax - rmin))).floor().long().clamp(max=nr - 1)
    az = ((2 * (ok // spec.n_elev) + 1) * naz) // (2 * spec.n_beams)
    P = torch.zeros(nr * naz, dtype=torch.float64, device=DEV).index_add(0, row * naz + az, score)
    b = torch.arange(nr * naz, device=DEV)
    words = torch.stack(_philox([torch.arange((nr * naz + 3) // 4, device=DEV), frame, 1, 0], seed), -1)
    w_sa = prm.sigma_sa * torch.sqrt(-2.0 * torch.log(_uniform(words.reshape(-1)[:nr * naz])))
    x = _philox([b, frame, 0, 0], seed)
    w_sm = prm.sigma_sm * torch.sqrt(-2.0 * torch.log(_uniform(x[1]))) * torch.cos(2 * math.pi * _uniform(x[2]))
    rc = rmin + (b // naz + 0.5) * ((rmax - rmin) / nr)
    pc = -hf / 2 + (b % naz + 0.5) * (hf / naz)
    noised = (P * (0.5 + w_sm) + (rc / rmax) ** 2 * (1.0 + 0.5 * torch.exp(-pc * pc / prm.sigma_phi) * w_sa))
    noised = noised.reshape(nr, naz)
    if normalise == 0:
        return noised, noised
    top = noised.amax(1, keepdim=True) if normalise == 1 else noised.amax()
    return noised, noised / torch.where(top > 0, top, 1.0)


def _fan(spec, N):
    w, h, nr, naz = spec.fan_w, spec.fan_h, spec.n_range_bins, spec.n_az_bins
    rmin, rmax, hf = _f32(spec.r_min), _f32(spec.r_max), _f32(spec.hfov)
    scale = min(w / (2.0 * rmax * math.sin(hf / 2)), h / rmax)
    v, u = torch.meshgrid(torch.arange(h, dtype=torch.float64, device=DEV),
                          torch.arange(w, dtype=torch.float64, device=DEV), indexing="ij")
    x, y = (u + 0.5 - 0.5 * w) / scale, (h - v - 0.5) / scale
    r, phi = torch.hypot(x, y), torch.atan2(x, y)
    fr, fa = (r - rmin) * nr / (rmax - rmin) - 0.5, (phi + hf / 2) * naz / hf - 0.5
    i0, j0 = fr.floor(), fa.floor()
    wr, wa = fr - i0, fa - j0
    ia, ib = i0.long().clamp(0, nr - 1), (i0.long() + 1).clamp(0, nr - 1)
    ja, jb = j0.long().clamp(0, naz - 1), (j0.long() + 1).clamp(0, naz - 1)
    val = (1 - wr) * ((1 - wa) * N[ia, ja] + wa * N[ia, jb]) + wr * ((1 - wa) * N[ib, ja] + wa * N[ib, jb])
    return torch.where((r >= rmin) & (r <= rmax) & (phi.abs() <= hf / 2), val, 0.0)


def _theta(mu):
    return torch.cat([torch.tensor([_f32(ALPHA), _f32(GAIN)], dtype=torch.float64),
                      torch.tensor(mu, dtype=torch.float64)]).to(DEV)


def exact(case, seed):
    kind = case["kind"]
    if kind == "camera":
        J, depth, coef = _camera_inputs(case, np.random.default_rng(seed))
        k = torch.tensor(coef, dtype=torch.float64, device=DEV)
        d = depth.double()[..., None]
        return J.double() * torch.exp(-k[:3] * d) + k[6:] * (1.0 - torch.exp(-k[3:6] * d))
    if kind == "dvl":
        return _exact_dvl(case, seed)
    prm = _params(case)
    if kind == "mixed":
        meshes, mu, items = _mixed(case, np.random.default_rng(seed))
    else:
        mesh, mu, specs, noise, g = _frame_inputs(case, seed)
        first = 0 if kind == "batch" else 7
        meshes, items = [mesh], [(0, spec, noise, first + k) for k, spec in enumerate(specs)]
    theta = _theta(mu)
    hits = [None] * len(items)
    grids = [_Grid(m) for m in meshes]
    for si, grid in enumerate(grids):
        mine = [k for k, it in enumerate(items) if it[0] == si]
        for k0 in range(0, len(mine), 16):
            part = mine[k0:k0 + 16]
            rays = [_rays(items[k][1]) for k in part]
            if not rays:
                continue
            tmax = torch.cat([torch.full((len(r[0]),), _f32(items[k][1].r_max), dtype=torch.float64, device=DEV)
                              for k, r in zip(part, rays)])
            t, f = grid.closest(torch.cat([r[0] for r in rays]), torch.cat([r[1] for r in rays]), tmax)
            at = 0
            for k, r in zip(part, rays):
                hits[k] = (r[1], t[at:at + len(r[0])], f[at:at + len(r[0])])
                at += len(r[0])
    if kind == "fit":
        theta.requires_grad_(True)
        _, N = _image(specs[0], grids[0], *hits[0], theta, prm.normalise, noise, 7, prm)
        loss = torch.mean((N - _target(case, g).double()) ** 2)
        grad, = torch.autograd.grad(loss, theta)
        return {"polar": N.detach(), "loss": loss.detach(), "dtheta": grad}
    adjoint = bool(case.get("adjoint"))
    G, at, dtheta = None, 0, torch.zeros_like(theta)
    if adjoint:
        G = _grad_image(sum(it[1].n_range_bins * it[1].n_az_bins for it in items), g)
        theta.requires_grad_(True)
    fan_on = case.get("fan", True) and any(it[1].fan_w for it in items)
    polar, noised, fans = [], [], []
    for k, (si, spec, s, f) in enumerate(items):
        In, N = _image(spec, grids[si], *hits[k], theta, prm.normalise, s, f, prm)
        if adjoint:
            n = N.numel()
            dtheta += torch.autograd.grad((N.reshape(-1) * G[at:at + n].double()).sum(), theta)[0]
            at += n
        polar.append(N.detach())
        noised.append(In.detach())
        if fan_on:
            fans.append(_fan(spec, polar[-1]))
        hits[k] = None
    single = kind in ("frame", "upload")

    def pack(xs):
        return xs[0] if single else torch.cat([x.reshape(-1) for x in xs])
    out = {"polar": pack(polar), "noised": pack(noised)}
    if case.get("hits"):
        out["hits"] = None
    if fan_on:
        out["fan"] = pack(fans)
    if adjoint:
        out["dtheta"] = dtheta
    return out


def _exact_dvl(case, seed):
    mesh, poses, vel, key = _dvl_inputs(case, np.random.default_rng(seed))
    p = DvlParams()
    grid = _Grid(mesh)
    n = len(poses)
    q = poses.double()
    R, o = q[:, 3:].reshape(n, 3, 3), q[:, :3]
    tilt = _f32(p.tilt)
    beams = torch.tensor([[_f32(math.sin(tilt) * math.cos(a)), _f32(math.sin(tilt) * math.sin(a)),
                           _f32(-math.cos(tilt))] for a in (math.pi / 4 + k * math.pi / 2 for k in range(4))],
                         dtype=torch.float64, device=DEV)
    d = torch.einsum("nij,kj->nki", R, beams).reshape(-1, 3)
    t, f = grid.closest(o.repeat_interleave(4, 0), d, torch.full((4 * n,), math.inf, dtype=torch.float64, device=DEV))
    ranges = torch.where(f >= 0, t, math.inf).reshape(n, 4)
    valid = (ranges >= _f32(p.r_min)) & (ranges <= _f32(p.r_max))
    vs = torch.einsum("nij,ni->nj", R, vel.double())
    idx = torch.arange(n, device=DEV)
    w = []
    for half in range(2):
        x = _philox([idx, 0, 2, half], key)
        for a, b in ((x[0], x[1]), (x[2], x[3])):
            w.append(torch.sqrt(-2.0 * torch.log(_uniform(a))) * torch.cos(2 * math.pi * _uniform(b)))
    u = vs @ beams.T + _f32(p.sigma_b) * torch.stack(w, -1)
    m = valid.double()
    A = torch.einsum("nk,ki,kj->nij", m, beams, beams)
    y = torch.einsum("nk,ki->ni", m * u, beams)
    fit = valid.sum(1) >= p.min_beams
    A[~fit] = torch.eye(3, dtype=torch.float64, device=DEV)
    v = torch.where(fit[:, None], torch.linalg.solve(A, y[..., None])[..., 0], 0.0)
    far = torch.where(valid, ranges, 0.0).amax(1)
    period = torch.where(fit, _f32(p.t0) + _f32(p.t1) * far, _f32(p.t_lost))
    return {"ranges": ranges, "vel": v, "flags": None, "period": period, "emit": None}
