"""Rays at the edges of a small object a long way off, beside one coarse quad.  The
boxes of the hierarchy are padded for the rounding of the ray that walks them (some
1e-7 of the range); the padding follows the scene's size, which here only the
vertices of the quad tell: its two triangles have one box centre, at the object.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2503_01074_gb300 import scenes as S

from tests._parity import hit_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar, hits_numpy  # noqa: E402


N_SLATS, BEAMS, ELEV = 480, 600_000, 8


def scene():
    """A 2 km quad and, at its middle, 480 upright slats 1 mm wide and 0.6 m high."""
    x = 0.0012247 * (np.arange(N_SLATS) - 0.5 * (N_SLATS - 1))   # no multiple of the rays' spacing
    corners = np.array([[-0.0005, 0.0, -0.3], [0.0005, 0.0, -0.3], [0.0005, 0.0, 0.3], [-0.0005, 0.0, 0.3]])
    v = (corners[None] + np.stack([x, 0.0 * x, 0.0 * x], -1)[:, None, :]).reshape(-1, 3).astype(np.float32)
    t = (np.array([[0, 1, 2], [0, 2, 3]])[None] + 4 * np.arange(N_SLATS)[:, None, None]).reshape(-1, 3).astype(np.int32)
    return S.merge([S.quad(-0.31, 1000.0, 0), S.Mesh(v, t, np.ones(len(t), np.int32))])


def sensor(dist):
    """The slats at 0.9 rad off the axis and straight along y: the x of such a ray is
    a difference of two large products, wrong by 1e-7 and nearly zero."""
    return S.SensorSpec(np.array([0.0, -dist, 0.0], np.float32), S.pose_matrix(0.9), BEAMS, ELEV, 100, 64, 2.0,
                        0.4 / dist, 1.0, 2.0 * dist)


def rays_at_the_slats(dist):
    """Indices of the beams within 0.35 m of the slats' middle, every elevation."""
    i = np.arange(BEAMS)
    near = np.abs(((i + 0.5) / BEAMS - 0.5) * 2.0 - 0.9) < 0.35 / dist
    return (i[near][:, None] * ELEV + np.arange(ELEV)[None]).ravel()


@pytest.mark.parametrize("dist", [300.0, 500.0, 900.0])
def test_no_hit_is_culled_at_long_range(dist):
    son = Sonar(0)
    mesh, sp, mu, ids = scene(), sensor(dist), np.array([0.5, 0.7], np.float32), rays_at_the_slats(dist)
    sid = son.upload_mesh(mesh)
    out = son.render(sid, sp, son.theta(0.01, 1.0, mu), RenderParams(), 1, 2, hits=True, fan=False)
    torch.cuda.synchronize()
    ref = O.render(mesh, mu, 0.01, 1.0, sp, O.Params(), seed=1, frame=2, ray_ids=ids)
    assert (ref["hits"]["tri"] >= 2).sum() > 400
    hit_parity(ref, hits_numpy(out["hits"]), ids)
    son.release(sid)
    son.close()
