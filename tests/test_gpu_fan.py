"""The batched fan at the edges of its tiling (squares of 64 pixels, two rows and
two frames at a time per thread): frames that share a coordinate table, one that
does not, odd numbers of frames, and fans of one pixel, one square, a little less
and a little more.  Every fan equals the single render's, bit for bit, since the
table holds what the single render computes and both blend with the same
roundings.  And a single render captured in a CUDA graph by its caller, where the
launches wait for one another in full, equals a plain one.
"""
import math

import pytest

from paper_2503_01074_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar  # noqa: E402


@pytest.fixture(scope="module")
def env():
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    yield son, son.upload_mesh(mesh), son.theta(0.05, 1.0, mu)
    son.close()


def frames(sid, w, h, n):
    base = S.sensor_tiny(40.0)
    base.fan_w, base.fan_h = w, h
    return [(sid, base.replace_pose((0.2 * k, 0.1 * k, 0.0), S.pose_matrix(0.05 * k, math.radians(40.0))), 5, k)
            for k in range(n)]


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("w,h", [(1, 1), (64, 4), (63, 9), (65, 64), (64, 65), (130, 131), (701, 403)])
def test_batched_fan_equals_single(env, w, h, n):
    son, sid, theta = env
    items = frames(sid, w, h, n)
    b = son.batch(items)
    for moved in (False, True):
        if moved:   # the last frame leaves the shared table
            s, spec, seed, frame = items[-1]
            spec = spec.replace_pose(spec.pos, spec.rot)
            spec.hfov *= 0.8
            items[-1] = (s, spec, seed, frame)
            b.update(items)
        b.render(theta, RenderParams(), fan=True)
        torch.cuda.synchronize()
        for k, (s, spec, seed, frame) in enumerate(items):
            one = son.render(s, spec, theta, RenderParams(), seed, frame, fan=True)
            assert torch.equal(one["fan"], b.view(k)["fan"]), (moved, k)
    b.close()


@pytest.mark.parametrize("mode", [1, 2])
def test_captured_single_render_equals_plain(env, mode):
    son, sid, theta = env
    (_, spec, seed, frame), = frames(sid, 200, 150, 1)
    prm = RenderParams(normalise=mode)
    plain = son.render(sid, spec, theta, prm, seed, frame, hits=True, fan=True)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = son.render(sid, spec, theta, prm, seed, frame, hits=True, fan=True)
    for rep in range(2):
        for v in out.values():
            v.zero_()
        g.replay()
        torch.cuda.synchronize()
        for key, v in plain.items():
            assert torch.equal(v, out[key]), (rep, key)
    # calls one after another, each starting while the one before it ends
    for rep in range(5):
        again = son.render(sid, spec, theta, prm, seed, frame, hits=True, fan=True)
    torch.cuda.synchronize()
    for key, v in plain.items():
        assert torch.equal(v, again[key]), key
