"""The ray cast with several lanes per ray (launches of up to 20 tiles of 32 rays
per SM) against one lane per ray: a closest hit does not depend on how the
boxes are visited, so the hit records are the same, bit for bit.  The same poses
are cast alone (eight or four lanes by the frame's size) and inside a batch too
large for that, pinned to each one-lane variant by a tuning row.
"""
import math

import numpy as np
import pytest

from paper_2503_01074_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar  # noqa: E402

CAP, WIDE = 8, 16


@pytest.fixture(scope="module")
def son():
    s = Sonar(0)
    yield s
    s.close()


def one_triangle():
    v = np.array([[-3.0, 4.0, -3.0], [3.0, 4.0, -3.0], [0.0, 5.0, 2.0]], np.float32)
    return S.Mesh(v, np.array([[0, 1, 2]], np.int32), np.zeros(1, np.int32))


def scene(name):
    if name == "tri":
        return one_triangle()
    if name == "empty":
        return S.Mesh(np.zeros((0, 3), np.float32), np.zeros((0, 3), np.int32), np.zeros(0, np.int32))
    if name == "tiny":
        return S.tiny_scene()[0]
    return S.random_soup(int(name), 9)


# beams x elevations: 5 and 37 x 11 rays (eight lanes, ragged tiles), 300 x 90 (four
# lanes); `copies` frames put the batch beyond 20 tiles per SM
@pytest.mark.parametrize("name", ["empty", "tri", "tiny", "400", "30000"])
@pytest.mark.parametrize("nb,ne,copies", [(5, 1, 3300), (37, 11, 330), (300, 90, 6)])
def test_lanes_per_ray_give_the_same_records(son, name, nb, ne, copies):
    sid = son.upload_mesh(scene(name))
    mu = np.array([0.2, 0.5, 0.7, 0.9], np.float32)
    theta = son.theta(0.03, 1.7, mu)
    base = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.05, math.radians(25)), nb, ne, 64, nb,
                        math.radians(90.0), math.radians(40.0), 0.5, 20.0)
    specs = [base, base.replace_pose((0.3, -0.2, 0.1), S.pose_matrix(-0.4, math.radians(-20)))]
    for prm in (RenderParams(), RenderParams(two_sided=0, clip_tmax=0)):
        alone = [son.render(sid, s, theta, prm, 1, 2, hits=True)["hits"].clone() for s in specs]
        for v in (0, CAP, WIDE, CAP | WIDE):
            son.tune_set([[nb, ne, 64, nb, 1, 8, 128, v]])
            b = son.batch([(sid, specs[k % 2], 1, 2) for k in range(copies)])
            b.render(theta, prm, hits=True, fan=False)
            torch.cuda.synchronize()
            for k in (0, 1, copies - 1):
                assert torch.equal(b.view(k)["hits"], alone[k % 2]), (v, k)
            b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0
    son.release(sid)
