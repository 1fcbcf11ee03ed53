"""Updates of a planned batch that change what its captured launches rest on."""
import math

import numpy as np
import pytest

from paper_2503_01074_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar  # noqa: E402

MU = np.array([0.2, 0.5, 0.7, 0.9], np.float32)


@pytest.fixture()
def son():
    s = Sonar(0)
    yield s
    s.close()


def frames(sid, n, spec=None):
    base = spec or S.sensor_tiny(40.0)
    return [(sid, base.replace_pose((0.2 * k, 0.1 * k, 0.0), S.pose_matrix(0.05 * k, math.radians(40.0))), 5, k)
            for k in range(n)]


def step(b, theta, prm, grad):
    d = b.step(theta, prm, grad).clone()
    torch.cuda.synchronize()
    return [d] + [t.clone() for t in (b.polar, b.noised, b.hits, b.fan)]


def test_step_after_an_update_to_a_scene_uploaded_since(son):
    """The scene table moves when an item goes to a scene that the plan did not know:
    every captured graph, the combined step's among them, must follow."""
    theta, prm = son.theta(0.05, 1.0, MU), RenderParams()
    first = son.upload_mesh(S.tiny_scene()[0])
    b = son.batch(frames(first, 3))
    grad = torch.randn(b.n_polar, generator=torch.Generator().manual_seed(2)).to(son.device)
    step(b, theta, prm, grad)
    b.render(theta, prm)
    b.backward(theta, prm, grad)
    for seed in (3, 4):
        sid = son.upload_mesh(S.random_soup(300, seed))
        items = frames(sid, 3)
        b.update(items)
        got = step(b, theta, prm, grad)
        fresh = son.batch(items)
        want = step(fresh, theta, prm, grad)
        assert all(torch.equal(x, y) for x, y in zip(got, want))
        b.render(theta, prm)
        assert torch.equal(b.backward(theta, prm, grad), want[0])
        fresh.close()
    b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0
