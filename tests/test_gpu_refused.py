"""A frame that no launch can take (its columns do not fit a block's shared memory) is
refused, and only that call: the next one of any kind is not told of it again.
"""
import math

import numpy as np
import pytest

from paper_2503_01074_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar, SonarError  # noqa: E402


def spec(nb, ne, nr, naz):
    return S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(40.0)), nb, ne, nr, naz,
                        math.radians(70.0), math.radians(25.0), 0.5, 10.0)


@pytest.mark.parametrize("next_call", ["render", "batch", "step", "upload", "dvl", "image", "philox"])
@pytest.mark.parametrize("how", ["render", "batch", "step"])
def test_the_call_after_a_refused_frame(how, next_call):
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    sid, prm = son.upload_mesh(mesh), RenderParams()
    theta = son.theta(0.05, 1.0, mu)
    grad = torch.ones(60000, device=son.device)

    def run(kind, sp):
        if kind == "render":
            son.render(sid, sp, theta, prm, 1, 2)
        elif kind in ("batch", "step"):
            b = son.batch([(sid, sp, 1, 2)])
            try:
                b.render(theta, prm) if kind == "batch" else b.step(theta, prm, grad)
            finally:
                b.close()
        elif kind == "upload":
            son.release(son.upload_mesh(mesh))
        elif kind == "dvl":
            poses = torch.tensor([[0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0]], device=son.device)
            son.dvl(sid, poses, torch.zeros(1, 3, device=son.device))
        elif kind == "image":
            son.uw_image(torch.rand(4, 4, 3, device=son.device), torch.rand(4, 4, device=son.device), [0.1] * 9)
        else:
            son.philox(torch.zeros(4, 4, dtype=torch.int32, device=son.device), 1)

    run("render", spec(16, 8, 100, 16))
    with pytest.raises(SonarError):
        run(how, spec(1, 30000, 60000, 1))
    run(next_call, spec(17, 9, 100, 17))
    torch.cuda.synchronize()
    st, bits = son.check()
    assert st == 0 and bits == 0
    son.close()
