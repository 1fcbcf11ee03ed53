"""The row kernel (noise, range-wise normalisation) in launches that its widest
sensor alone does not describe.
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


@pytest.fixture(scope="module")
def env():
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    yield son, mu, son.upload_mesh(mesh)
    son.close()


def spec(nb, ne, nr, naz):
    return S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(40.0)), nb, ne, nr, naz,
                        math.radians(70.0), math.radians(25.0), 0.5, 10.0)


# 8192 columns are the widest whose column tables a block keeps in shared memory
@pytest.mark.parametrize("widths", [(9001, 64, 61), (64, 61, 9000), (8192, 8193, 512), (8193, 12000), (8192, 3)])
@pytest.mark.parametrize("mode", [1, 2])
def test_widths_on_both_sides_of_the_staged_limit(env, widths, mode):
    son, mu, sid = env
    theta, prm = son.theta(0.05, 1.3, mu), RenderParams(normalise=mode)
    items = [(sid, spec(12, 8, 40, w), 11, k) for k, w in enumerate(widths)]
    b = son.batch(items)
    b.render(theta, prm, hits=True, fan=False, binned=True)
    torch.cuda.synchronize()
    for k, (_, s, seed, frame) in enumerate(items):
        one = son.render(sid, s, theta, prm, seed, frame, hits=True, fan=False, binned=True)
        got = b.view(k)
        for key in ("hits", "binned", "noised", "polar"):
            assert torch.equal(one[key], got[key]), (widths, k, key)
    b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0
