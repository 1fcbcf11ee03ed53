"""The row terms of the adjoint with two rows per warp (launches of 20,000 rows and
more) against one: rows of fewer, exactly and more than 512 bins, widths off the
16-byte vectors, an odd number of rows.  Frames of 16 rays are one unit of the
gather each, so a batch's gradient is the FP64 sum of the same per-frame terms
however its frames are grouped, rounded to FP32 once.
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


@pytest.mark.parametrize("naz", [8, 61, 512, 516, 1021, 1028])
def test_two_rows_per_warp(naz):
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    sid = son.upload_mesh(mesh)
    theta, prm = son.theta(0.05, 1.2, mu), RenderParams()
    base = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(40.0)), 8, 2, 1853, naz,
                        math.radians(70.0), math.radians(25.0), 0.5, 10.0)
    items = [(sid, base.replace_pose((0.1 * k, 0.05 * k, 0.0), S.pose_matrix(0.03 * k, math.radians(40.0))), 3, k)
             for k in range(11)]   # 20,383 rows
    n = base.n_range_bins * naz
    grad = torch.randn(11 * n, generator=torch.Generator().manual_seed(1)).to(son.device)

    def gradient(k0, k1):
        b = son.batch(items[k0:k1])
        b.render(theta, prm)
        d = b.backward(theta, prm, grad[k0 * n:k1 * n].contiguous()).double().cpu().numpy()
        b.close()
        return d

    whole, parts = gradient(0, 11), [gradient(0, 5), gradient(5, 11)]
    assert np.abs(whole).max() > 0.0
    bound = 2.0 ** -23 * (np.abs(whole) + sum(np.abs(p) for p in parts)) + 1e-30
    assert (np.abs(whole - sum(parts)) <= bound).all()
    son.close()
