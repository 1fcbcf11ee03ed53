"""The autotuner on batches whose ray cast takes several lanes per ray whatever the
tuning row says: the row's variant then governs larger batches of the shape only,
and must not be the outcome of timing equal launches.
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

CAP = 8


@pytest.mark.parametrize("hits", [True, False])
def test_small_batches_keep_the_default_variant(hits):
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    sid, theta, prm = son.upload_mesh(mesh), son.theta(0.05, 1.0, mu), RenderParams()
    shapes = [(64, 16, 100, 64), (37, 11, 65, 61), (128, 33, 40, 128), (1, 1, 1, 1), (5, 300, 33, 2), (300, 9, 70, 3)]
    items = [(sid, S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(40.0)), *shape,
                                math.radians(70.0), math.radians(25.0), 0.5, 10.0), 3, k)
             for k, shape in enumerate(shapes)]
    b = son.batch(items)
    b.autotune(theta, prm, hits=hits)
    rows = {tuple(r[:4]): r[4:] for r in son.tune_get().tolist()}
    assert set(rows) == set(shapes)
    assert all(r[3] == CAP for r in rows.values()), rows
    b.close()
    son.close()
