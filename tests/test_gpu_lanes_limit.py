"""The ray cast on both sides of the launch sizes where its lanes per ray change: up to 4
tiles of 32 rays per SM eight lanes a ray, up to 22 four, beyond that one.  The hit
records do not depend on it.  Frames of one ragged tile, so that a batch can be put
exactly at, below and above either limit.
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

MESHES = {"tri": lambda: S.random_soup(1, 5, degenerate_frac=0.0), "400": lambda: S.random_soup(400, 9),
          "30000": lambda: S.random_soup(30000, 9)}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("prm", [RenderParams(), RenderParams(two_sided=0, clip_tmax=0)])
def test_records_at_the_limits(name, prm):
    son = Sonar(0)
    sid = son.upload_mesh(MESHES[name]())
    theta = son.theta(0.03, 1.7, np.array([0.2, 0.5, 0.7, 0.9], np.float32))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    base = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.05, math.radians(25)), 5, 3, 64, 5,
                        math.radians(90.0), math.radians(40.0), 0.5, 20.0)
    specs = [base.replace_pose((0.05 * k, -0.03 * k, 0.01 * k), S.pose_matrix(0.3 * k, math.radians(-20 + 7 * k)))
             for k in range(8)]
    alone = torch.stack([son.render(sid, s, theta, prm, 1, 2, hits=True)["hits"] for s in specs])
    assert (alone[:, :, 1] >= 0).any() or name == "tri"
    for frames in (4 * sms, 4 * sms + 1, 22 * sms, 22 * sms + 1, 26 * sms):
        for row in (None, 0, 8, 16, 24):   # the variants of a tuning row, and none
            if row is not None:
                son.tune_set([[5, 3, 64, 5, 1, 8, 128, row]])
            b = son.batch([(sid, specs[k % 8], 1, 2) for k in range(frames)])
            assert b.info()["rays"] == 15 * frames
            b.render(theta, prm, hits=True, fan=False)
            torch.cuda.synchronize()
            got = b.hits.view(frames, 15, 4)
            want = alone[torch.arange(frames, device=son.device) % 8]
            assert torch.equal(got, want), (frames, row)
            b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0
    son.close()
