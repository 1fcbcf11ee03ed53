"""The fold of hit records into bins and the row kernel (noise, normalisation)
at the sizes where their tiling has edges: rows of one, few, odd and more than
1024 azimuth bins, range bins around the 32-row bands, fewer and more beams than
columns.  The reference is numpy on the records that the same render returns:
sums in FP64, the oracle's noise, and the IEEE division of I~ by its maximum.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2503_01074_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import NO_KEY, RenderParams, Sonar, hits_numpy  # noqa: E402

ALPHA, GAIN = 0.05, 1.3


@pytest.fixture(scope="module")
def env():
    son = Sonar(0)
    mesh, mu = S.tiny_scene()
    yield son, mesh, mu, son.upload_mesh(mesh)
    son.close()


# (beams, elevations, range bins, azimuth bins, normalise)
SHAPES = [
    (1, 1, 1, 1, 1), (3, 5, 31, 2, 1), (64, 33, 32, 61, 1), (64, 32, 33, 64, 1), (97, 7, 65, 128, 2),
    (50, 40, 300, 13, 1), (130, 20, 100, 3, 0), (300, 9, 70, 1, 1), (256, 4, 96, 512, 1), (300, 4, 40, 513, 1),
    (128, 6, 50, 1021, 1), (128, 6, 50, 1024, 2), (200, 5, 37, 1030, 1), (100, 4, 20, 2052, 1), (64, 16, 1200, 24, 1),
    (40, 8, 20000, 8, 1), (12, 3, 9, 9001, 1),
]


@pytest.mark.parametrize("nb,ne,nr,naz,mode", SHAPES)
def test_fold_and_rows(env, nb, ne, nr, naz, mode):
    son, mesh, mu, sid = env
    spec = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(40.0)), nb, ne, nr, naz,
                        math.radians(70.0), math.radians(25.0), 0.5, 10.0)
    theta = son.theta(ALPHA, GAIN, mu)
    out = son.render(sid, spec, theta, RenderParams(normalise=mode), 11, 5, hits=True, binned=True)
    torch.cuda.synchronize()
    h = hits_numpy(out["hits"])
    ok = h["key"] != NO_KEY
    score = (mu.astype(np.float64)[mesh.mat[h["tri"][ok]]] * h["cos"][ok] *
             np.exp(-2.0 * float(np.float32(ALPHA)) * h["r"][ok]) * float(np.float32(GAIN)))
    P = np.zeros(nr * naz)
    np.add.at(P, h["key"][ok].astype(np.int64), score)
    got = out["binned"].double().cpu().numpy().ravel()
    # every addend within 2^-21 (products and expf), the FP32 sum of n addends within n 2^-24 more
    n = np.bincount(h["key"][ok].astype(np.int64), minlength=nr * naz).max(initial=1)
    np.testing.assert_allclose(got, P, rtol=2.0 ** -21 + n * 2.0 ** -24, atol=0)
    noised = out["noised"].cpu().numpy()
    # the draws agree to a few 1e-6 of themselves; both terms of Eq. 3 are positive here
    np.testing.assert_allclose(noised.ravel(), O.noise(spec, got, 11, 5).ravel(), rtol=1e-5, atol=0)
    top = {0: np.ones(1, np.float32), 1: noised.max(1, keepdims=True), 2: noised.max()}[mode]
    assert np.array_equal(out["polar"].cpu().numpy(), noised / top)   # correctly rounded division
    st, bits = son.check()
    assert st == 0 and bits == 0


def test_negative_reflectivity_rows(env):
    """Negative bins (a fit may pass through negative reflectivities) leave the
    short division; rows whose maximum is not positive are not divided."""
    son, mesh, mu, sid = env
    spec = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.0, math.radians(40.0)), 64, 32, 60, 64,
                        math.radians(60.0), math.radians(25.0), 0.0, 10.0)
    theta = son.theta(0.01, 1.0, -50.0 * mu)
    out = son.render(sid, spec, theta, RenderParams(), 3, 4)
    torch.cuda.synchronize()
    noised = out["noised"].cpu().numpy()
    top = noised.max(1, keepdims=True)
    assert (noised < 0).any()
    assert np.array_equal(out["polar"].cpu().numpy(), np.where(top > 0, noised / top, noised))
