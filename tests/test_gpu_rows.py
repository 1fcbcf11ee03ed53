"""The row kernel (noise, range-wise normalisation): launches that its widest
sensor alone does not describe, and bins that are not finite.
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


# rows in registers and written back, with 16-byte vectors and without, quads over their ends
@pytest.mark.parametrize("naz", [64, 61, 62, 513, 516, 1021, 1030, 1032])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("value", [-math.inf, math.inf, math.nan])
def test_bins_that_are_not_finite(env, naz, mode, value):
    """A reflectivity of +-inf or NaN (a fit that diverges) stays in the bins that it
    reaches, and its neighbours keep the values that they have without it: a bin
    without such a return is what a render with that material at zero gives."""
    son, mu, sid = env
    sp, prm = spec(64, 32, 60, naz), RenderParams(normalise=mode)
    bad, zero = np.array(mu, np.float32), np.array(mu, np.float32)
    bad[0], zero[0] = value, 0.0
    out = son.render(sid, sp, son.theta(0.05, 1.0, bad), prm, 3, 4, fan=False, binned=True)
    ref = son.render(sid, sp, son.theta(0.05, 1.0, zero), prm, 3, 4, fan=False, binned=True)
    torch.cuda.synchronize()
    P, I, N = (out[k].cpu().numpy() for k in ("binned", "noised", "polar"))
    hit = ~np.isfinite(P)
    assert hit.any() and not hit.all()
    assert np.array_equal(I[hit], P[hit], equal_nan=True)
    assert np.array_equal(I[~hit], ref["noised"].cpu().numpy()[~hit])
    # the maximum passes over NaN; a row or image whose maximum is not positive is not divided
    finite = np.where(np.isnan(I), -np.inf, I)
    top = {0: np.ones(1, np.float32), 1: finite.max(1, keepdims=True), 2: finite.max()}[mode]
    with np.errstate(invalid="ignore"):
        want = np.where(top > 0, I / top, I)
    assert np.array_equal(N, want, equal_nan=True)
