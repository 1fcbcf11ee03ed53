"""The emission schedule on both sides of the sizes where its kernel changes (a warp
per vehicle, a thread per vehicle for short schedules of many vehicles): the same rows
whichever takes them, for ordinary periods and for those no sensor gives.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import Sonar  # noqa: E402


def by_steps(period, dt):
    """Emissions of [n, steps] periods, all vehicles a step at a time (FP32 quotients, as stated)."""
    n, steps = period.shape
    with np.errstate(divide="ignore", invalid="ignore", over="ignore"):
        q = np.ceil(period / np.float32(dt))
    wait = np.where(q >= 1.0, np.minimum(q, 1e6), 1.0).astype(np.int64)   # NaN and less than a step: the next one
    out, due = np.zeros((n, steps), np.int32), np.zeros(n, np.int64)
    for s in range(steps):
        now = due == s
        out[now, s] = 1
        due[now] += wait[now, s]
    return out


@pytest.mark.parametrize("n,steps", [(32767, 48), (32768, 48), (32768, 49), (32769, 47), (40000, 1), (33000, 7), (5, 48),
                                     (3, 700)])
def test_schedule_forms(n, steps):
    son = Sonar(0)
    rng = np.random.default_rng(n + steps)
    p = rng.choice(np.float32([0.05, 0.1, 0.25, 0.31, 1.7, 40.0]), (n, steps))
    odd = np.float32([np.nan, np.inf, -np.inf, 0.0, -3.0, 1e-40, 3e38, 1e12])
    where = rng.random((n, steps)) < 0.1
    p[where] = rng.choice(odd, where.sum())
    emit = son.dvl_schedule(torch.from_numpy(p).to(son.device), 0.1)
    assert np.array_equal(emit.cpu().numpy(), by_steps(p, 0.1))
    son.close()
