"""The scene build at the sizes where its launches have edges: one and two
triangles (a scene of one leaf), three, the sort's tiles (3072 keys) and their
neighbours, equal keys throughout, and a tree much deeper than its size suggests.
A scene's hits must not depend on the build: they are compared with the
oracle's brute force, and a rebuilt scene must give the same records.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_2503_01074_gb300 import scenes as S

from tests._parity import hit_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2503_01074_gb300.sonar import RenderParams, Sonar, SonarError, hits_numpy  # noqa: E402


@pytest.fixture(scope="module")
def son():
    s = Sonar(0)
    yield s
    s.close()


def spec():
    return S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(15)), 40, 24, 100, 40,
                        math.radians(100.0), math.radians(30.0), 0.5, 20.0)


def stacked(n):
    """n coincident triangles and one beside them: every key but one is equal."""
    m = S.random_soup(1, 3, degenerate_frac=0.0, sliver_frac=0.0)
    v = np.concatenate([np.tile(m.verts, (n, 1)), m.verts + np.float32(1.0)])
    return S.Mesh(v, np.arange(3 * (n + 1), dtype=np.int32).reshape(-1, 3), np.zeros(n + 1, np.int32))


def geometric(n):
    """Triangles at halving distances from a corner: a comb-shaped tree."""
    c = 6.0 * 0.5 ** np.arange(n)
    base = np.array([[0.0, 0.0, 0.0], [0.3, 0.0, 0.0], [0.0, 0.0, 0.3]])
    v = (base[None] * np.minimum(1.0, c)[:, None, None] + np.stack([c, c + 4.0, -c], -1)[:, None, :]).reshape(-1, 3)
    return S.Mesh(v.astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(-1, 3), np.zeros(n, np.int32))


MESHES = {"1": lambda: S.random_soup(1, 5, degenerate_frac=0.0), "2": lambda: S.random_soup(2, 5), "3": lambda: S.random_soup(3, 5),
          "33": lambda: S.random_soup(33, 5), "3071": lambda: S.random_soup(3071, 5), "3072": lambda: S.random_soup(3072, 5),
          "3073": lambda: S.random_soup(3073, 5), "9217": lambda: S.random_soup(9217, 5),
          "stacked": lambda: stacked(700), "comb": lambda: geometric(20)}


@pytest.mark.parametrize("name", list(MESHES))
def test_hits_against_brute_force(son, name):
    mesh, sp, prm = MESHES[name](), spec(), RenderParams()
    theta = son.theta(0.03, 1.2, np.array([0.2, 0.5, 0.7, 0.9], np.float32))
    sids = [son.upload_mesh(mesh) for _ in range(2)]
    out = [son.render(sid, sp, theta, prm, 1, 2, hits=True)["hits"] for sid in sids]
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
    ref = O.render(mesh, np.array([0.2, 0.5, 0.7, 0.9]), 0.03, 1.2, sp, O.Params(), seed=1, frame=2, fan=False)
    hit_parity(ref, hits_numpy(out[0]))
    st, bits = son.check()
    assert st == 0 and bits == 0
    for sid in sids:
        son.release(sid)


def test_refused_scenes_leave_the_context_usable(son):
    """A refused upload (its build stops after the validation) and good ones in turn."""
    mesh = S.random_soup(5000, 5)
    bad = [(mesh.verts, np.where(mesh.tris == 7, 10 ** 6, mesh.tris), mesh.mat, "index"),
           (mesh.verts, mesh.tris, mesh.mat - 4, "material"),
           (np.where(np.arange(mesh.verts.shape[0])[:, None] == 9, np.float32(np.nan), mesh.verts), mesh.tris, mesh.mat,
            "finite")]
    want = None
    theta = son.theta(0.03, 1.2, np.array([0.2, 0.5, 0.7, 0.9], np.float32))
    for v, t, m, what in bad:
        with pytest.raises(SonarError, match=what):
            son.upload(v, t, m)
        sid = son.upload_mesh(mesh)
        h = son.render(sid, spec(), theta, RenderParams(), 1, 2, hits=True)["hits"].clone()
        want = h if want is None else want
        assert torch.equal(h, want)
        son.release(sid)
