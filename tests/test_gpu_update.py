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


def deep_scene():
    """Clusters in seven octants of every cube, the eighth halved again, 18 times: an
    8-wide tree of more levels than its walk's stack takes, a 4-wide one that fits."""
    r = np.random.default_rng(0)
    tris = []
    for level in range(18):
        side = 8.0 * 0.5 ** level
        for q in range(1, 8):
            corner = np.array([q & 1, q >> 1 & 1, q >> 2 & 1]) * side / 2
            for _ in range(4):
                x = corner + side / 2 * (0.2 + 0.6 * r.random(3))
                tris.append(x + 0.15 * side * (r.random((3, 3)) - 0.5))
    v = np.array(tris).reshape(-1, 3).astype(np.float32) + np.float32([-2.0, 1.0, -2.0])
    return S.Mesh(v, np.arange(len(v), dtype=np.int32).reshape(-1, 3), np.zeros(len(tris), np.int32))


@pytest.mark.parametrize("variant", [None, 16])
@pytest.mark.parametrize("n", [3, 300])
def test_update_to_a_scene_without_an_8_wide_tree(son, variant, n):
    """A batch planned for the 8-wide trees (several lanes per ray, or by its tuning
    row) walks the 4-wide ones once an item's scene has no other, and its own again
    after; the records do not depend on the tree."""
    theta, prm = son.theta(0.05, 1.0, MU), RenderParams()
    wide, deep, one = (son.upload_mesh(m) for m in (S.tiny_scene()[0], deep_scene(), S.random_soup(2, 5)))
    info = son.scene_info(deep)
    assert info["bytes"] == 52 * info["n_tris"] + 128 * info["n_pairs"]   # no 8-wide nodes
    spec = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(15)), 64, 32, 100, 64,
                        math.radians(100.0), math.radians(40.0), 0.5, 20.0)
    if variant is not None:
        son.tune_set([[64, 32, 100, 64, 1, 8, 128, variant]])
    alone = {}
    b = son.batch(frames(wide, n, spec))
    grad = torch.randn(b.n_polar, generator=torch.Generator().manual_seed(2)).to(son.device)
    for sids in ([wide], [wide, deep], [deep], [one, wide], [one, deep], [wide]):
        items = [(sids[k % len(sids)],) + it[1:] for k, it in enumerate(frames(wide, n, spec))]
        b.update(items)
        step(b, theta, prm, grad)
        d = b.backward(theta, prm, grad, hits=False).clone()
        torch.cuda.synchronize()
        assert torch.isfinite(d).all()
        for k in {0, 1, n - 1}:
            sid, sp, seed, frame = items[k]
            if (sid, k) not in alone:
                alone[sid, k] = son.render(sid, sp, theta, prm, seed, frame, hits=True)["hits"].clone()
            assert torch.equal(b.view(k)["hits"], alone[sid, k]), (sids, k)
    assert (alone[deep, 1][:, 1] >= 0).any()
    b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0


def test_tables_follow_every_change_of_the_fields_of_view(son):
    """Changes of the fields of view one after another: every block of the exact-ray and
    of the fan coordinate tables is built whole each time (a block whose stamp is
    current has nothing to do, and no warp of it may see the stamp of its own build)."""
    theta, prm = son.theta(0.05, 1.0, MU), RenderParams()
    sid = son.upload_mesh(S.random_soup(3000, 9))
    base = S.SensorSpec(np.zeros(3, np.float32), S.pose_matrix(0.1, math.radians(15)), 200, 90, 64, 128,
                        math.radians(90.0), math.radians(40.0), 0.5, 20.0, 211, 130)
    n = 16   # all alike: one shared fan table
    b = son.batch(frames(sid, n, base))
    for k in range(12):
        spec = base.replace_pose(base.pos, base.rot)
        if k % 4 != 3:   # the last of four is the one before: nothing to rebuild
            spec.hfov, spec.vfov = base.hfov * (1.0 - 0.02 * k), base.vfov * (1.0 - 0.015 * k)
        else:
            spec.hfov, spec.vfov = last.hfov, last.vfov
        last = spec
        items = frames(sid, n, spec)
        b.update(items)
        b.render(theta, prm)
        torch.cuda.synchronize()
        for q in (0, n // 2, n - 1):
            _, sp, seed, frame = items[q]
            one = son.render(sid, sp, theta, prm, seed, frame, hits=True, fan=True)
            got = b.view(q)
            assert all(torch.equal(one[key], got[key]) for key in ("hits", "polar", "fan")), (k, q)
    b.close()
