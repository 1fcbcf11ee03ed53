"""The row kernel (noise, range-wise normalisation): launches that its widest
sensor alone does not describe, bins that are not finite, rows that a block shares.
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


def off_by_one(n, like=None):
    """n floats that start four bytes past a 16-byte boundary."""
    v = torch.zeros(n + 1, device="cuda")[1:]
    assert v.data_ptr() % 16 == 4
    return v if like is None else v.copy_(like.reshape(-1))


# rows in registers by pairs and alone, in two passes, no multiple of 4; one and two rows per warp of the adjoint
@pytest.mark.parametrize("nr,naz", [(60, 64), (41, 512), (33, 516), (20, 1024), (20, 1028), (30, 61), (7000, 64)])
@pytest.mark.parametrize("mode", [1, 2])
def test_images_off_the_16_byte_boundary(env, nr, naz, mode):
    """Images and gradients may start at any float.  Forward: the same images, bit for
    bit.  Adjoint: the same gradient, since one nonzero element of G per row (per
    image with whole-image normalisation) leaves no order of summation in its row terms."""
    son, mu, sid = env
    theta, prm = son.theta(0.05, 1.3, mu), RenderParams(normalise=mode)
    items = [(sid, spec(64, 16, nr, naz).replace_pose((0.1 * k, 0.0, 0.0), S.pose_matrix(0.1, math.radians(40.0))), 5, k)
             for k in range(3)]
    _, sp, seed, frame = items[0]
    n = nr * naz
    rng = np.random.default_rng(1)
    G = np.zeros((3, nr, naz), np.float32)
    for k in range(3):
        for row in range(nr) if mode == 1 else (int(rng.integers(nr)),):
            G[k, row, rng.integers(naz)] = rng.uniform(0.5, 2.0)
    G = torch.from_numpy(G).to(son.device)

    one = son.render(sid, sp, theta, prm, seed, frame, hits=True, fan=False)
    views = {key: off_by_one(n).view(nr, naz) for key in ("polar", "noised")}
    got = son.render(sid, sp, theta, prm, seed, frame, hits=True, fan=False, outputs=dict(views))
    assert torch.equal(got["polar"], one["polar"]) and torch.equal(got["noised"], one["noised"])
    d = son.backward(sid, sp, theta, prm, seed, frame, G[0].contiguous(), one["noised"], one["hits"])
    for g, x in ((off_by_one(n, G[0]), one["noised"]), (G[0].contiguous(), views["noised"]),
                 (off_by_one(n, G[0]), views["noised"])):
        assert torch.equal(son.backward(sid, sp, theta, prm, seed, frame, g.view(nr, naz), x, one["hits"]), d)

    b, c = son.batch(items), son.batch(items)
    c.polar, c.noised = off_by_one(3 * n), off_by_one(3 * n)
    grads = []
    for x, g in ((b, G.reshape(-1)), (c, off_by_one(3 * n, G))):
        x.render(theta, prm, fan=False)
        grads.append(x.backward(theta, prm, g).clone())
        grads.append(x.step(theta, prm, g, fan=False).clone())
    torch.cuda.synchronize()
    assert torch.equal(b.polar, c.polar) and torch.equal(b.noised, c.noised)
    assert torch.isfinite(grads[0]).all()
    if mode == 1:   # one element of a whole image may lie where nothing returned
        assert grads[0].abs().max() > 0
    assert all(torch.equal(g, grads[0]) for g in grads[1:])
    b.close()
    c.close()
    st, bits = son.check()
    assert st == 0 and bits == 0


# a block a row, its last quads of fewer than a warp's or a block's: below and above the limit of four rows per SM
@pytest.mark.parametrize("nr,naz", [(1, 1025), (1, 1028), (3, 4095), (33, 1151), (9, 8192), (2, 8193), (607, 1030), (609, 1032)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_rows_shared_by_a_block(env, nr, naz, mode):
    """The same rows in a batch that has too many for a block each (a warp a row)."""
    son, mu, sid = env
    theta, prm = son.theta(0.05, 1.3, mu), RenderParams(normalise=mode)
    sp = spec(50, 12, nr, naz)
    one = son.render(sid, sp, theta, prm, 3, 4, hits=True, fan=False, binned=True)
    b = son.batch([(sid, sp, 3, 4)] + [(sid, spec(1, 1, 700, 2), 3, 4)])
    b.render(theta, prm, fan=False, binned=True)
    torch.cuda.synchronize()
    got = b.view(0)
    for key in ("hits", "binned", "noised", "polar"):
        assert torch.equal(one[key], got[key]), key
    top = {0: torch.ones(1, device=son.device), 1: one["noised"].amax(1, keepdim=True), 2: one["noised"].max()}[mode]
    assert torch.equal(one["polar"], one["noised"] / top)
    b.close()


# columns of 1023 to 2560 rays, beams that do not divide evenly, more rows than a block keeps per beam
@pytest.mark.parametrize("nb,ne,nr,naz", [(11, 93, 70, 1), (64, 64, 9000, 4), (255, 1024, 100, 255), (500, 20, 8000, 7),
                                          (2050, 5, 6000, 9), (31, 33, 40, 31)])
def test_fold_by_blocks_and_by_warps(env, nb, ne, nr, naz):
    """Few columns of many rays are folded by a block each, in a batch of more columns by
    a warp each: the same sums, bit for bit."""
    son, mu, sid = env
    theta, prm = son.theta(0.05, 1.3, mu), RenderParams()
    sp = spec(nb, ne, nr, naz)
    one = son.render(sid, sp, theta, prm, 3, 4, hits=True, fan=False, binned=True)
    light = (sid, spec(5, 3, 40, 1), 3, 4)   # in a launch with the blocks, by warps of a block of 16
    for others in ([], [light], [(sid, spec(3, 2, 5, 300), 3, 4)]):
        b = son.batch([(sid, sp, 3, 4)] + others)
        b.render(theta, prm, fan=False, binned=True)
        torch.cuda.synchronize()
        got = b.view(0)
        for key in ("hits", "binned", "noised", "polar"):
            assert torch.equal(one[key], got[key]), (key, len(others))
        if others and others[0] is light:
            small = son.render(sid, light[1], theta, prm, 3, 4, hits=True, fan=False, binned=True)
            assert all(torch.equal(small[key], b.view(1)[key]) for key in ("hits", "binned", "noised", "polar"))
        b.close()
    st, bits = son.check()
    assert st == 0 and bits == 0
