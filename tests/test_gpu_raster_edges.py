"""Pixels an ulp inside a splat's edge in the persistent schedule, whose fused
squared distance can lie below the cutoff where the separately rounded one lies
above it.  The splat is composited there whatever rectangle the warp culls with:
half a block (a view alone) or a whole one (copies of it), and the backward
sees the same points as the forward."""
import ctypes as C

import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu
F = np.float32
SIDE = 16  # blocks a side


def _edge_points():
    """A splat per 8 x 8 block that reaches one pixel of the block's row 4 by its
    fused distance only, and rows above it anyhow: (px, py, radius, pixel)."""
    rng = np.random.default_rng(3)
    out = []
    for by in range(SIDE):
        for bx in range(SIDE):
            while True:
                px = F(8 * bx + rng.uniform(2.0, 6.0))
                py = F(8 * by + rng.uniform(1.0, 3.0))
                cx, cy = F(np.floor(px)) + F(0.5), F(8 * by + 4.5)
                dx, dy = cx - px, cy - py
                dx2 = dx * dx
                plain = dx2 + dy * dy
                exact = np.float64(dy) * np.float64(dy) + np.float64(dx2)
                fused = F(exact)
                if not fused < plain:
                    continue
                r = F(np.sqrt(np.float64(fused)) / 3.0)
                for cand in (np.nextafter(r, F(0)), r, np.nextafter(r, F(9))):
                    rc = F(3.0) * cand
                    if fused <= rc * rc < plain:
                        out.append((px, py, cand, int(cy) * 8 * SIDE + int(cx)))
                        break
                else:
                    continue
                break
    return out


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _lanes(pbr, scene, cams, opts, st):
    """[forward, backward]: whether the warps of a pass take whole blocks."""
    f, two, info = pbr.lib().pbr_test_raster_lanes, (C.c_int32 * 2)(), st.info()
    f.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_int32,
                  C.c_int64, C.c_int64, C.c_void_p]
    assert f(C.byref(scene.points()), 1, None, pbr.make_cameras(cams), len(cams), C.byref(opts),
             int(st.read("n_comp").size > 0), info["n_visible"], info["n_pairs"], two) == 0
    return list(two)


@pytest.mark.parametrize("sched", [dict(bwd_mode=1), dict(bwd_mode=2), dict(tile=(16, 32))],
                         ids=["recompute", "store", "16x32"])
def test_an_edge_pixel_in_half_and_whole_blocks(env, sched):
    import torch
    pbr, R = env
    pts = _edge_points()
    n, copies = len(pts), 1500
    pos = np.array([(x, y, 1.0) for x, y, _, _ in pts], F)  # px = X / z, py = Y / z
    rad = np.array([r for _, _, r, _ in pts], F)
    edge = [p for _, _, _, p in pts]
    scene = pbr.Scene(pos, scenes.sh_coeffs(np.random.default_rng(4), n, 0, std=0.2),
                      np.full(n, 0.5, F), rad, 0)
    W = 8 * SIDE
    cam = dict(fx=F(1), fy=F(1), cx=F(0), cy=F(0), R=np.eye(3, dtype=F), t=np.zeros(3, F),
               width=W, height=W)
    opts = pbr.default_opts(persistent=1, **sched)
    g = torch.from_numpy(np.random.default_rng(5).normal(size=(W * W, 3)).astype(F)).cuda()
    img, st = R.forward([scene], [cam], opts)
    one = R.backward(st, g)
    last, lanes = st.read("n_contrib"), [_lanes(pbr, scene, [cam], opts, st)]
    st.close()
    assert (last[edge] > 0).all()
    imgs, st = R.forward([scene], [cam] * copies, opts)
    many = R.backward(st, g.repeat(copies, 1))
    lanes.append(_lanes(pbr, scene, [cam] * copies, opts, st))
    assert np.array_equal(st.read("n_contrib").reshape(copies, -1), np.tile(last, (copies, 1)))
    st.close()
    assert lanes == [[0, 0], [1, 1]]
    assert torch.equal(imgs.view(copies, -1, 3), img.view(1, -1, 3).expand(copies, -1, 3))
    for a, b in zip(many, one):
        b = copies * b.cpu().numpy().astype(np.float64)
        d = np.linalg.norm(a.cpu().numpy().reshape(-1) - b.reshape(-1))
        assert d <= copies * 2.0 ** -24 * np.linalg.norm(b)
