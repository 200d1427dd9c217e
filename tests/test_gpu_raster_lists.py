"""The compositing kernels where their loops can go wrong: 8 x 8 blocks with
0, 1 and a few hits around the loops' unrolling and the 32-entry chunks, images
whose last blocks and tiles are cut, amplitudes below, at and above the alpha
clamp in one list, and colours that are not finite.

Tolerances: the repository's parity bounds against the FP64 oracle (image
1e-4, gradients rel L2 1e-3)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu

SCHEDS = [dict(), dict(tile=(8, 8)), dict(tile=(16, 32)), dict(persistent=1),
          dict(persistent=1, tile=(16, 32)), dict(bwd_mode=1), dict(bwd_mode=1, persistent=1),
          dict(store_depth=4), dict(store_depth=255, persistent=1), dict(max_per_pixel=3),
          dict(max_per_pixel=3, bwd_mode=1, no_pair_stats=1)]


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _pile(n, seed):
    """n small splats behind one another around the image centre, amplitudes
    0 to 1.5 (the clamp is 0.99)."""
    rng = np.random.default_rng(seed)
    pos = rng.normal(0.0, 0.02, (n, 3)).astype(np.float32)
    pos[:, 2] = rng.uniform(-0.5, 0.5, n)
    return dict(pos=pos, sh=scenes.sh_coeffs(rng, n, 1, std=0.2), deg=1,
                opacity=rng.choice(np.float32([0.0, 0.02, 0.05, 0.3, 0.99, 1.5]), n),
                radius=rng.uniform(0.01, 0.03, n).astype(np.float32))


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64).reshape(-1) - b.reshape(-1))
                 / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("sched", SCHEDS, ids=[str(i) for i in range(len(SCHEDS))])
@pytest.mark.parametrize("n", [1, 2, 5, 31, 32, 33, 64, 131])
def test_list_lengths(env, n, sched):
    import torch
    pbr, R = env
    sc = _pile(n, n)
    cams = [scenes.camera((0.0, 0.0, 2.5), 17, 33), scenes.camera((0.5, 0.1, 2.4), 8, 8),
            scenes.camera((-0.4, 0.2, 2.4), 1, 1)]
    npix = pbr.n_pixels(cams)
    g = np.random.default_rng(n + 1).normal(size=(npix, 3))
    scene = pbr.Scene(sc["pos"], sc["sh"], sc["opacity"], sc["radius"], sc["deg"])
    img, st = R.forward([scene], cams, pbr.default_opts(**sched))
    grads = R.backward(st, torch.from_numpy(g.astype(np.float32)).cuda())
    st.close()
    kw = {k: v for k, v in sched.items() if k == "max_per_pixel"}
    args = (sc["pos"], sc["sh"], sc["opacity"], sc["radius"], sc["deg"], cams)
    ref, _, _ = O.render(*args, **kw)
    assert np.abs(img.cpu().numpy() - ref).max() <= 1e-4
    for a, b in zip(grads, O.backward(*args, g.astype(np.float32).astype(np.float64), **kw)):
        assert _rel(a.cpu().numpy(), np.asarray(b)) <= 1e-3


@pytest.mark.parametrize("sched", [dict(), dict(persistent=1), dict(max_per_pixel=2)],
                         ids=["streamed", "persistent", "capped"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_bad_colour_stays_in_its_pixels(env, sched, bad):
    """A splat of non-finite colour leaves the pixels outside its disc as they
    are without it."""
    pbr, R = env
    sc = _pile(40, 3)
    sc["pos"][:20, 0] -= 0.25
    cam = [scenes.camera((0.0, 0.0, 2.5), 48, 24)]
    out = []
    for sh0 in (0.0, bad):
        sh = sc["sh"].copy()
        sh[0, 0, :] = sh0
        scene = pbr.Scene(sc["pos"], sh, sc["opacity"] * 0 + 0.5, sc["radius"], 1)
        img, _ = R.forward([scene], cam, pbr.default_opts(**sched), keep_state=False)
        out.append(img.cpu().numpy())
    touched = ~np.isfinite(out[1]).all(1)
    assert 0 < touched.sum() < 300
    assert np.array_equal(out[0][~touched], out[1][~touched])


@pytest.mark.parametrize("sched", [dict(), dict(persistent=1), dict(bwd_mode=1, tile=(8, 8)),
                                   dict(bwd_mode=1, persistent=1, tile=(16, 32)),
                                   dict(max_per_pixel=7), dict(store_depth=5)],
                         ids=["streamed", "persistent", "8x8", "persistent-16x32", "capped",
                              "depth-5"])
def test_half_blocks_and_blocks_agree(env, sched):
    """A small view alone (a warp per half of an 8 x 8 block) and 900 copies of
    it in one batch (a warp per block): the same image bit for bit, and the
    batch's gradients are 900 times the view's (fp32 sums of 900 equal terms:
    relative error below 900 * 2^-24)."""
    import torch
    pbr, R = env
    rng = np.random.default_rng(8)
    n, copies = 700, 900
    pos = rng.uniform(-0.8, 0.8, (n, 3)).astype(np.float32)
    scene = pbr.Scene(pos, scenes.sh_coeffs(rng, n, 1, std=0.2),
                      rng.choice(np.float32([0.1, 0.5, 0.99, 1.5]), n),
                      rng.uniform(0.03, 0.2, n).astype(np.float32), 1)
    cam = scenes.camera((0.3, 0.2, 2.4), 61, 44)
    g = torch.from_numpy(rng.normal(size=(61 * 44, 3)).astype(np.float32)).cuda()
    opts = pbr.default_opts(**sched)
    img, st = R.forward([scene], [cam], opts)
    one = R.backward(st, g)
    last = st.read("n_contrib")
    st.close()
    imgs, st = R.forward([scene], [cam] * copies, opts)
    many = R.backward(st, g.repeat(copies, 1))
    assert np.array_equal(st.read("n_contrib").reshape(copies, -1), np.tile(last, (copies, 1)))
    st.close()
    assert torch.equal(imgs.view(copies, -1, 3), img.view(1, -1, 3).expand(copies, -1, 3))
    for a, b in zip(many, one):
        assert _rel(a.cpu().numpy(), copies * b.cpu().numpy().astype(np.float64)) <= 900 * 2.0 ** -24
