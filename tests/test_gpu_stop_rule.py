"""Where a pixel stops: after the point that takes its T below t_eps, and not
before one was composited.  Thresholds at and above 1 (a pixel takes one point)
against the FP64 oracle in every schedule, at the repository's parity bounds
(image 1e-4, gradients rel L2 1e-3); and a T that is not a number does not stop
a pixel: the list positions of every schedule are the block-staged walk's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu

SCHEDS = [dict(), dict(tile=(8, 8), bwd_mode=1), dict(persistent=1, tile=(16, 32)),
          dict(bwd_mode=2, persistent=1), dict(max_per_pixel=2), dict(batch_depth=64)]


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _scene(n=60):
    rng = np.random.default_rng(5)
    pos = rng.normal(0.0, 0.1, (n, 3)).astype(np.float32)
    return dict(pos=pos, sh=scenes.sh_coeffs(rng, n, 1, std=0.2), deg=1,
                opacity=rng.choice(np.float32([0.05, 0.5, 1.5]), n),
                radius=rng.uniform(0.02, 0.08, n).astype(np.float32))


CAMS = [scenes.camera((0.0, 0.0, 2.5), 45, 33), scenes.camera((0.4, 0.1, 2.4), 16, 16)]


@pytest.mark.parametrize("sched", SCHEDS, ids=[str(i) for i in range(len(SCHEDS))])
@pytest.mark.parametrize("t_eps", [0.999, 1.0, 1.5, float("inf")])
def test_high_thresholds(env, t_eps, sched):
    import torch
    pbr, R = env
    sc = _scene()
    g = np.random.default_rng(6).normal(size=(pbr.n_pixels(CAMS), 3)).astype(np.float32)
    scene = pbr.Scene(sc["pos"], sc["sh"], sc["opacity"], sc["radius"], sc["deg"])
    img, st = R.forward([scene], CAMS, pbr.default_opts(t_eps=t_eps, **sched))
    grads = R.backward(st, torch.from_numpy(g).cuda())
    st.close()
    args = (sc["pos"], sc["sh"], sc["opacity"], sc["radius"], sc["deg"], CAMS)
    kw = dict(t_eps=t_eps, **{k: v for k, v in sched.items() if k == "max_per_pixel"})
    ref, _, _ = O.render(*args, **kw)
    assert ref.max() > 0.1
    assert np.abs(img.cpu().numpy() - ref).max() <= 1e-4
    for a, b in zip(grads, O.backward(*args, g.astype(np.float64), **kw)):
        b = np.asarray(b).reshape(-1)
        d = np.linalg.norm(a.cpu().numpy().astype(np.float64).reshape(-1) - b)
        assert d <= 1e-3 * np.linalg.norm(b)
    # the other ways in
    buf = torch.empty_like(img)
    pbr.render_forward_noalloc([scene], CAMS, pbr.default_opts(t_eps=t_eps, **sched), out=buf)
    assert np.abs(buf.cpu().numpy() - ref).max() <= 1e-4
    G = pbr.Graph(R, [scene], CAMS, pbr.default_opts(t_eps=t_eps, **sched))
    G.launch(pbr.Graph.FORWARD)
    assert np.abs(G.out.cpu().numpy() - ref).max() <= 1e-4
    G.close()


@pytest.mark.parametrize("sched", SCHEDS[:-1], ids=[str(i) for i in range(len(SCHEDS) - 1)])
def test_a_t_that_is_not_a_number(env, sched):
    pbr, R = env
    sc = _scene()
    sc["opacity"][np.argmax(sc["pos"][:, 2])] = -np.inf  # the first camera's nearest
    scene = pbr.Scene(sc["pos"], sc["sh"], sc["opacity"], sc["radius"], sc["deg"])
    last = []
    for s in (sched, dict(batch_depth=64, tile=sched.get("tile", (16, 16)),
                          max_per_pixel=sched.get("max_per_pixel", 0))):
        _, st = R.forward([scene], CAMS, pbr.default_opts(**s))
        last.append((np.isnan(st.read("T_final")), st.read("n_contrib")))
        st.close()
    assert last[0][0].any()
    assert np.array_equal(last[0][0], last[1][0]) and np.array_equal(last[0][1], last[1][1])
