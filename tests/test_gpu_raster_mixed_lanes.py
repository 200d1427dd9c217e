"""Forward with a warp per half block and backward with a warp per block (the
middle of the rule's range) against the FP64 oracle, at the repository's parity
bounds (image 1e-4, gradients rel L2 1e-3)."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as O
from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sched,size", [
    (dict(bwd_mode=1, no_pair_stats=1), (420, 330)),
    (dict(bwd_mode=2, no_pair_stats=1), (800, 450)),
    (dict(bwd_mode=2, persistent=1), (800, 450)),
    (dict(bwd_mode=2, no_pair_stats=1, tile=(16, 32)), (797, 453))], ids=["recompute", "store", "persistent", "16x32"])
def test_half_forward_whole_backward(sched, size):
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    rng = np.random.default_rng(1)
    n = 1200
    sc = dict(pos=rng.uniform(-1.0, 1.0, (n, 3)).astype(np.float32),
              sh=scenes.sh_coeffs(rng, n, 1, std=0.2),
              opacity=rng.choice(np.float32([0.1, 0.6, 0.99, 1.5]), n),
              radius=np.full(n, 20.0 / size[0], np.float32), deg=1)
    cams = [scenes.camera((0.1, 0.2, 3.0), *size)]
    opts = pbr.default_opts(**sched)
    R = pbr.Renderer(0)
    scene = pbr.Scene(sc["pos"], sc["sh"], sc["opacity"], sc["radius"], 1)
    img, st = R.forward([scene], cams, opts)
    f, two, info = pbr.lib().pbr_test_raster_lanes, (C.c_int32 * 2)(), st.info()
    f.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_void_p, C.c_int32, C.c_void_p, C.c_int32,
                  C.c_int64, C.c_int64, C.c_void_p]
    assert f(C.byref(scene.points()), 1, None, pbr.make_cameras(cams), 1, C.byref(opts),
             int(st.read("n_comp").size > 0), info["n_visible"], info["n_pairs"], two) == 0
    assert list(two) == [0, 1]
    grad = rng.normal(size=(size[0] * size[1], 3)).astype(np.float32)
    grads = R.backward(st, torch.from_numpy(grad).cuda())
    st.close()
    args = (sc["pos"], sc["sh"], sc["opacity"], sc["radius"], 1, cams)
    ref, _, _ = O.render(*args)
    assert np.abs(img.cpu().numpy() - ref).max() <= 1e-4
    for a, b in zip(grads, O.backward(*args, grad.astype(np.float64))):
        b = np.asarray(b).reshape(-1)
        d = np.linalg.norm(a.cpu().numpy().astype(np.float64).reshape(-1) - b)
        assert d <= 1e-3 * np.linalg.norm(b)
    R.close()
