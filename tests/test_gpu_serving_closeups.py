"""Requests from cameras inside a scene, whose host bounds are loose: they share a
batch by what they need, not by their bounds."""
import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


def test_closeups_share_a_batch():
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    rng = np.random.default_rng(7)
    n = 200_000
    data = dict(pos=scenes.surface_points(rng, n, 8), sh=scenes.sh_coeffs(rng, n, 0, 0.2),
                opacity=np.full(n, 0.8, np.float32),
                radius=scenes.log_uniform(rng, n, 0.003, 0.01), deg=0)
    scene = pbr.Scene(data["pos"], data["sh"], data["opacity"], data["radius"], 0)
    R = pbr.Renderer(0)
    # a bound here is every point in all 3,600 tiles of the view, 16 bytes a
    # pair: 11.5 GB, of which the budget holds one
    budget = 20 << 30
    sv = pbr.Server(R, max_batch_views=16, n_streams=1, hbm_budget=budget)
    sid = sv.upload(data)
    cams = [scenes.camera((0.2 * np.cos(a), 0.1, 0.2 * np.sin(a)), 1280, 720) for a in range(6)]
    for c in cams:
        exact, _ = R.workspace_size([scene], [c], keep_state=False)
        assert 6 * exact < budget // 2
        assert sv.estimate(sid, c) == exact
    # a large view keeps the one stream busy while the close-ups are queued
    big = sv.submit(sid, scenes.camera((0.0, 0.5, 4.0), 12288, 12288))
    subs = [sv.submit(sid, c) for c in cams]
    assert [sv.wait(r) for r, _ in [big] + subs] == [0] * 7
    st = sv.stats()
    assert st["completed"] == 7 and st["max_batch_views"] >= 2
    for c, (_, out) in zip(cams, subs):
        ref, _ = R.forward([scene], [c], keep_state=False)
        assert torch.equal(ref.view(-1), out.view(-1))
    sv.stop()
    R.close()
