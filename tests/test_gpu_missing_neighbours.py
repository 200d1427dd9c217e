"""Points without neighbours (a coordinate that is not a number: at no finite
distance to any other): the update and the frame initialisation leave the other
points as they are without them and mark the point itself NaN."""
import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _cloud(n):
    """Points in a ball (the corner cell of their grid, where NaN goes, is empty)."""
    rng = np.random.default_rng(n)
    p = rng.normal(size=(n, 3))
    p *= (rng.uniform(size=(n, 1)) ** (1 / 3)) / np.linalg.norm(p, axis=1, keepdims=True)
    return (p.astype(np.float32), scenes.sh_coeffs(rng, n, 1, std=0.2),
            rng.uniform(0.1, 0.9, n).astype(np.float32), np.full(n, 0.02, np.float32))


@pytest.mark.parametrize("n,k,stages", [(500, 1, 7), (500, 4, 5), (3000, 8, 5), (40_000, 2, 5)])
def test_refine(env, n, k, stages):
    pbr, R = env
    a = _cloud(n)
    b = [np.concatenate([x, x[:1]]) for x in a]
    b[0][-1] = np.nan
    base, (m, m2, total) = pbr.refine_points(R, pbr.Scene(*a, 1), n_vox=16, k=k, stages=stages,
                                             eps=1e9)
    got, counts = pbr.refine_points(R, pbr.Scene(*b, 1), n_vox=16, k=k, stages=stages, eps=1e9)
    assert list(counts) == [m + 1, m2 + 1, total + 2]
    at = np.r_[0, m2 + 1]  # the point itself (first cell) and the one made from it
    rest = np.setdiff1d(np.arange(total + 2), at)
    for x, y in ((base.pos, got.pos), (base.sh, got.sh), (base.opacity, got.opacity),
                 (base.radius, got.radius)):
        x, y = x.cpu().numpy()[:total], y.cpu().numpy()[:total + 2]
        assert np.array_equal(x, y[rest])
        assert np.isnan(y[m2 + 1]).all()
    assert np.isnan(got.pos.cpu().numpy()[0]).all()


@pytest.mark.parametrize("n", [700, 20_000])
@pytest.mark.parametrize("where", ["new", "previous"])
def test_frame(env, n, where):
    import torch
    pbr, R = env
    a = _cloud(n)
    p2 = torch.from_numpy(a[0][::-1].copy()).cuda() + 0.001
    prev = pbr.Scene(*a, 1)
    bad = 17
    (p2 if where == "new" else prev.pos)[bad, 0] = float("nan")
    loss, g, nn12, nn21 = pbr.chamfer(R, prev.pos, p2)
    assert torch.isnan(loss)
    lost = nn21 if where == "new" else nn12
    assert (lost < 0).nonzero().view(-1).tolist() == [bad]
    ok = torch.ones(n, dtype=torch.bool, device="cuda")
    if where == "new":
        ok[bad] = False
        assert torch.isnan(g[bad]).all()
    assert torch.isfinite(g[ok]).all()
    sc, hist = pbr.frame_init(R, prev, p2, iters=3, k=4)
    assert np.isnan(hist).all()
    assert torch.isfinite(sc.pos[ok]).all() and torch.isfinite(sc.sh[ok]).all()
    if where == "new":
        assert torch.isnan(sc.sh[bad]).all()
