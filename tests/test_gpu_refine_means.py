"""Parameter means and copies of the coarse-to-fine update, which read several
points at a time: voxels of every small size, every small neighbour count and
point counts that are no multiple of a warp's share."""
import numpy as np
import pytest

from oracle import refine_ref as RR
from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu

# a compensated fp32 sum is off by 2u of the sum of magnitudes, the division
# and the stored value by u each (u = 2^-24)
MEAN_TOL = 4 * 2.0 ** -24


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _rows(d):
    n = len(d["pos"])
    return np.concatenate([np.asarray(d["pos"]).reshape(n, 3), np.asarray(d["sh"]).reshape(n, -1),
                           np.asarray(d["opacity"]).reshape(n, 1),
                           np.asarray(d["radius"]).reshape(n, 1)], 1).astype(np.float32)


def _run(env, d, **kw):
    pbr, r = env
    out, counts = pbr.refine_points(r, pbr.Scene(d["pos"], d["sh"], d["opacity"], d["radius"],
                                                 d["deg"]), **kw)
    return _rows({k: getattr(out, k).cpu().numpy() for k in ("pos", "sh", "opacity", "radius")}), \
        counts


@pytest.mark.parametrize("n,deg,n_vox", [(1, 0, 4), (9, 3, 1), (2501, 0, 12), (4003, 3, 24)])
def test_voxel_means(env, n, deg, n_vox):
    d = scenes.refine_cloud(seed=n, n=n, n_shapes=3, outlier_frac=0.05, deg=deg)
    got, _ = _run(env, d, n_vox=n_vox, stages=1)
    rows = _rows(d).astype(np.float64)
    ids = RR.voxel_ids(d["pos"], n_vox)
    order = np.argsort(ids, kind="stable")
    starts = np.flatnonzero(np.r_[True, np.diff(ids[order]) != 0])
    cnt = np.diff(np.r_[starts, n])[:, None]
    mean = np.add.reduceat(rows[order], starts, axis=0) / cnt
    scale = np.add.reduceat(np.abs(rows[order]), starts, axis=0) / cnt
    assert got.shape == mean.shape
    assert (np.abs(got - mean) <= MEAN_TOL * scale).all()


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 7, 9, 17, 32])
def test_generated_means(env, k):
    d = scenes.refine_cloud(seed=k, n=1203, n_shapes=3, outlier_frac=0.02, deg=k % 4)
    got, counts = _run(env, d, k=k, stages=4)
    rows = _rows(d).astype(np.float64)
    n = len(rows)
    assert counts[2] == 2 * n
    assert np.array_equal(got[:n], _rows(d))
    idx, _ = RR.knn(d["pos"], k)
    mean, scale = rows[idx].mean(1), np.abs(rows[idx]).mean(1)
    assert (np.abs(got[n:] - mean) <= MEAN_TOL * scale).all()


@pytest.mark.parametrize("n", [2, 31, 33, 1501])
def test_survivors_are_copied(env, n):
    d = scenes.refine_cloud(seed=n, n=n, n_shapes=2, outlier_frac=0.3, deg=3)
    eps = float(np.median(RR.outlier_delta(d["pos"], 4)[0]))
    got, counts = _run(env, d, k=4, eps=eps, stages=2)
    rows = _rows(d)
    assert 0 < counts[1] <= n and len(got) == counts[1]
    at = -1
    for row in got:  # an ordered subsequence of the input, bit for bit
        at = next(i for i in range(at + 1, n) if np.array_equal(rows[i], row))
