"""The exact neighbour search at the sizes where its start changes (a thread
or a warp per query), with clouds that send queries on to the coarse grid and
to the exhaustive scan, ties, duplicates and queries far outside the grid.
Compared entry by entry with a brute-force fp32 search in PyTorch (the same
rounded operations, ties by lower index); nothing is approximate."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    r = pbr.Renderer(0)
    yield pbr, r
    r.close()


def _cloud(kind, n, seed=0):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(n, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    if kind == "outliers":  # a sphere, 2% of the points spread around it
        m = n // 50
        v[:m] = rng.uniform(-4.0, 4.0, (m, 3))
    elif kind == "ties":  # lattice points, every one at least twice
        v = np.round(v * 6.0) / 8.0
    elif kind == "clump":  # most points in one cell, a few far away
        v *= 1e-3
        v[:7] *= 1e4
    return v.astype(np.float32)


def _brute(ref, q, k, self_):
    import torch
    idx, d2 = [], []
    for a in range(0, len(q), 512):
        d = ref[None, :, :] - q[a:a + 512, None, :]
        e = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
        if self_:
            rows = torch.arange(len(e), device=e.device)
            e[rows, a + rows] = float("inf")
        s = torch.sort(e, dim=1, stable=True)
        idx.append(s.indices[:, :k].int())
        d2.append(s.values[:, :k])
    return torch.cat(idx), torch.cat(d2)


@pytest.mark.parametrize("kind", ["sphere", "outliers", "ties", "clump"])
@pytest.mark.parametrize("n,k,grid_n", [(8191, 1, 0), (8192, 1, 0), (8193, 2, 0), (16400, 3, 0),
                                        (33000, 8, 0), (16384, 1, 700), (20000, 4, 400),
                                        (9000, 1, 1)])
def test_self_search(env, kind, n, k, grid_n):
    import torch
    if kind == "clump" and n > 10_000:
        pytest.skip("one clump is every point against every other")
    pbr, R = env
    p = torch.from_numpy(_cloud(kind, n)).cuda()
    idx, d2 = pbr.knn(R, p, k, grid_n=grid_n)
    ri, rd = _brute(p, p, k, True)
    assert torch.equal(d2, rd) and torch.equal(idx, ri)


@pytest.mark.parametrize("k", [1, 7, 12, 16])
@pytest.mark.parametrize("shift", [0.0, 0.3, 40.0])
def test_queries_of_another_cloud(env, k, shift):
    import torch
    pbr, R = env
    ref = torch.from_numpy(_cloud("outliers", 9000, 1)).cuda()
    q = torch.from_numpy(_cloud("sphere", 4096 * max(k, 2) + 3, 2)).cuda() + shift
    idx, d2 = pbr.knn(R, ref, k, query=q)
    ri, rd = _brute(ref, q, k, False)
    assert torch.equal(d2, rd) and torch.equal(idx, ri)


@pytest.mark.parametrize("n1,n2", [(9000, 20000), (20000, 100), (8192, 8192)])
def test_chamfer_maps(env, n1, n2):
    import torch
    pbr, R = env
    p1 = torch.from_numpy(_cloud("outliers", n1, 3)).cuda()
    p2 = torch.from_numpy(_cloud("sphere", n2, 4)).cuda()
    _, _, nn12, nn21 = pbr.chamfer(R, p1, p2)
    assert torch.equal(nn12, _brute(p2, p1, 1, False)[0][:, 0])
    assert torch.equal(nn21, _brute(p1, p2, 1, False)[0][:, 0])
