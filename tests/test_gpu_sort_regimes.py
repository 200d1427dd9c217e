"""The radix sort's regimes (one sweep with small and with large tiles, three
kernels a pass) against one another: the tile lists of a view must be the same,
entry by entry, whether the view is rendered alone or in a batch whose sorts
are long enough for another regime.  (tile, depth, point) order is checked
against the oracle elsewhere, on small scenes.  Sizes lie at the edges of the
sort tiles (1024 and 4096 keys) and of the regimes (2^17 and 2^22)."""
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


def _lists(st, n, views, cam):
    """[(tile keys, point indices) of each view], ids relative to the view."""
    info = st.info()
    keys, vals, rng = st.read("tile_keys"), st.read("tile_vals"), st.read("ranges")
    per = info["n_tiles"] // views
    out = []
    for v in range(views):
        r = rng[v * per:(v + 1) * per]
        r = r[r[:, 1] > r[:, 0]]
        a, b = (int(r[:, 0].min()), int(r[:, 1].max())) if len(r) else (0, 0)
        out.append((keys[a:b] - np.uint32(v * per << 4), vals[a:b] - np.uint32(v * n)))
    return out


@pytest.mark.parametrize("n,views", [(1023, 3), (1024, 5), (1025, 130), (4097, 33), (65536, 2),
                                     (131071, 2), (131073, 33), (524_288, 9), (1_000_001, 5)])
@pytest.mark.parametrize("far", [False, True], ids=["all-visible", "mostly-culled"])
def test_a_view_alone_and_in_a_batch(env, n, views, far):
    pbr, R = env
    rng = np.random.default_rng(n)
    pos = rng.uniform(-1.0, 1.0, (n, 3)).astype(np.float32)
    if far:  # most points behind the camera: compacted before the sort
        pos[rng.random(n) < 0.6] += np.float32([0, 0, 9.0])
    pos[: n // 8] = pos[n // 8: 2 * (n // 8)]  # equal depths: the lower index first
    sc = pbr.Scene(pos, np.full((n, 1, 3), 1.0, np.float32), np.full(n, 0.5, np.float32),
                   scenes.log_uniform(rng, n, 0.002, 0.02), 0)
    cam = scenes.camera((0.0, 0.0, 3.0), 240, 176)
    _, st = R.forward([sc], [cam], pbr.default_opts(bwd_mode=1))
    one = _lists(st, n, 1, cam)[0]
    st.close()
    _, st = R.forward([sc], [cam] * views, pbr.default_opts(bwd_mode=1))
    many = _lists(st, n, views, cam)
    assert st.info()["n_visible"] % views == 0
    st.close()
    assert len(one[0]) > 0
    for k, v in many:
        assert np.array_equal(k, one[0]) and np.array_equal(v, one[1])
