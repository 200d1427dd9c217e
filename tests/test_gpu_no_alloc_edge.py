"""pbr_render_forward_noalloc where its scratch is all but full: the sorts fall back
to the passes that need least, and the image stays the allocating forward's.  The
view's height is raised until one more row is refused: what is then left of the
scratch is less than a row's bytes, below what the faster sort would need more."""
import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(30_000, (16, 16)), (60_000, (8, 8))])
def test_the_last_rows_that_fit(n, tile):
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    rng = np.random.default_rng(n)
    scene = pbr.Scene(rng.uniform(-0.4, 0.4, (n, 3)).astype(np.float32),
                      scenes.sh_coeffs(rng, n, 0, std=0.2), np.full(n, 0.6, np.float32),
                      np.full(n, 0.01, np.float32), 0)
    opts = pbr.default_opts(tile=tile)

    def cam(h):  # the points stay in the top rows, whatever the height
        c = scenes.camera((0.0, 0.0, 2.5), 256, 256)
        c["height"] = h
        return [c]

    def fits(h):
        try:
            return pbr.render_forward_noalloc([scene], cam(h), opts)
        except pbr.PBRError as e:
            assert e.code == -4
            return None

    lo, hi = 256, 8192
    assert fits(lo) is not None and fits(hi) is None
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (mid, hi) if fits(mid) is not None else (lo, mid)
    out = fits(lo)
    ref, st = pbr.Renderer(0).forward([scene], cam(lo), opts)
    assert st.info()["n_pairs"] > n
    assert torch.equal(out.view(-1), ref.view(-1))
