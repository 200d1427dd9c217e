"""Visual-hull initialisation where its batching can go wrong: one view (no
survivor queue after the first group), view counts around the group sizes,
candidate limits inside a block of candidates and inside a batch, more kept
points than the first batch holds, and no point kept at all.  Compared with
the CPU oracle on the same counter-based stream: the same candidates in the
same order (positions to fp32 rounding)."""
import numpy as np
import pytest

from oracle import hull_ref as H
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


@pytest.mark.parametrize("views,n,limit", [(1, 50, 0), (2, 500, 0), (3, 700, 0), (4, 33, 5000),
                                           (5, 100_000, 70_001), (9, 300, 4096), (17, 900, 4097),
                                           (6, 4000, 0)])
def test_matches_the_oracle(env, views, n, limit):
    pbr, R = env
    h = scenes.hull_scene(seed=views, n_spheres=3, n_cams=views, width=61, height=47)
    masks = pbr.pack_masks(h["masks"])
    pos, sh, drawn = pbr.visual_hull_init(R, h["lo"], h["hi"], h["cams"], masks, n, seed=7,
                                          sh_degree=1, max_candidates=limit)
    ref, rdrawn = H.hull_init(h["lo"], h["hi"], h["cams"], h["masks"], n, 7,
                              **({"max_candidates": limit} if limit else {}))[:2]
    assert drawn == rdrawn and pos.shape == tuple(ref.shape) and sh.shape == (len(ref), 4, 3)
    assert np.abs(pos.cpu().numpy() - ref).max() <= 2.0 ** -22 * 3  # the box is 3 wide


def test_nothing_kept(env):
    pbr, R = env
    h = scenes.hull_scene(seed=1, n_spheres=1, n_cams=4, width=32, height=32)
    masks = pbr.pack_masks([m * 0 for m in h["masks"]])
    pos, sh, drawn = pbr.visual_hull_init(R, h["lo"], h["hi"], h["cams"], masks, 10, seed=2,
                                          max_candidates=200_000)
    assert len(pos) == len(sh) == 0 and drawn == 200_000
