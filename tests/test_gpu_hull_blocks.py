"""The visual hull's two block sizes (by the batch's) and the blocks it leaves out
once enough was found below them: the points of a small target are the first
points of a large one, and as many candidates are drawn for them.  Targets around
the blocks (1,024 and 2,048 candidates), the least batch (2^16) and the switch
between the blocks (2^21 candidates, 2^16 points).
"""
import numpy as np
import pytest

from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [None, 60.0, 25.0], ids=["all", "most", "few"])
def test_small_targets_are_prefixes(radius):
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    R = pbr.Renderer(0)
    cams = [scenes.camera((2.5 * np.cos(a), 0.4, 2.5 * np.sin(a)), 160, 120) for a in (0.0, 1.1, 2.3)]
    y, x = np.mgrid[0:120, 0:160]
    disc = np.ones((120, 160), bool) if radius is None else \
        (x - 80.0) ** 2 + (y - 60.0) ** 2 < radius ** 2
    masks = torch.from_numpy(np.concatenate([disc.reshape(-1)] * 3).astype(np.uint8)).cuda()

    def hull(n):
        return pbr.visual_hull_init(R, (-0.5,) * 3, (0.5,) * 3, cams, masks, n, seed=9, sh_degree=0)

    pos, _, drawn = hull((1 << 21) + 5000)
    assert len(pos) == (1 << 21) + 5000 and drawn >= len(pos)
    last = 0
    for n in (1, 1023, 1025, 2049, 4097, 65_535, 65_537, 300_001, (1 << 21) - 1, (1 << 21) + 1):
        p, _, d = hull(n)
        assert torch.equal(p, pos[:n])
        assert last < d <= drawn
        last = d
    R.close()
