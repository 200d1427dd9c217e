"""The training-step kernels at the edges of their work split: image heights
around a multiple of the rows a thread takes, single rows, columns and pixels,
and optimiser arrays of every length modulo four and every alignment."""
import numpy as np
import pytest

from oracle import train_ref as TR
from paper_2205_14330_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pbr():
    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr as m
    return m


@pytest.mark.parametrize("lam", [0.0, 0.25])
@pytest.mark.parametrize("kind", ["l2", "l1"])
@pytest.mark.parametrize("sizes", [[(1, 1)], [(1, 9)], [(9, 1)], [(3, 2), (1, 3), (2, 4)],
                                   [(17, 5), (1, 1), (86, 7), (5, 8)], [(700, 463)]])
def test_loss_tv_sizes(pbr, sizes, kind, lam):
    """Per element: 2 (a - t) has one rounding of a number below 1, the TV
    signs are exact, their sum one more: below 4 x 2^-24.  The loss's terms
    are non-negative with three roundings each and are summed with
    compensation: below 4 x 2^-24 of itself."""
    import torch
    cams = [scenes.camera((0, 0, 2), w, h) for w, h in sizes]
    n = sum(w * h for w, h in sizes)
    rng = np.random.default_rng(11)
    pred = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    tgt = rng.uniform(0, 1, (n, 3)).astype(np.float32)
    pred[::5] = tgt[::5]  # signs of zero
    lam = float(np.float32(lam))
    loss, grad = pbr.image_loss_tv(torch.from_numpy(pred).cuda(), torch.from_numpy(tgt).cuda(),
                                   cams, lam, kind)
    ref_loss, ref_grad = TR.batch_loss_and_grad(pred, tgt, sizes, lam, kind)
    assert abs(loss.item() - ref_loss) <= 4 * 2.0 ** -24 * ref_loss
    assert np.abs(grad.cpu().numpy() - ref_grad).max() <= 4 * 2.0 ** -24


@pytest.mark.parametrize("kind", ["sgd", "adam"])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1026, 700_003])
def test_optimizer_lengths_and_alignments(pbr, n, kind):
    """An element's update does not depend on how its array is accessed: the
    same bits at every alignment, and nothing written outside."""
    import torch
    gen = torch.Generator().manual_seed(n)
    src = [torch.randn(n, generator=gen), torch.randn(n, generator=gen),
           0.1 * torch.randn(n, generator=gen), torch.rand(n, generator=gen)]
    results = []
    for offs in ((0, 0, 0, 0), (1, 1, 1, 1), (0, 0, 0, 2), (3, 0, 0, 0)):
        buf = [torch.full((n + 8,), 7.0, device="cuda") for _ in src]
        arr = [b[o:o + n] for b, o in zip(buf, offs)]
        for a, x in zip(arr, src):
            a.copy_(x)
        for t in (3, 4):
            pbr.optimizer_step(arr[0], arr[1], arr[2], arr[3], lr=3e-3, step=t, kind=kind)
        for b, o in zip(buf, offs):
            assert bool((b[:o] == 7).all()) and bool((b[o + n:] == 7).all())
        results.append([a.cpu() for a in arr])
    for r in results[1:]:
        for a, b in zip(r, results[0]):
            assert torch.equal(a, b)
    p, m, v = (src[i].double().numpy() for i in (0, 2, 3))
    g = src[1].double().numpy()
    for t in (3, 4):
        if kind == "adam":
            p, m, v = TR.adam_step(p, g, m, v, t, 3e-3)
        else:
            p = TR.sgd_step(p, g, 3e-3)
    # two steps, each rounding p (|p| < 8) and an increment of below 0.2 made
    # of a dozen roundings
    assert np.abs(results[0][0].numpy() - p).max() <= 2 * (8 * 2.0 ** -24 + 0.2 * 16 * 2.0 ** -24)
