"""pbr_forward_workspace_size gives the bytes that the pass takes from the memory
pool: every buffer with its padding to 256 bytes."""
import pytest

from paper_2205_14330_gb300 import scenes
from test_zz_no_alloc import _PoolWatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,size", [(1, (1, 1)), (1001, (33, 47)), (20_003, (333, 201))])
@pytest.mark.parametrize("kw", [dict(), dict(persistent=1), dict(bwd_mode=1), dict(batch_depth=64)],
                         ids=["store", "persistent", "recompute", "staged"])
def test_the_bytes_are_those_allocated(n, size, kw):
    import numpy as np
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    rng = np.random.default_rng(n)
    R = pbr.Renderer(0)
    scene = pbr.Scene(rng.uniform(-0.5, 0.5, (n, 3)).astype(np.float32),
                      scenes.sh_coeffs(rng, n, 0, std=0.2), np.full(n, 0.5, np.float32),
                      np.full(n, 0.02, np.float32), 0)
    cams, opts = [scenes.camera((0.0, 0.0, 2.5), *size)], pbr.default_opts(**kw)
    told, _ = R.workspace_size([scene], cams, opts)
    torch.cuda.synchronize()
    watch = _PoolWatch(torch.cuda.current_device())
    before = watch.reset()
    _, st = R.forward([scene], cams, opts)
    torch.cuda.synchronize()
    used = watch.high() - before
    st.close()
    R.close()
    # four allocations, each of whole 256-byte pieces
    assert told % 256 == 0 and told <= used
