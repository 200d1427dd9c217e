"""Calls that return before their GPU work has run take their camera tables with
them: held up behind other work on the stream, while the host's memory is reused,
they give what they give on an idle stream."""
import ctypes as C

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


def _reuse_the_heap():
    libc = C.CDLL(None)
    libc.malloc.restype, libc.malloc.argtypes = C.c_void_p, [C.c_size_t]
    libc.free.argtypes = [C.c_void_p]
    got = []
    for size in list(range(32, 4096, 16)) + list(range(4096, 40000, 512)):
        for _ in range(8):
            p = libc.malloc(size)
            C.memset(p, 0x5A, size)
            got.append(p)
    for p in got:
        libc.free(p)


@pytest.mark.parametrize("views", [1, 4, 29, 33, 100])  # one to several pieces of 3,840 bytes
def test_tables_outlive_the_call(env, views):
    import torch
    pbr, R = env
    rng = np.random.default_rng(views)
    cams = [scenes.camera((0.1 * v, 0.3, 2.5), 20 + v % 7, 17) for v in range(views)]
    npix = pbr.n_pixels(cams)
    pred, target = torch.rand(npix, 3, device="cuda"), torch.rand(npix, 3, device="cuda")
    masks = (torch.rand(npix, device="cuda") < 0.9).to(torch.uint8)
    pos = torch.from_numpy(rng.uniform(-0.4, 0.4, (5000, 3)).astype(np.float32)).cuda()

    def calls():
        loss, grad = pbr.image_loss_tv(pred, target, cams)
        return grad, pbr.consistency_check(R, pos, cams, masks), loss

    calls()
    torch.cuda.synchronize()
    ref = calls()
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)  # some 0.2 s in front of the calls
    got = calls()
    _reuse_the_heap()
    torch.cuda.synchronize()
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    assert abs(float(got[2]) - float(ref[2])) <= 1e-12 * float(ref[2])  # fp64 atomics
