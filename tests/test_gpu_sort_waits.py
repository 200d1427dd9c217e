"""The one-sweep radix sort when a block does not wait for the counts of the
blocks before it, or hardly: it counts their keys itself, and the sort is the
stable sort whatever the order in which the blocks run.  Sizes at the edges of
the small (1024 keys) and large (4096) tiles, of the switch between them (2^17)
and of the one-sweep sort (2^22); exact comparison."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sort():
    import torch

    import __graft_entry__ as g
    g.build()
    from paper_2205_14330_gb300 import pbr
    f = pbr.lib().pbr_test_sort_pairs
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_int64, C.c_int32, C.c_int32, C.c_void_p]

    def run(keys, bits, polls):
        k = torch.from_numpy(keys.view(np.int32)).cuda()
        v = torch.arange(len(keys), dtype=torch.int32, device="cuda")
        s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert f(k.data_ptr(), v.data_ptr(), len(keys), bits, polls, s) == 0
        torch.cuda.synchronize()
        return k.cpu().numpy().view(np.uint32), v.cpu().numpy()
    return run


@pytest.mark.parametrize("n", [1, 1023, 1025, 4097, 131071, 131073, 1_000_001, 1 << 22])
@pytest.mark.parametrize("polls", [0, 1, 1 << 22])
@pytest.mark.parametrize("dist,bits", [("uniform", 32), ("uniform", 17), ("few", 9), ("equal", 12)])
def test_the_order_does_not_hang_on_the_wait(sort, n, polls, dist, bits):
    rng = np.random.default_rng(n)
    keys = {"uniform": lambda: rng.integers(0, 1 << bits, n, dtype=np.uint64),
            "few": lambda: rng.choice(np.uint64([0, 1, 300, 511]), n),
            "equal": lambda: np.full(n, 77, np.uint64)}[dist]().astype(np.uint32)
    order = np.argsort(keys, kind="stable")
    k, v = sort(keys, bits, polls)
    assert np.array_equal(v, order) and np.array_equal(k, keys[order])
