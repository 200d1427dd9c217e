"""The visual hull's batches of candidates: hardly more are drawn than the points
need, whatever share the masks accept, in few batches (a synchronisation each).
Host arithmetic only."""
import ctypes as C

import numpy as np
import pytest


@pytest.fixture(scope="module")
def batch():
    from paper_2205_14330_gb300 import build
    build.build()
    from paper_2205_14330_gb300 import pbr
    f = pbr.lib().pbr_test_hull_batch
    f.argtypes, f.restype = [C.c_int64] * 3, C.c_int64
    return f


@pytest.mark.parametrize("n", [65536, 65537, 200_000, 1_000_000, 30_000_000])
@pytest.mark.parametrize("share", [1.0, 0.5, 0.15, 1 / 23, 1 / 300, 1e-4])
def test_draws_and_batches(batch, n, share):
    rng = np.random.default_rng(n)
    done = drawn = batches = 0
    while done < n:
        c = batch(n, done, drawn)
        assert c % 4096 == 0 and 1 << 16 <= c <= 1 << 24
        done, drawn, batches = done + int(rng.binomial(c, share)), drawn + c, batches + 1
    most = 1.2 * n / share + (1 << 16)
    assert drawn <= most and batches <= 4 + most / (1 << 24)


def test_the_first_batch_is_what_is_needed_anyhow(batch):
    assert batch(500_000, 0, 0) == -(-500_000 // 4096) * 4096
    assert batch(10, 0, 0) == 1 << 16
    assert batch(1 << 30, 0, 0) == 1 << 24
