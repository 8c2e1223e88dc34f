"""Morton keys and their stable sort (Sec. 5: particles addressed through
sorted keys) at the sizes where the sort changes its tiling or its kernel.
Integer results: the permutation is compared exactly with a stable host sort of
each point's key."""
import numpy as np
import pytest

from gpu_common import ensure_built, torch_cuda

pytestmark = pytest.mark.gpu


def keys_of(x, dtype, polls=None):
    """(keys, permutation) of fmm_build for points x."""
    torch = torch_cuda()
    ensure_built()
    from paper_1106_2176_gb300 import FMM
    from paper_1106_2176_gb300.fmm import lib
    xt = torch.tensor(x.astype(dtype), device="cuda")
    f = FMM(len(x), p=2, theta=0.5, ncrit=64)
    if polls is not None:
        assert lib().fmm_set_sort_polls(f._h, polls) == 0
    f.build(xt, torch.ones(len(x), dtype=xt.dtype, device="cuda"))
    t = f.export_tree()
    f.close()
    return t["keys"], t["perm"]


# one block, its edge and the tile edges at 1024 and 4096 keys per tile
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1025, 4095, 4096, 4097, 8191, (1 << 19) - 1, (1 << 19) + 1, (1 << 21) + 2049])
def test_sorted_stably_at_tile_edges(n):
    rng = np.random.default_rng(n)
    # clustered, with many equal keys, so that ties test the stability
    x = (rng.integers(0, 50, size=(n, 3)) / 50.0 + (rng.random((n, 3)) < 0.3) * rng.random((n, 3))).astype(np.float32)
    keys, perm = keys_of(x, np.float32)
    inv = np.empty(n, np.int64)
    inv[perm] = np.arange(n)
    assert np.array_equal(np.sort(perm), np.arange(n))
    raw = keys[inv]  # key of each input point
    assert np.array_equal(np.argsort(raw, kind="stable"), perm) and np.array_equal(np.sort(raw), keys)


# blocks that give up waiting for the ones before (at the first or second look in
# vain) count the keys themselves: the same keys and order, with tiles of 1024 and of
# 4096 keys and the last one partly filled
@pytest.mark.parametrize("polls", [0, 1])
@pytest.mark.parametrize("n", [4097, 70001, (1 << 19) + 1])
def test_sorted_stably_without_waiting_for_other_blocks(n, polls):
    rng = np.random.default_rng(n)
    x = (rng.integers(0, 50, size=(n, 3)) / 50.0 + (rng.random((n, 3)) < 0.3) * rng.random((n, 3))).astype(np.float32)
    keys, perm = keys_of(x, np.float32)
    k2, p2 = keys_of(x, np.float32, polls)
    assert np.array_equal(keys, k2) and np.array_equal(perm, p2)
