"""The in-cell order kernel at the edges of its cell-size classes (one to
32 entries per lane of a warp, one block, a network in global memory):
whole numbers, compared exactly with numpy's stable sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sort(keys, ncells):
    import torch

    import paper_2506_23917_gb300 as sp

    k = torch.from_numpy(keys.view(np.int32)).cuda()
    start = torch.zeros(ncells + 1, dtype=torch.int32, device="cuda")
    perm = torch.full((max(len(keys), 1),), -7, dtype=torch.int32, device="cuda")
    sp.sort_cells_static(k.data_ptr(), len(keys), ncells, start.data_ptr(), perm.data_ptr())
    torch.cuda.synchronize()
    return start.cpu().numpy(), perm.cpu().numpy()


SIZES = [0, 1, 2, 16, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047,
         2048, 3071, 3500, 8191, 8192, 8193]


@pytest.mark.parametrize("order", ["random", "sorted", "runs", "reversed"])
@pytest.mark.parametrize("sizes", [SIZES, SIZES[::-1], [1025] * 40 + [3] * 700, [40] * 5000])
def test_cell_order(sizes, order):
    rng = np.random.Generator(np.random.PCG64(11))
    keys = np.repeat(np.arange(len(sizes), dtype=np.uint32), sizes)
    if order == "random":
        rng.shuffle(keys)
    elif order == "reversed":
        keys = keys[::-1].copy()
    elif order == "runs":  # a moved state: entries displaced by a few hundred places, a few removed
        at = np.argsort(np.arange(len(keys)) + rng.integers(-300, 300, len(keys)), kind="stable")
        keys = keys[at]
        keys[rng.random(len(keys)) < 0.01] = 0xFFFFFFFF
    start, perm = _sort(keys, len(sizes))
    kept = np.flatnonzero(keys < len(sizes))
    want = kept[np.argsort(keys[kept], kind="stable")]
    assert np.array_equal(start[1:], np.cumsum(np.bincount(keys[kept], minlength=len(sizes))))
    assert np.array_equal(perm[: len(want)], want)
    assert np.all(perm[len(want):] == -7)
