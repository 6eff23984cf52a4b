"""In-cell order of cells above 8192 entries (chunks in order, then merged):
whole numbers, compared exactly with numpy's stable sort, and the time of one
such cell against that of the chunks it is made of."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHUNK = 8192


def _sort(keys, ncells, reps=0):
    import torch

    import paper_2506_23917_gb300 as sp

    k = torch.from_numpy(keys.view(np.int32)).cuda()
    start = torch.zeros(ncells + 1, dtype=torch.int32, device="cuda")
    perm = torch.full((len(keys),), -7, dtype=torch.int32, device="cuda")
    ms = []
    for _ in range(1 + reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        sp.sort_cells_static(k.data_ptr(), len(keys), ncells, start.data_ptr(), perm.data_ptr(),
                             sp.current_stream())
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    return start.cpu().numpy(), perm.cpu().numpy(), min(ms)


@pytest.mark.parametrize("order", ["random", "sorted", "reversed"])
@pytest.mark.parametrize("sizes", [
    [CHUNK + 1], [2 * CHUNK - 1, 2 * CHUNK, 2 * CHUNK + 1], [3 * CHUNK, 0, 3 * CHUNK + 1, 5, CHUNK],
    [40001, 1, 20000, 1025, 8193], [5 * CHUNK - 2049, 5 * CHUNK + 2049], [16 * CHUNK + 7], [1 << 20]])
def test_order_above_a_chunk(sizes, order):
    rng = np.random.Generator(np.random.PCG64(3))
    keys = np.repeat(np.arange(len(sizes), dtype=np.uint32), sizes)
    if order == "random":
        rng.shuffle(keys)
        keys[rng.random(len(keys)) < 0.001] = 0xFFFFFFFF
    elif order == "reversed":
        keys = keys[::-1].copy()
    start, perm, _ = _sort(keys, len(sizes))
    kept = np.flatnonzero(keys < len(sizes))
    want = kept[np.argsort(keys[kept], kind="stable")]
    assert np.array_equal(start[1:], np.cumsum(np.bincount(keys[kept], minlength=len(sizes))))
    assert np.array_equal(perm[: len(want)], want)
    assert np.all(perm[len(want):] == -7)


def test_time_of_a_dense_cell():
    """One cell of 12 chunks is ordered by one block: its chunks one by one,
    then, for each of 4 doublings, every chunk once more and the stages across
    chunks (10 in all, each a pass over the cell that compares once).  A merge
    of a chunk compares 13 times against the 91 of a full network, a pass
    once: 12 + 4 x 12 x 13 / 91 + 10 x 12 / 91 < 21 chunks' time, to which the
    passes over global memory may add as much again; 12 cells of one chunk
    are ordered side by side in one chunk's time.  (The network over all of
    the cell in global memory takes 153 passes.)"""
    rng = np.random.Generator(np.random.PCG64(4))
    one = rng.permutation(np.repeat(np.arange(12, dtype=np.uint32), CHUNK))
    _, _, t12 = _sort(one, 12, reps=10)
    _, _, t1 = _sort(np.zeros(12 * CHUNK, dtype=np.uint32)[rng.permutation(12 * CHUNK)], 1, reps=10)
    assert t1 < 42 * t12, (t1, t12)
