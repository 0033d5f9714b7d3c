"""Cilksort's serial leaves at the edges of their networks and merge windows (GPU).

Leaf ranges of 31..65 keys (the 32- and 64-key networks and the insertion sort above them), merges
around the eight-key window, and keys equal to the padding value.
"""
import numpy as np
import pytest

from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 129, 4099])
@pytest.mark.parametrize("sort_cutoff,merge_cutoff", [(1, 1), (31, 8), (64, 9), (65, 256), (256, 1 << 20)])
def test_leaf_edges(n, sort_cutoff, merge_cutoff):
    keys = inputs.keys_u32(n, seed=n)
    keys[::3] = 0xFFFFFFFF
    keys[1::5] = 0
    src = torch.from_numpy(keys.view(np.int32)).cuda()
    dst = torch.full_like(src, -1)
    tmp = torch.empty_like(src)
    torch.cuda.synchronize()
    runner.cilksort_ptrs(src.data_ptr(), dst.data_ptr(), tmp.data_ptr(), n, sort_cutoff, merge_cutoff,
                         pool_bytes=1 << 24, grid_blocks=8)
    assert np.array_equal(dst.cpu().numpy().view(np.uint32), np.sort(keys))
