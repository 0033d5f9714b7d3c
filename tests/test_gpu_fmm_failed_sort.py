"""The gather after a radix sort that gave up (GPU): the order's unwritten entries are any numbers.

The kernel's own bounds check turns them into the failed-build flag.
"""
import ctypes

import pytest

from paper_2604_05982_gb300 import gtap as G

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _gather(order):
    fn = G.load_library().gtap_debug_fmm_gather
    fn.restype, fn.argtypes = ctypes.c_int, [ctypes.c_void_p] * 3 + [ctypes.c_int64] + [ctypes.c_void_p] * 2
    n = len(order)
    pos = torch.arange(3 * n, dtype=torch.float64, device="cuda")
    q = torch.arange(n, dtype=torch.float64, device="cuda") - 0.5
    idx = torch.tensor(order, dtype=torch.int64).to(torch.int32).cuda()   # (wraps to the unsigned bit pattern)
    pts = torch.full((n, 4), -7.0, dtype=torch.float64, device="cuda")
    flags = torch.zeros(4, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert fn(pos.data_ptr(), q.data_ptr(), idx.data_ptr(), n, pts.data_ptr(), flags.data_ptr()) == 0
    return pts.cpu(), int(flags[1])


def test_order_entries_out_of_range_are_flagged_and_skipped():
    n = 1000
    order = list(reversed(range(n)))
    pts, failed = _gather(order)
    want = torch.tensor([[3.0 * i, 3.0 * i + 1, 3.0 * i + 2, i - 0.5] for i in order], dtype=torch.float64)
    assert failed == 0 and torch.equal(pts, want)
    for k, bad in ((0, n), (17, 0xFFFFFFFF), (999, 0x80000000), (500, 123456789)):
        order[k] = bad
        want[k] = -7.0
    pts, failed = _gather(order)
    assert failed == 1 and torch.equal(pts, want)
