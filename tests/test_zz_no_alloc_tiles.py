"""The allocation-free projection over more tiles (8192 rows each) than thread blocks fit
on the GPU at once, and around the ends of tiles and of the groups of 16 tiles that
are counted together.  Rows must equal numpy's, in order, on consecutive calls
over the one scratch array, also after a call that overflowed."""
import ctypes

import numpy as np
import pytest

from paper_1709_00700_gb300 import pv

pytestmark = pytest.mark.gpu


def _call(lib, dev, n, bounds, capacity):
    import torch
    out_a = torch.empty(max(capacity, 1), dtype=torch.int32, device="cuda")
    out_p = torch.empty(max(capacity, 1), dtype=torch.int64, device="cuda")
    count = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 12345, dtype=torch.int32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.pv_filter_project_noalloc(p(dev["a"]), p(dev["b"]), p(dev["price"]), n, *bounds, p(out_a), p(out_p),
                                         capacity, p(count), p(status),
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    k = int(count.item())
    return int(status.item()), k, out_a[:max(k, 0)].cpu().numpy(), out_p[:max(k, 0)].cpu().numpy()


@pytest.mark.parametrize("n", [1, 8192, 8193, 16 * 8192, 16 * 8192 + 1, 311_297, 16_000_003])
def test_tiles(n):
    import torch
    lib = pv.load()
    r = np.random.default_rng(n)
    a, b = (r.integers(0, 100, n).astype(np.int32) for _ in range(2))
    price = r.integers(100, 10**7, n).astype(np.int64)
    dev = {"a": torch.from_numpy(a).cuda(), "b": torch.from_numpy(b).cuda(), "price": torch.from_numpy(price).cuda()}
    for a_hi, b_hi in ((0, 0), (1, 40), (49, 60), (99, 99), (-1, 99)):
        hit = (a <= a_hi) & (b <= b_hi)
        m = int(hit.sum())
        for cap in (n, m // 2):
            status, k, ga, gp = _call(lib, dev, n, (0, a_hi, 0, b_hi), cap)
            assert status == (0 if m <= cap else -7) and k == min(m, cap)
            assert np.array_equal(ga, a[hit][:cap]) and np.array_equal(gp, price[hit][:cap])
