"""The cell sort on both sides of the scan's change from one block to three
kernels, and where its counts per thread change: keys in order, nobody lost."""
import numpy as np
import pytest

from paper_2107_01723_gb300 import hpic

pytestmark = pytest.mark.gpu


# cells rounded up to tiles of 64: 1, 63, 64 and 65 tiles (4 counts per thread, and 8),
# 255 and 256 tiles (16384 counts: the last of the short scan and the first beyond)
@pytest.mark.parametrize("n", [(4, 4, 4), (252, 4, 4), (256, 3, 2), (260, 4, 4), (60, 67, 4), (64, 62, 3)])
def test_sorted_keys(n):
    import torch
    rng = np.random.default_rng(sum(n))
    N = 50_001
    x = [torch.tensor(rng.uniform(0, m, N).astype(np.float32)).cuda() for m in n]
    u = [torch.tensor(rng.normal(size=N).astype(np.float32)).cuda() for _ in range(4)]
    ids = torch.arange(N, dtype=torch.int32).cuda()
    ids[rng.integers(0, N, 500)] = -1  # dead slots
    ins = x + u + [ids]
    outs = [torch.empty_like(v) for v in ins]
    live = torch.zeros(1, dtype=torch.int64).cuda()
    hpic.hpic_sort_cells_noalloc(*n, hpic.HPIC_FP32_MIXED, N, [v.data_ptr() for v in ins],
                                 [v.data_ptr() for v in outs], live.data_ptr())
    m = int(live.item())
    alive = (ids >= 0).cpu().numpy()
    assert m == alive.sum()
    got = [v[:m].cpu().numpy() for v in outs]
    i, j, k = (np.minimum(np.floor(v).astype(int), c - 1) for v, c in zip(got[:3], n))
    nt = [(c + 3) // 4 for c in n]
    key = (((k // 4) * nt[1] + j // 4) * nt[0] + i // 4) * 64 + (k % 4) * 16 + (j % 4) * 4 + i % 4
    assert np.all(np.diff(key) >= 0)
    assert np.array_equal(np.sort(got[7]), np.sort(ids.cpu().numpy()[alive]))
    back = np.argsort(got[7])
    for a, b in zip(got[:7], ins[:7]):
        assert np.array_equal(a[back], b.cpu().numpy()[alive])
