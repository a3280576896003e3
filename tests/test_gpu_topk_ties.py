"""Top-K selection on rows where few values differ: a handful of finite ones among +inf (the pruned
top-K's second stage), equal values, values in order, and small values in few of a block's lanes
(more candidates than the kernel keeps).  Order as a stable sort of the float bits; rows of equal
values take about as long as others, since both are read twice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _row(kind, n, rng):
    t = rng.random(n, dtype=np.float32)
    if kind == "few_finite":
        t[rng.permutation(n)[: n - 40]] = np.inf
    elif kind == "lanes":  # three lanes of each warp: at K = 32 and 15,625 values a block 1,464 candidates
        t[np.isin(np.arange(n) % 32, (0, 11, 22))] *= np.float32(2.0 ** -20)
    elif kind == "equal_lanes":
        t[np.isin(np.arange(n) % 32, (0, 11, 22))] = 0.0
    elif kind == "descending":
        t = np.sort(t)[::-1].copy()
    return t


@pytest.mark.parametrize("n", [4095, 60000, 1000000])
@pytest.mark.parametrize("kind", ["few_finite", "lanes", "equal_lanes", "descending"])
def test_order(n, kind):
    import torch

    import paper_1812_02091_gb300 as emd
    rng = np.random.Generator(np.random.PCG64(n + len(kind)))
    t = np.stack([_row(kind, n, rng) for _ in range(2)])
    dev = torch.from_numpy(t).cuda()
    keys = t.view(np.uint32).astype(np.uint64) << np.uint64(32) | np.arange(n, dtype=np.uint64)[None]
    for K in (1, 9, 16, 24, 32):
        idx = torch.empty(2, K, dtype=torch.int64, device="cuda")
        dist = torch.empty(2, K, device="cuda")
        emd.emd_topk_select_static(dev, K, idx, dist)
        want = np.sort(np.partition(keys, K - 1, axis=1)[:, :K], axis=1)
        np.testing.assert_array_equal(idx.cpu().numpy(), (want & np.uint64(0xffffffff)).astype(np.int64))
        np.testing.assert_array_equal(dist.cpu().numpy().view(np.uint32), (want >> np.uint64(32)).astype(np.uint32))


@pytest.mark.parametrize("K", [16, 32])
def test_time_does_not_depend_on_ties(K):
    import torch

    import paper_1812_02091_gb300 as emd
    rows, n = 64, 1000000
    t = torch.rand(rows, n, device="cuda")
    idx = torch.empty(rows, K, dtype=torch.int64, device="cuda")
    dist = torch.empty(rows, K, device="cuda")

    def best(x):
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            emd.emd_topk_select_static(x, K, idx, dist)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    plain = best(t)
    for other in (torch.where(t < 1e-4, t, torch.full_like(t, float("inf"))), torch.full_like(t, 0.5)):
        assert best(other) < 2 * plain
