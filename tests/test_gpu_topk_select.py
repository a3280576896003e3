"""Top-K selection kernels on distance rows with ties, infinities, NaN and sizes around the block
and candidate limits: the (distance, index) order of a stable sort of the float bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 31, 33, 255, 257, 1024, 1025, 2048, 4095, 4096, 4097, 20001, 131072])
@pytest.mark.parametrize("kind", ["random", "ties", "equal", "special", "ascending"])
def test_selection_order(n, kind):
    import torch

    import paper_1812_02091_gb300 as emd
    rng = np.random.Generator(np.random.PCG64(n + len(kind)))
    rows = 3
    t = rng.random((rows, n), dtype=np.float32)
    if kind == "ties":
        t = np.floor(t * 4).astype(np.float32)
    elif kind == "equal":
        t[:] = 0.25
    elif kind == "special":
        t[rng.random(t.shape) < 0.3] = np.inf
        t[rng.random(t.shape) < 0.2] = np.nan
    elif kind == "ascending":
        t = np.sort(t, axis=1)[:, ::-1].copy()
    dev = torch.from_numpy(t).cuda()
    keys = np.abs(t).view(np.uint32).astype(np.uint64) << np.uint64(32) | np.arange(n, dtype=np.uint64)[None]
    for K in (1, 5, 16, 17, 32, 33, 64):
        if K > n:
            continue
        idx = torch.empty(rows, K, dtype=torch.int64, device="cuda")
        dist = torch.empty(rows, K, device="cuda")
        emd.emd_topk_select_static(dev, K, idx, dist)
        torch.cuda.synchronize()
        want = np.sort(keys, axis=1)[:, :K]
        np.testing.assert_array_equal(idx.cpu().numpy(), (want & np.uint64(0xffffffff)).astype(np.int64))
        np.testing.assert_array_equal(dist.cpu().numpy().view(np.uint32), (want >> np.uint64(32)).astype(np.uint32))
