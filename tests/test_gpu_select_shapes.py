"""Global mask selection at the edges of its launch rules: one block and several, rows cut into segments, rows that do not
fit into shared memory, ragged row lengths (masks that start off a 16-byte boundary), ties across blocks, every k."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def reference(loss, order, k):
    R, d = loss.shape
    key = np.maximum.accumulate(loss, axis=1)
    row = np.repeat(np.arange(R), d)
    first = np.argsort(key.ravel(), kind="stable")[:k]      # ties: lowest row, then step
    counts = np.bincount(row[first], minlength=R)
    mask = np.ones((R, d), np.uint8)
    for r in range(R):
        mask[r, order[r, :counts[r]]] = 0
    return counts, mask


@pytest.mark.parametrize("R,d", [(1, 1), (3, 7), (32, 64), (200, 576), (149, 301), (3000, 37), (5, 5120), (8000, 1000), (40000, 9)])
@pytest.mark.parametrize("tied", [False, True])
def test_select_matches_sorting(R, d, tied):
    import paper_2208_11580_b200 as obc
    rng = np.random.default_rng(R * 10007 + d)
    loss = rng.random((R, d)).astype(np.float32)
    loss = np.floor(5 * loss) if tied else loss ** 2 * np.float32(1e-4) + np.linspace(0, 1, d, dtype=np.float32) ** 4
    loss[0, -1] = np.inf
    order = np.argsort(rng.random((R, d)), axis=1).astype(np.int32)
    L, P = torch.from_numpy(loss).cuda(), torch.from_numpy(order).cuda()
    for k in sorted({0, 1, R * d // 2, R * d - 1, R * d}):
        counts = torch.full((R,), -7, dtype=torch.int32, device="cuda")
        mask = torch.full((R, d), 7, dtype=torch.uint8, device="cuda")
        obc.obc_select_global_mask(L, P, k, counts, mask)
        want = reference(loss, order, k)
        assert np.array_equal(counts.cpu().numpy(), want[0])
        assert np.array_equal(mask.cpu().numpy(), want[1])
