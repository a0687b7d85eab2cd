"""Global mask selection where a block's keys do not fit into shared memory and much of a row shares the digits decided so far
(equal losses, saturated prefix maxima): against a stable sort, as in test_gpu_select_shapes."""
import numpy as np
import pytest
import torch

from test_gpu_select_shapes import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,d", [(1, 60001), (2, 131072), (3, 70017), (50, 60003), (4000, 2100)])
@pytest.mark.parametrize("kind", ["random", "tied", "constant"])
def test_long_runs_of_equal_digits(R, d, kind):
    import paper_2208_11580_b200 as m
    rng = np.random.default_rng(R * 101 + d)
    loss = rng.random((R, d)).astype(np.float32)
    loss = np.floor(5 * loss) if kind == "tied" else np.full_like(loss, 0.25) if kind == "constant" else loss
    loss[0, 5:9] = [np.nan, -1.0, 0.0, 3e-39]
    order = np.argsort(rng.random((R, d)), axis=1).astype(np.int32)
    L, P = torch.from_numpy(loss).cuda(), torch.from_numpy(order).cuda()
    key = np.where(np.isnan(loss), np.float32(np.inf), np.maximum(loss, 0))
    for k in (1, 7, R * d // 3, R * d - 1):
        counts = torch.full((R,), -7, dtype=torch.int32, device="cuda")
        mask = torch.full((R, d), 7, dtype=torch.uint8, device="cuda")
        m.obc_select_global_mask(L, P, k, counts, mask)
        want = reference(key, order, k)
        assert np.array_equal(counts.cpu().numpy(), want[0])
        assert np.array_equal(mask.cpu().numpy(), want[1])


def test_more_keys_than_32_bits_count():
    """All losses equal: one bin of the histograms holds all 2^32 + 2^20 keys."""
    import paper_2208_11580_b200 as m
    R, d = 4097, 1 << 20
    loss = torch.full((R, d), 0.5, device="cuda")
    order = torch.arange(d, dtype=torch.int32, device="cuda").repeat(R, 1)
    counts = torch.full((R,), -7, dtype=torch.int32, device="cuda")
    mask = torch.full((R, d), 7, dtype=torch.uint8, device="cuda")
    for k in (R * d - 5, (1 << 32) + 3, 12345):
        m.obc_select_global_mask(loss, order, k, counts, mask)
        full, rest = divmod(k, d)
        want = torch.zeros(R, dtype=torch.int32, device="cuda")
        want[:full] = d
        want[full] = rest
        assert torch.equal(counts, want)
        assert bool((mask[:full] == 0).all()) and bool((mask[full + 1:] == 1).all())
        assert bool((mask[full, :rest] == 0).all()) and bool((mask[full, rest:] == 1).all())
    del loss, order, mask
    torch.cuda.empty_cache()
