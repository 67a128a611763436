"""Streams whose packed count wraps, counted again by ranges of 57344 bins or, from 170 million ids per further range on, by the hot /
cold kernels: both sides of the line, vocabularies at the ranges' edges, fewer clusters than ranges, odd starts, skipped ids.
Integer work: the tolerance is zero."""
import pytest
import torch

import paper_2506_22694_b200 as vt

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("V,n", [
    (57_345, 9_000), (114_688, 1_000_003), (114_689, 60_000), (128_256, 3_000_017), (172_032, 5_000_011),
    (172_033, 40_001), (655_360, 3_000_001),
    (128_256, 84_999_999), (128_256, 85_000_005),                         # the line between the two recounts
])
def test_recount_is_exact(V, n):
    g = torch.Generator(device=DEV).manual_seed(V + n)
    hot = torch.tensor([5, V // 2, V - 1], dtype=torch.int32, device=DEV)
    ids = hot[torch.randint(0, 3, (n + 3,), device=DEV, generator=g)]
    every = torch.randint(0, V, (n // 50 + 1,), device=DEV, generator=g, dtype=torch.int32)
    ids[::50][: every.numel()] = every[: ids[::50].numel()]
    ids[17::3001], ids[18::4001] = V, -7
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_HISTOGRAM, n, V))
    for off in (0, 3):
        part = ids[off:off + n]
        good = part[(part >= 0) & (part < V)]
        want = torch.bincount(good.long(), minlength=V)
        counts = vt.vt_histogram(part, V, ws=ws)
        assert torch.equal(counts.long(), want)
        assert ws.read_status()[2] == n - good.numel()
        vt.vt_histogram(part, V, counts=counts, accumulate=True, ws=ws)
        assert torch.equal(counts.long(), 2 * want)
        assert ws.read_status()[2] == n - good.numel()
