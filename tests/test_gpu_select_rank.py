"""Selection by counted ranks (small vocabularies) at the edges of a CTA's ids, of the one-id and two-id instances and of the cluster
kernel's range, with ties throughout, counts that fp32 does not hold, and every kind of K.  Integer work: the tolerance is zero."""
import pytest
import torch

import paper_2506_22694_b200 as vt

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _check(V, counts):
    order = torch.argsort(counts, descending=True, stable=True).to(torch.int32)
    stored = torch.where(counts >= 1 << 31, counts - (1 << 32), counts).to(torch.int32)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_SELECT_TOPK, 0, V, V))
    for K in sorted({1, V // 4 + 1, V - 1, V} - {0}):
        map_, inv = vt.vt_select_topk(stored, K, ws=ws)
        assert torch.equal(map_, order[:K])
        want = torch.full((V,), -1, dtype=torch.int32, device=DEV)
        want[order[:K].long()] = torch.arange(K, dtype=torch.int32, device=DEV)
        assert torch.equal(inv, want)
    assert ws.read_status() == (0, 0, 0)


@pytest.mark.parametrize("V", [1, 2, 31, 32, 33, 127, 128, 129, 1000, 4096, 4735, 4736, 4737, 4800, 9471, 9472, 9473])
@pytest.mark.parametrize("top", [1, 3, 1 << 20, (1 << 24) - 1, 1 << 24, (1 << 32) - 1])
def test_ranks_match_a_stable_sort(V, top):
    g = torch.Generator(device=DEV).manual_seed(V + top)
    counts = torch.randint(0, top + 1, (V,), generator=g, device=DEV, dtype=torch.int64)
    counts[torch.randint(0, V, (V // 3 + 1,), generator=g, device=DEV)] = top           # many ids tie at the top
    counts[torch.randint(0, V, (V // 5 + 1,), generator=g, device=DEV)] = max(top - 1, 0)
    _check(V, counts)


@pytest.mark.parametrize("V", [5, 64, 130, 4736, 4737, 9472])
@pytest.mark.parametrize("share", [0.002, 0.5, 1.0])
def test_counts_that_fp32_rounds_to_the_same_value(V, share):
    """Neighbours from 2^24 on, among counts below it: some, half, all of the ids."""
    g = torch.Generator(device=DEV).manual_seed(V)
    counts = torch.randint(0, 50, (V,), generator=g, device=DEV, dtype=torch.int64)
    counts[::7] = (1 << 24) - 1
    base = torch.tensor([(1 << 24) - 2, 1 << 24, 1 << 25, (1 << 31) - 3, (1 << 32) - 600], device=DEV)
    large = torch.rand(V, generator=g, device=DEV) < share
    large[V // 2] = True
    some = base[torch.randint(0, 5, (V,), generator=g, device=DEV)] + torch.randint(0, 6, (V,), generator=g, device=DEV)
    _check(V, torch.where(large, some, counts))
