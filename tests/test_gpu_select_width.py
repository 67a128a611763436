"""The selection where its cluster changes from eight to sixteen CTAs (65536 ids) and where a slice of the wide cluster
passes its sixteen-bit counters (16 * 65535 ids).  Integer work: the tolerance is zero."""
import numpy as np
import pytest
import torch

import oracle
import paper_2506_22694_b200 as vt

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("V", [65_535, 65_536, 65_537, 65_551, 131_073, 16 * 65_535, 16 * 65_535 + 1])
@pytest.mark.parametrize("shape", ["rare", "heavy", "ties"])
def test_selection_around_the_cluster_width(V, shape):
    g = torch.Generator(device=DEV).manual_seed(V % 1009)
    r = torch.rand(V, generator=g, device=DEV)
    counts = {"rare": (r * 40).int(), "heavy": (1.0 / (r + 1e-7)).clamp(max=3e8).int() + 900, "ties": (r * 3).int() * 700}[shape]
    host = counts.cpu().numpy().view(np.uint32)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_SELECT_TOPK, 0, V, V))
    for K in (1, V // 5, V - 1):
        m, inv = vt.vt_select_topk(counts, K, ws=ws)
        rm, rinv = oracle.select_topk(host, K)[:2]
        assert np.array_equal(m.cpu().numpy(), rm) and np.array_equal(inv.cpu().numpy(), rinv)
    total = int(host.astype(np.uint64).sum())
    order = np.lexsort((np.arange(V), -host.astype(np.int64)))           # count descending, id ascending
    k, m, inv = vt.vt_select_topp(counts, 0.8, ws=ws)
    want = int(np.searchsorted(np.cumsum(host[order].astype(np.uint64)), np.ceil(0.8 * float(total))) + 1)
    assert int(k) == want and np.array_equal(m[:want].cpu().numpy(), order[:want])
    k, m, inv = vt.vt_select_minfreq(counts, 20, ws=ws)
    want = max(1, int((host >= 20).sum()))
    assert int(k) == want and np.array_equal(m[:want].cpu().numpy(), order[:want])
