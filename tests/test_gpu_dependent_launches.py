"""What a launch that takes its seats early may find of the work in front of it."""
import pytest
import torch

import paper_2506_22694_b200 as vt
import vt_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("between", [False, True])
def test_the_gather_does_not_let_a_head_call_in_before_its_rows_are_written(between):
    """An overlapped head call behind vt_trim_head breaks the caller's promise about W_trim, but the gather keeps the launch
    gate shut: the head fetches the new rows, also with a small dependent launch in between."""
    V, K, d, topk = 40_000, 20_000, 1536, 8
    fulls = [vt_inputs.gaussian_bf16((V, d), 0.02, seed=5 + i, device=DEV) for i in range(2)]
    m = torch.randperm(V, device=DEV)[:K].to(torch.int32)
    h = vt_inputs.gaussian_bf16((1, d), 1.0, seed=9, device=DEV)
    T = torch.ones(1, device=DEV)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, 1, topk))
    pool = vt.tree_pool(64)
    pool[2].zero_(), pool[1].fill_(-1), pool[0].zero_()
    want = [vt.vt_draft_head(h, vt.vt_trim_head(W, m), m, T, topk, ws=ws) for W in fulls]
    buf = torch.zeros((K, d), dtype=torch.bfloat16, device=DEV)
    torch.cuda.synchronize()
    got = []
    for i in range(20):
        vt.vt_trim_head(fulls[i & 1], m, W_trim=buf)
        if between:
            vt.vt_tree_rerank(pool, 64, 8)
        got.append(vt.vt_draft_head(h, buf, m, T, topk, ws=ws, overlapped=True))
    torch.cuda.synchronize()
    for i, (ids, lps) in enumerate(got):
        assert torch.equal(ids, want[i & 1][0]) and torch.equal(lps, want[i & 1][1])


@pytest.mark.parametrize("B", [1, 10, 100])
def test_ids_of_a_head_call_are_counted_right_behind_it(B):
    """Accumulating into the counts of a small vocabulary (one kernel, no clear in front) while the head's merge, which lets the
    next launch in with its first instruction, still writes the ids: every step's ids once, those of other buffers never."""
    K, d, topk, steps = 5000, 512, 8, 200
    W = vt_inputs.gaussian_bf16((K, d), 0.02, seed=21, device=DEV)
    hs = [vt_inputs.gaussian_bf16((B, d), 1.0, seed=30 + i, device=DEV) for i in range(4)]
    T = torch.ones(B, device=DEV)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    wsc = vt.Workspace(max(256, vt.workspace_bytes(vt.VT_OP_HISTOGRAM, B * (1 + topk), K)))
    want = torch.zeros(K, dtype=torch.int64, device=DEV)
    for i in range(steps):
        ids = vt.vt_draft_head(hs[i % 4], W, None, T, topk, ws=ws)[0]
        torch.cuda.synchronize()
        want += torch.bincount(ids.flatten().long(), minlength=K)
    out = (torch.empty((B, 1 + topk), dtype=torch.int32, device=DEV), torch.empty((B, 1 + topk), device=DEV))
    counts = torch.zeros(K, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    for i in range(steps):                                             # the same buffer every step: a stale line would be the step's before
        vt.vt_draft_head(hs[i % 4], W, None, T, topk, ws=ws, out=out, overlapped=True)
        vt.vt_histogram(out[0], K, counts=counts, accumulate=True, ws=wsc)
    torch.cuda.synchronize()
    assert torch.equal(counts.long(), want)
