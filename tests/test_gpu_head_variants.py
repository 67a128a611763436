"""Head variants that only large heads or many new nodes reach: the streaming kernel's 33-to-64-row instance, just above and just
below the size at which it takes over from the batched kernel, and the tree expansion as a kernel behind the merge."""
import pytest
import torch

import paper_2506_22694_b200 as vt
import vt_inputs
from parity_util import check_head, oracle_head

pytestmark = pytest.mark.gpu
DEV = "cuda"
MB = 1 << 20


def _inputs(B, K, d, topk, sample, seed):
    W = vt_inputs.gaussian_bf16((K, d), 0.02, seed=seed, device=DEV)
    h = vt_inputs.gaussian_bf16((B, d), 1.0, seed=seed + 1, device=DEV)
    T = vt_inputs.temperatures(B, 0.5, 1.5, seed=seed + 2, device=DEV)
    u = vt_inputs.uniforms((B, K), seed=seed + 3, device=DEV) if sample else None
    m = torch.randperm(K + 1000, device=DEV)[:K].to(torch.int32)
    return h, W, m, T, u


@pytest.mark.parametrize("B,d,mb,extra,topk,sample", [
    (33, 1032, 192, 1, 16, True), (40, 4096, 192, 1, 8, True), (48, 2056, 224, 3, 10, False),     # streaming, several tiles per slab
    (33, 1032, 192, -1, 16, True), (64, 4096, 192, -1, 8, True),                                   # one vocabulary row less: batched
    (49, 2048, 200, 5, 8, True), (64, 4104, 240, 1, 16, True),
    (17, 1032, 30, 1, 16, True), (32, 2056, 60, 7, 8, False),
])
def test_many_rows_over_large_heads(B, d, mb, extra, topk, sample):
    K = -(-mb * MB // (2 * d)) + extra - (1 if extra < 0 and (mb * MB) % (2 * d) == 0 else 0)
    h, W, m, T, u = _inputs(B, K, d, topk, sample, seed=B + d)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    gi, gl, lg, lse = vt.vt_draft_head(h, W, m, T, topk, u, ws=ws, debug=True)
    # logits against 64-bit sums: each addition in the tensor core is off by at most 2^-23 of a partial sum no larger than
    # sum |w h|, and a batched kernel's accumulator makes one per sixteen columns of d (the streaming kernel a few per phase)
    hd, Wd = h.double(), W.double()
    exact = hd @ Wd.t()
    bound = (hd.abs() @ Wd.abs().t()) * 2.0 ** -23 * (d / 16 + 2 if B > 32 else 40 + d / 512)
    err = (lg.double() - exact).abs()
    assert bool((err <= bound).all())
    # lse: a mean of the same errors, the rounding of its own size, and the sum (2^-22 per exponential, 64 additions in a row)
    want = torch.logsumexp(exact / T.double()[:, None], 1)
    slack = err.max(dim=1).values / T.double() + want.abs() * 2.0 ** -23 + 2.0 ** -22 + 64 * 2.0 ** -24
    assert bool(((lse.double() - want).abs() <= slack).all())
    # ids and log-probabilities of eight of the rows against the oracle
    rows = torch.tensor(sorted({0, 1, 7, 8, 15, B // 2, B - 2, B - 1}), device=DEV)
    ref = oracle_head(h[rows], W, m, T[rows], topk, None if u is None else u[rows])
    check_head(ref, gi[rows], gl[rows], T[rows], m, sampled=sample)
    for overlapped in (False, True):
        ids, lps = vt.vt_draft_head(h, W, m, T, topk, u, ws=ws, overlapped=overlapped)
        assert torch.equal(ids, gi) and torch.equal(lps, gl)
    assert ws.read_status() == (0, 0, 0)


@pytest.mark.parametrize("B,K,d,topk,depths", [
    (8, 33_001, 2048, 8, 4), (13, 33_001, 2048, 5, 4),   # 64 new nodes: in the merge; 65: a kernel behind it, the next depth's head behind that
    (64, 3000, 256, 8, 2), (57, 3000, 256, 9, 2), (64, 2000, 264, 16, 2),     # 512, 513 and 1024 of them
])
def test_expansion_behind_the_merge_equals_head_then_expansion(B, K, d, topk, depths):
    """Depths back to back, nothing in between: ids, log-probabilities, pool and frontier are those of the two calls."""
    h, W, m, T, u = _inputs(B, K, d, topk, True, seed=K + B)
    hs = [vt_inputs.gaussian_bf16((B, d), 1.0, seed=200 + i, device=DEV) for i in range(depths)]
    cap = B + depths * B * topk
    first = (torch.zeros(cap, dtype=torch.int32, device=DEV), torch.full((cap,), -1, dtype=torch.int32, device=DEV),
             -torch.arange(cap, dtype=torch.float32, device=DEV) / 7)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    torch.cuda.synchronize()
    results = []
    for fused in (False, True):
        pool = tuple(t.clone() for t in first)
        front = torch.arange(B, dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
        base, outs = B, []
        for i in range(depths):
            if fused:
                ids, lps, front = vt.vt_draft_head_expand(hs[i], W, m, T, topk, u, front, pool, base, B, ws=ws)
            else:
                ids, lps = vt.vt_draft_head(hs[i], W, m, T, topk, u, ws=ws)
                front = vt.vt_tree_expand(ids, lps, front, pool, base, B, col0=1)
            outs += [ids, lps.view(torch.int32), front]
            base += B * topk
        results.append(outs + [pool[0], pool[1], pool[2].view(torch.int32)])
    for a, b in zip(*results):
        assert torch.equal(a, b)
    assert ws.read_status() == (0, 0, 0)
