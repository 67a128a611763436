"""The streaming head at the edges of its tiling: 128 vocabulary rows per tile, phases of eight 64-column steps of d,
ring stages of up to four steps, 8 / 16 / 32 hidden rows per variant (64: over large heads only, tested with those),
full and growing candidate lists."""
import pytest
import torch

import paper_2506_22694_b200 as vt
import vt_inputs
from parity_util import check_head, oracle_head

pytestmark = pytest.mark.gpu
DEV = "cuda"
SMS = 148                                                # one slab per SM: K = SMS * 128 fills one tile per slab


@pytest.mark.parametrize("B,K,d,topk,sample", [
    (8, SMS * 128, 64, 8, True), (1, SMS * 128 + 1, 72, 33, True), (9, SMS * 128 - 1, 512, 64, False),   # tile edges, one phase
    (16, SMS * 256 + 1, 520, 10, True), (2, 7, 576, 7, True), (3, SMS * 8 + 3, 4096, 64, True),          # two phases; tiny slabs
    (17, 2000, 520, 16, True), (32, SMS * 128 + 1, 448, 1, False), (33, 3001, 1032, 16, True),           # last streaming row counts
    (64, SMS * 128 + 3, 264, 8, True), (65, 1500, 136, 8, True),                                         # and batched ones
])
def test_streaming_head_at_tile_phase_and_variant_edges(B, K, d, topk, sample):
    W = vt_inputs.gaussian_bf16((K, d), 0.05, seed=K + d, device=DEV)
    h = vt_inputs.gaussian_bf16((B, d), 1.0, seed=B + 5, device=DEV)
    T = vt_inputs.temperatures(B, 0.5, 1.5, seed=K, device=DEV)
    u = vt_inputs.uniforms((B, K), seed=d + 1, device=DEV) if sample else None
    m = torch.randperm(K * 2, device=DEV)[:K].to(torch.int32)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    gi, gl, lg, lse = vt.vt_draft_head(h, W, m, T, topk, u, ws=ws, debug=True)
    torch.cuda.synchronize()
    check_head(oracle_head(h, W, m, T, topk, u), gi, gl, T, m, lg, lse, sampled=sample)
    # fp32 accumulation split over many accumulators: 2^-24 per rounding on partial sums no larger than sum |w h|, eight
    # phases of three pairwise levels and one addition each behind chains of at most four 16-column products
    exact = h.double() @ W.double().t()
    bound = (h.double().abs() @ W.double().abs().t()) * 2.0 ** -24 * 16
    if B <= 16:
        assert bool(((lg.double() - exact).abs() <= bound).all())
    a = vt.vt_draft_head(h, W, m, T, topk, u, ws=ws)
    b = vt.vt_draft_head(h, W, m, T, topk, u, ws=ws, overlapped=True)
    torch.cuda.synchronize()
    for o in (a, b):                                     # without the logits dump, plain and chained: the same bits
        assert torch.equal(o[0], gi) and torch.equal(o[1], gl)
    assert ws.read_status() == (0, 0, 0)


@pytest.mark.parametrize("B,K,d,topk", [(1, 5000, 2048, 8), (8, 3000, 512, 10), (20, 4000, 1024, 8)])
def test_an_expired_wait_with_every_copy_already_asked_for(B, K, d, topk):
    """A CTA's whole share fits its ring: the producer has made its last request by the time a wait of another role expires
    (bound of 1 ns, set by the host), and still nothing may be in flight when the CTA leaves.  The calls right behind it
    use the same shared memory and must return what an undisturbed call does."""
    W = vt_inputs.gaussian_bf16((K, d), 0.02, seed=31, device=DEV)
    h = vt_inputs.gaussian_bf16((B, d), 1.0, seed=32, device=DEV)
    T = vt_inputs.temperatures(B, 1.0, 1.0, 0, device=DEV)
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    good = tuple(t.clone() for t in vt.vt_draft_head(h, W, None, T, topk, ws=ws))
    for overlapped in (False, True):
        ws.set_wait_limit(1)
        gi, gl = vt.vt_draft_head(h, W, None, T, topk, ws=ws, overlapped=overlapped)
        ws.set_wait_limit(0)
        after = [vt.vt_draft_head(h, W, None, T, topk, ws=ws, overlapped=overlapped) for _ in range(3)]
        st, flags, _ = ws.read_status()
        assert st == 5 and flags & vt.VT_FLAG_TIMEOUT    # (every role reads the bound before its first wait)
        assert bool((gi == -1).all()) and bool(torch.isnan(gl).all())
        for ids, lps in after:
            assert torch.equal(ids, good[0]) and torch.equal(lps, good[1])
    assert ws.read_status() == (0, 0, 0)
