"""The batched head's epilogue against its own logits: candidate lists, sampled ids and log-probabilities recomputed from the logits
that the same call leaves, at the edges of tiles, column shares, lane quadrants and lists, with ties, infinities and NaN."""
import pytest
import torch

import paper_2506_22694_b200 as vt
import vt_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _check(h, W, T, topk, u, flags=0):
    B, K, d = h.shape[0], W.shape[0], W.shape[1]
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_DRAFT_HEAD, 0, 0, K, d, B, topk))
    ids, lps, logits, lse = vt.vt_draft_head(h, W, None, T, topk, u, ws=ws, debug=True)
    z = logits * (1.0 / T)[:, None]                                    # the kernel's own two roundings
    # candidates: by descending z, equal ones by index, NaN and -inf never.  Exact.
    ranked = torch.where(torch.isnan(z), torch.full_like(z, -float("inf")), z)
    order = torch.argsort(ranked, dim=1, descending=True, stable=True)[:, :topk]
    best = ranked.gather(1, order)
    want = torch.where(best > -float("inf"), order, torch.full_like(order, -1)).to(torch.int32)
    assert torch.equal(ids[:, 1:], want)
    got = lps[:, 1:]
    expect = torch.where(want >= 0, best - lse[:, None], torch.full_like(best, float("nan")))
    assert torch.equal(torch.isnan(got), torch.isnan(expect))
    assert torch.equal(got[~torch.isnan(got)], expect[~torch.isnan(expect)])
    if u is None:
        assert torch.equal(ids[:, 0], ids[:, 1])
    else:
        # a score is off by the fast logarithms' 2^-21 and one rounding of its own size at most
        uc = u.double().clamp(2.0 ** -24, 1 - 2.0 ** -24)
        score = ranked.double() - torch.log(-torch.log(uc))
        top = score.max(dim=1).values
        mine = score.gather(1, ids[:, :1].long().clamp(min=0))[:, 0]
        live = top > -float("inf")
        size = torch.where(torch.isfinite(ranked), ranked.abs(), torch.zeros_like(ranked)).double().amax(dim=1)
        slack = 2.0 ** -20 + size * 2.0 ** -23
        assert bool(((ids[:, 0] >= 0) == live).all())
        ok = torch.where(torch.isinf(top), top == mine, top - mine <= slack)       # (a winner of +inf: one of +inf)
        assert bool(ok[live].all())
    # a NaN logit leaves no log-sum-exp, and neither does +inf (inf - inf)
    assert torch.equal(torch.isnan(lse), (torch.isnan(z) | (z == float("inf"))).any(dim=1))
    got_flags = ws.read_status()[1]
    assert got_flags == flags, got_flags
    again = vt.vt_draft_head(h, W, None, T, topk, u, ws=ws, overlapped=True)
    assert torch.equal(again[0], ids) and torch.equal(again[1].view(torch.int32), lps.view(torch.int32))


def _inputs(B, K, d, sample, seed):
    W = vt_inputs.gaussian_bf16((K, d), 0.02, seed=seed, device=DEV)
    h = vt_inputs.gaussian_bf16((B, d), 1.0, seed=seed + 1, device=DEV)
    T = vt_inputs.temperatures(B, 0.5, 1.5, seed=seed + 2, device=DEV)
    u = vt_inputs.uniforms((B, K), seed=seed + 3, device=DEV) if sample else None
    return h, W, T, u


@pytest.mark.parametrize("B,K,d,topk,sample", [
    (33, 17, 64, 16, True), (64, 2369, 128, 8, True), (65, 2369, 128, 7, True),                  # tiles of 16 and 32 columns: one chunk, empty shares
    (40, 20_001, 256, 8, True), (63, 37_888, 64, 1, False), (64, 37_889, 64, 9, True),           # halved tiles: one per CTA, two, a last one of 17
    (48, 14_200, 512, 8, True), (40, 16_576, 64, 16, False), (50, 14_208, 1024, 7, True),        # the narrowest that are halved
    (64, 11_840, 64, 8, True), (33, 9973, 512, 16, True), (45, 3476, 512, 1, False),             # up to 64 rows in one piece
    (96, 20_004, 192, 8, True), (97, 19_999, 192, 16, True), (128, 80_001, 64, 3, True),         # three and four quadrants, three tiles and more
    (129, 2368, 128, 8, True), (129, 2369, 72, 16, True), (160, 18_944, 64, 8, False),           # pairs: second CTA with one row and with 32
    (161, 18_945, 64, 10, True), (255, 60_000, 64, 8, True), (256, 33_000, 136, 5, True),        # three to seven tiles
    (100, 37_000, 1024, 8, True), (64, 60_000, 512, 8, True), (256, 33_000, 2048, 8, True),      # two and three wide ones
    (140, 9475, 3080, 8, True), (140, 18_941, 3080, 16, True), (256, 16_573, 3080, 9, True),     # uneven uniforms over a long d: long and short ring
])
def test_lists_and_samples_follow_from_the_logits(B, K, d, topk, sample):
    h, W, T, u = _inputs(B, K, d, sample, seed=B + K)
    _check(h, W, T, topk, u)


@pytest.mark.parametrize("B,K,topk", [(40, 20_001, 8), (100, 40_001, 5), (200, 40_001, 8), (70, 20_001, 16), (130, 3000, 16)])
def test_ties_go_to_the_lower_index(B, K, topk):
    """Logits of a few distinct values (small whole numbers, exact in every order): tens to thousands of columns tie at the threshold."""
    g = torch.Generator(device=DEV)
    g.manual_seed(K + topk)
    W = torch.randint(-1, 2, (K, 64), generator=g, device=DEV).to(torch.bfloat16)
    W[:, 4:] = 0                                                       # nine values
    h = torch.ones((B, 64), device=DEV).to(torch.bfloat16)
    h[1] = 0                                                           # all columns tie
    h[2] = -1
    _check(h, W, torch.ones(B, device=DEV), topk, None)
    _check(h, W, torch.ones(B, device=DEV), topk, vt_inputs.uniforms((B, K), seed=3, device=DEV))


@pytest.mark.parametrize("B,K", [(40, 20_001), (200, 40_001)])
def test_infinite_and_nan_logits(B, K):
    h, W, T, u = _inputs(B, K, 64, True, seed=B)
    W[:, 0] = 0
    W[5, 0] = float("inf")                                             # +inf, -inf or (times 0) NaN in that column, by row
    W[K - 3, 0] = float("nan")
    h[:, 0] = 0
    h[3, 0] = 1
    h[B - 1, 0] = -1
    _check(h, W, T, 8, u, flags=vt.VT_FLAG_NAN_ROW)
    W[K - 3, 0] = 0
    _check(h, W, T, 8, None, flags=vt.VT_FLAG_NAN_ROW)


@pytest.mark.parametrize("B,K", [
    (8, 19_953), (10, 129),                                            # streaming
    (33, 17), (40, 19_953), (64, 33),                                  # the last column alone in a half of its tile, the other share empty
    (65, 17), (100, 2369), (128, 145),                                 # alone in the last tile
    (129, 33), (200, 2369), (256, 4737),                               # pairs
])
def test_a_nan_or_minus_infinity_alone_in_the_last_column(B, K):
    """Beside shares of a tile that have no column at all, or none but -inf."""
    h, W, T, u = _inputs(B, K, 64, True, seed=B + 1)
    W[K - 1] = float("nan")
    _check(h, W, T, 8, None, flags=vt.VT_FLAG_NAN_ROW)
    _check(h, W, T, 8, u, flags=vt.VT_FLAG_NAN_ROW)
    W[:, 0], W[K - 1], h[:, 0] = 0, 0, 1
    W[K - 1, 0] = float("-inf")                                        # (no candidate, and nothing of the sum)
    _check(h, W, T, 8, u)


@pytest.mark.parametrize("B,K", [(33, 14_209), (64, 4738), (70, 20_003), (130, 9474), (256, 7143)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_uniforms_at_every_offset_from_a_16_byte_boundary(B, K, shift):
    """Rows of every remainder, in a buffer that begins at any of the four places and ends with the last row."""
    h, W, T, u = _inputs(B, K, 128, True, seed=K + shift)
    flat = torch.empty(B * K + shift, device=DEV)
    flat[shift:].view(B, K).copy_(u)
    _check(h, W, T, 8, flat[shift:].view(B, K))


def test_uniforms_at_and_beyond_their_range_and_unaligned():
    B, K = 70, 20_003
    h, W, T, u = _inputs(B, K, 64, True, seed=9)
    u[0], u[1, ::2], u[2, 7], u[3] = 0.0, 1.0, 1.0, 1.0 - 2.0 ** -24
    flat = torch.empty(B * K + 1, device=DEV)
    flat[1:].view(B, K).copy_(u)
    _check(h, W, T, 8, flat[1:].view(B, K))
