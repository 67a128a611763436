"""The heads' log-sum-exp where the logits are large against their spread: a common offset, and temperatures small enough that
one candidate holds all the mass.  The reference is 64-bit arithmetic over the kernel's own fp32 logits."""
import pytest
import torch

import paper_2506_22694_b200 as vt
import vt_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _head(B, K, offset, T, seed):
    """Logits around `offset` with deviation about 1 (the first column of h and W makes the offset)."""
    d = 256
    W = vt_inputs.gaussian_bf16((K, d), 0.0625, seed=seed, device=DEV)
    h = vt_inputs.gaussian_bf16((B, d), 1.0, seed=seed + 1, device=DEV)
    W[:, 0], h[:, 0] = float(offset), 1.0
    return vt.vt_draft_head(h, W, None, torch.full((B,), T, device=DEV), 8, None, debug=True)


@pytest.mark.parametrize("B", [8, 64, 256])                # streaming, batched, batched in CTA pairs
@pytest.mark.parametrize("offset", [0, 40, 1000, 30000])
def test_lse_of_offset_logits(B, offset):
    ids, lps, logits, lse = _head(B, 6000, offset, 1.0, seed=offset + B)
    z = logits.double()
    want = torch.logsumexp(z, dim=1)
    # one rounding of the final max + log(sum) (half a unit: 2^-24 of its size; the next one for the fast logarithm's last
    # step), and the sum itself: 2^-22 per base-2 exponential, 2^-24 for each of at most 64 additions and rescales in a row
    bound = want.abs() * 2.0 ** -24 + 2.0 ** -22 + 64 * 2.0 ** -24
    assert bool(((lse.double() - want).abs() <= bound).all())


@pytest.mark.parametrize("B", [8, 64, 256])
@pytest.mark.parametrize("T", [1e-6, 1e-8, 1e-20])
def test_a_tiny_temperature_leaves_all_the_mass_on_the_best_candidate(B, T):
    """logit / T of 1e7 to 1e21: the best candidate's log-probability is 0 and every other's minus the (huge) difference."""
    ids, lps, logits, lse = _head(B, 6000, 5, T, seed=B)
    best = logits.max(dim=1)
    assert torch.equal(ids[:, 1].long(), best.indices) and bool((lps[:, 1] == 0).all())
    assert torch.equal(ids[:, 0], ids[:, 1]) and bool((lps[:, 2:] <= 0).all())
    z = torch.gather(logits, 1, ids[:, 1:].long()) * (1.0 / torch.tensor(T, device=DEV))
    assert torch.equal(lps[:, 1:], z - z[:, :1])
