"""Vocabularies that the packed counting kernel takes in two to four id ranges (more than 172032 ids): the sizes where the
number of ranges changes, hot ids at the ranges' edges, skipped ids, odd starts, accumulation, wrapping fields, and a
workspace that has no room for the packed counts.  Integer work: the tolerance is zero."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2506_22694_b200 as vt
import vt_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _u32(t):
    return t.cpu().numpy().view(np.uint32).astype(np.uint64)


@pytest.mark.parametrize("V", [172_033, 256_000, 344_063, 344_071, 516_100, 516_200, 655_360])
@pytest.mark.parametrize("n", [5, 9_001, 3_000_017])
def test_ranges_of_a_large_vocabulary(V, n):
    ids = vt_inputs.zipf_ids(n, V, 1.07, seed=V % 997, noise_frac=0.05, device=DEV)
    for p in (2, 3, 4):                                  # the ranges' edges, hot
        e = -(-V // p)
        if n > 1000:
            ids[p::97] = e
            ids[p + 7::89] = e - 1
    if n > 1000:
        ids[11::501], ids[12::5003], ids[13::7001] = V - 1, V, -1      # last id, one past it, negative
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_HISTOGRAM, n, V))
    for off in (0, 3):
        part = ids[off:]
        ref, bad = oracle.histogram(part.cpu().numpy(), V)
        counts = vt.vt_histogram(part, V, ws=ws)
        assert np.array_equal(_u32(counts), ref)
        assert ws.read_status()[2] == bad
        vt.vt_histogram(part, V, counts=counts, accumulate=True, ws=ws)
        assert np.array_equal(_u32(counts), 2 * ref)
        assert ws.read_status()[2] == bad


def test_a_wrapped_field_of_any_range_recounts_the_stream():
    V, n = 300_000, 8_000_000
    ws = vt.Workspace(vt.workspace_bytes(vt.VT_OP_HISTOGRAM, n, V))
    for hot in ((7, 8, 9), (150_001, 299_999, 151_000), (3, 299_000, 299_001)):
        g = torch.Generator(device=DEV).manual_seed(hot[0])
        ids = torch.tensor(hot, dtype=torch.int32, device=DEV)[torch.randint(0, 3, (n,), device=DEV, generator=g)]
        ids[::1_000_003] = V
        ref, bad = oracle.histogram(ids.cpu().numpy(), V)
        assert np.array_equal(_u32(vt.vt_histogram(ids, V, ws=ws)), ref)
        assert ws.read_status()[2] == bad


def test_a_workspace_without_room_for_the_packed_counts_still_serves():
    V, n = 256_000, 1_000_003
    ids = vt_inputs.zipf_ids(n, V, 1.07, seed=3, noise_frac=0.05, device=DEV)
    full = vt.workspace_bytes(vt.VT_OP_HISTOGRAM, n, V)
    ws = vt.Workspace(full)
    counts = torch.empty(V, dtype=torch.int32, device=DEV)
    ref, _ = oracle.histogram(ids.cpu().numpy(), V)
    need = vt.VT_CTRL_BYTES + (V * 4 + 255) // 256 * 256 + (-(-V // 32) * 8 + 255) // 256 * 256   # sampled counts + lookup table
    assert need < full
    for size, status in ((need, 0), (need - 1, 3)):
        got = vt.lib().vt_histogram(ctypes.c_void_p(ids.data_ptr()), n, V, ctypes.c_void_p(counts.data_ptr()), 0,
                                    ctypes.c_void_p(ws.ptr), size, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert got == status
        torch.cuda.synchronize()
        assert np.array_equal(_u32(counts), ref)
