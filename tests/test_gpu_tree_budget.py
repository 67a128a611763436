"""The rerank with a budget as large as its type: every entry beyond the pool's nodes is -1."""
import pytest
import torch

import paper_2506_22694_b200 as vt

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("budget", [1023, 1024, 1025, 2 ** 31 - 1])
def test_rerank_budget_up_to_the_largest(budget):
    if torch.cuda.mem_get_info()[0] < 3 * 4 * budget + (8 << 30):
        pytest.skip("needs the three outputs in device memory")
    n = 40
    pool = vt.tree_pool(n)
    pool[0].copy_(torch.arange(100, 100 + n)), pool[1].fill_(-1), pool[2].copy_(-torch.arange(n, dtype=torch.float32))
    nodes, token, parent = vt.vt_tree_rerank(pool, n, budget)
    assert nodes[:n].tolist() == list(range(n)) and token[:n].tolist() == list(range(100, 100 + n))
    assert bool((parent[:n] == -1).all())
    for t in (nodes, token, parent):
        for lo in range(n, budget, 1 << 28):
            assert bool((t[lo:min(budget, lo + (1 << 28))] == -1).all())
