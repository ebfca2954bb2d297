"""Block scores on either side of the line between the kernel for small calls and the ones for large
calls, and of the spans of the pooling kernel; tile remainders, different lengths of q and k."""
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Nq,Nk", [(1, 1, 5, 2100), (2, 3, 64 * 33 - 1, 64 * 31 + 7), (1, 7, 64 * 320, 64 * 319 + 1),
                                       (1, 8, 64 * 320, 64 * 293), (1, 2, 64 * 3000 + 3, 64 * 9)])
def test_scores_match_the_oracle(d, B, H, Nq, Nk):
    import paper_2512_05754_b200 as usv
    g = torch.Generator().manual_seed(d + Nq)
    q = torch.randn(B, Nq, H, d, generator=g).to(torch.bfloat16).permute(0, 2, 1, 3)
    k = torch.randn(B, H, Nk, d, generator=g).to(torch.bfloat16)
    got = usv.block_scores(q.to(DEV), k.to(DEV)).cpu().numpy()
    assert usv.workspace_status() == 0
    ref = oracle.block_scores(oracle.block_pool(q, Nq), oracle.block_pool(k, Nk))
    assert abs(got - ref).max() <= 2e-6 * max(1.0, abs(ref).max())
