"""Block scores of short sequences, pooled and multiplied by one cluster of CTAs per head, at the edges of that kernel's forms:
one block, fewer blocks than CTAs, shares that do not divide, the longest sequences, different lengths of q and k, partial last blocks,
strided views, one to four CTAs an SM, and one block or head beyond each line.  The fp32 kernel without scratch pools and multiplies in
the same order, so the scores are the same bit for bit."""
import pytest
import torch

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,Nq,Nk", [
    (1, 1, 1, 64), (1, 3, 65, 64 * 9 - 1), (2, 9, 64 * 32, 64 * 31 + 5), (1, 18, 64 * 48 - 63, 64 * 17), (1, 18, 64 * 49, 64 * 48),
    (1, 19, 64 * 16, 64 * 13 + 1), (2, 18, 64 * 33, 64 * 32), (1, 37, 64 * 11 + 2, 64 * 16), (5, 11, 64 * 16 - 7, 64 * 8),
    (4, 19, 64 * 17, 64 * 16), (2, 40, 64 * 16, 64 * 16)])
def test_scores_are_those_of_the_kernel_without_scratch(d, B, H, Nq, Nk):
    import paper_2512_05754_b200 as usv
    from paper_2512_05754_b200 import binding
    g = torch.Generator(device=DEV).manual_seed(Nq + d)
    q = torch.randn(B, Nq, 3, H, d, generator=g, device=DEV).to(torch.bfloat16)[:, :, 1].permute(0, 2, 1, 3)
    k = torch.randn(B, H, Nk, d, generator=g, device=DEV).to(torch.bfloat16)
    out = torch.full((B, H, -(-Nq // 64), -(-Nk // 64)), 7.0, device=DEV)
    assert torch.equal(usv.block_scores(q, k, out=out), binding.block_scores_noalloc(q, k))
    assert usv.workspace_status() == 0
