"""Attention over single kept blocks.  At head width 128 an item's list is one or two entries taken straight from the two
selection rows, at 64 many blocks run on the mma.sync kernel with one buffer: the same entry twice, either order, one or both
missing, out of range, an odd number of query blocks, a partial last block, many blocks, shared lists per head.  Against the exact
kernel (impl = 1) within the bf16 bound of its weights, 3e-3 in the 2-norm for white noise, and 4e-3 on the log-sum-exp."""
import pytest
import torch

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,N", [(1, 1, 64 * 3), (2, 3, 64 * 8 + 1), (1, 24, 64 * 71 - 5), (2, 40, 64 * 40)])
def test_single_blocks(d, B, H, N):
    import paper_2512_05754_b200 as usv
    NB = -(-N // 64)
    g = torch.Generator(device=DEV).manual_seed(N)
    q, k, v = (torch.randn(B, H, N, d, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    sel = torch.randint(NB, (B, H, NB, 1), generator=g, device=DEV, dtype=torch.int32)
    sel[:, :, 1::4] = sel[:, :, 0::4][:, :, :sel[:, :, 1::4].shape[2]]      # both rows of an item the same
    if NB > 7:
        sel[:, 0, 2] = -1
        sel[:, 0, 5] = -1
        sel[:, 0, 6:8] = -1
    k[:, -1, -5:] *= 60          # some logits far above: the exact kernel's rows
    (o, o32, lse), (_, r32, rl) = (usv.sparse_attn_fwd(q, k, v, sel, [1] * H, return_f32=True, return_lse=True, impl=i) for i in (0, 1))
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0
    assert (o32 - r32).norm() <= 3e-3 * r32.norm() and torch.equal(o, o32.to(torch.bfloat16))
    assert (lse - rl).abs().max() <= 4e-3 * max(1.0, rl.abs().max().item())
    if d == 64 and B * H * NB > 1800:
        assert torch.equal(o32, r32) and torch.equal(lse, rl)
    if NB > 7:
        assert not o32[:, 0, 64 * 6:64 * 8].any() and not o32[:, 0, 64 * 2:64 * 3].any()
