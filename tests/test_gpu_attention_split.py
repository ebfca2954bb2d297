"""Small attention calls at head width 64, where four groups of warps share a query block, against the kernel with one group
(impl = 1): lists of one entry (three groups without any) to ten (groups of two and three, one and two tiles in flight), holes,
rows without keys, a partial last block, views with shared heads, logits that differ a lot between a row's key blocks, and
values that are not finite, which stay in their rows.  Lists of up to four blocks give the same bits.  Longer ones round the same
weights to bf16, each group relative to a running maximum of its own: outputs of white noise differ by less than 3e-3 in the 2-norm,
log-sum-exps by 1e-4.  Both kernels share the code of a tile, so the results are compared with PyTorch in fp64 too, within 2^-9 (each
weight's rounding) and 1e-5 on the log-sum-exp per unit of its size."""
import pytest
import torch

DEV = "cuda:0"


def _run(q, k, v, sel, kph):
    import paper_2512_05754_b200 as usv
    out = [usv.sparse_attn_fwd(q, k, v, sel, kph, return_f32=True, return_lse=True, impl=i) for i in (0, 1)]
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0 and usv.sparse_attn_fallbacks() == 0
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,N,kph,shared", [
    (1, 1, 33, [1], False), (1, 2, 64 * 4, [4, 1], False), (2, 3, 64 * 9 + 7, [5, 2, 3], False), (1, 4, 64 * 37, [10, 9, 8, 6], False),
    (1, 2, 64 * 73 + 1, [7, 4], True), (1, 1, 64 * 147 + 63, [10], False)])
def test_small_calls_at_d64(B, H, N, kph, shared):
    g = torch.Generator(device=DEV).manual_seed(N)
    NB, kmax = -(-N // 64), max(kph)
    q = torch.randn(B, H, N, 64, generator=g, device=DEV).to(torch.bfloat16)
    k, v = (torch.randn(B, 1 if shared else H, N, 64, generator=g, device=DEV).to(torch.bfloat16).expand(B, H, N, 64) for _ in range(2))
    if not shared:
        k = k.contiguous()
        k[:, :, 64 * (NB // 2):64 * (NB // 2) + 5] *= 20      # a row's maxima differ by up to 200 from block to block
    sel = torch.full((B, H, NB, kmax), -1, dtype=torch.int32, device=DEV)
    for h in range(H):
        sel[:, h, :, :kph[h]] = torch.rand(B, NB, NB, generator=g, device=DEV).topk(kph[h], -1).indices.sort(-1).values.int()
    if NB > 3:
        sel[:, :, 1, 0] = -1
        sel[:, :, 2, kmax // 2:] = -1
        sel[:, :, 3] = -1
    (o, o32, lse), (_, r32, rlse) = _run(q, k, v, sel, kph)
    assert (o32 - r32).norm() <= 3e-3 * r32.norm()
    assert torch.equal(o, o32.to(torch.bfloat16))
    assert (lse - rlse).abs().max() <= 1e-4 * max(1.0, rlse.abs().max().item())
    if NB > 3:
        assert not o32[:, :, 64 * 3:64 * 4].any() and not lse[:, :, 64 * 3:64 * 4].any()


@pytest.mark.gpu
def test_values_that_are_not_finite_stay_in_their_rows():
    B, H, NB, kph = 1, 2, 12, [6, 3]
    g = torch.Generator(device=DEV).manual_seed(0)
    q, k, v = (torch.randn(B, H, 64 * NB, 64, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    q[0, 0, 70] = float("inf")
    k[0, 0, 64 * 4 + 1, 3] = float("nan")
    v[0, 1, 64 * 2] = float("inf")
    sel = torch.rand(B, H, NB, NB, generator=g, device=DEV).topk(6, -1).indices.sort(-1).values.int()
    (o, o32, lse), (_, r32, rlse) = _run(q, k, v, sel, kph)
    assert torch.equal(torch.isfinite(o32), torch.isfinite(r32)) and not torch.isfinite(r32).all()
    ok = torch.isfinite(r32)
    assert (o32[ok] - r32[ok]).norm() <= 3e-3 * r32[ok].norm()


def _fp64(q, k, v, sel):
    B, H, N, d = q.shape
    NB = -(-N // 64)
    s = (q.double() @ k.double().transpose(-1, -2)) * d ** -0.5
    kept = torch.zeros(B, H, NB, NB + 1, dtype=torch.bool, device=DEV).scatter_(3, torch.where(sel < 0, NB, sel).long(), True)[..., :NB]
    s = s.masked_fill(~kept.repeat_interleave(64, 2).repeat_interleave(64, 3)[:, :, :N, :N], -torch.inf)
    return torch.softmax(s, -1).nan_to_num(0.0) @ v.double(), torch.logsumexp(s, -1).clamp_min(-1e30)


@pytest.mark.gpu
@pytest.mark.parametrize("H,N,kph", [(2, 64 * 16, [4]), (3, 64 * 16 + 1, [2, 4, 1]), (1, 64 * 147 + 63, [3]), (2, 64 * 5, [4, 3]),
                                     (8, 64 * 16, [4, 3, 2, 1]), (1, 2 * 64 + 5, [2]), (2, 64 * 20 + 9, [5, 10]), (4, 64 * 32, [8, 7, 6, 9])])
def test_small_calls_are_the_exact_kernel_and_near_fp64(H, N, kph):
    g = torch.Generator(device=DEV).manual_seed(N)
    kph = (kph * H)[:H]
    NB, kmax = -(-N // 64), max(kph)
    q, k, v = (torch.randn(1, H, N, 64, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    k[:, :, 64:64 + 9] *= 3                     # maxima that move along a list
    sel = torch.full((1, H, NB, kmax), -1, dtype=torch.int32, device=DEV)
    for h in range(H):
        sel[:, h, :, :kph[h]] = torch.rand(1, NB, NB, generator=g, device=DEV).topk(kph[h], -1).indices.sort(-1).values.int()
    if NB > 4:
        sel[:, :, 1, 0] = -1
        sel[:, :, 2, kmax // 2:] = -1
        sel[:, :, 3] = -1
        sel[:, :, 4, 1:kmax - 1] = -1
    (o, o32, lse), (r, r32, rlse) = _run(q, k, v, sel, kph)
    if kmax <= 4:
        assert torch.equal(o.view(torch.int16), r.view(torch.int16)) and torch.equal(o32, r32) and torch.equal(lse, rlse)
    ref, ref_lse = _fp64(q, k, v, sel)
    assert (o32.double() - ref).norm() <= 2.0 ** -9 * ref.norm()
    some = ref_lse > -1e29
    assert (lse.double() - ref_lse)[some].abs().max() <= 1e-5 * max(1.0, ref_lse[some].abs().max().item()) and not lse[~some].any()


@pytest.mark.gpu
def test_values_that_are_not_finite_in_lists_of_four():
    g = torch.Generator(device=DEV).manual_seed(1)
    q, k, v = (torch.randn(1, 2, 64 * 12, 64, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    q[0, 0, 70] = float("inf")
    k[0, 0, 64 * 4 + 1, 3] = float("nan")
    k[0, 1, 64 * 3 + 7] = -float("inf")
    v[0, 1, 64 * 2] = float("inf")
    sel = torch.rand(1, 2, 12, 12, generator=g, device=DEV).topk(4, -1).indices.sort(-1).values.int()
    (o, o32, lse), (r, r32, rlse) = _run(q, k, v, sel, [4, 2])
    for x, y in ((o, r), (o32, r32), (lse, rlse)):
        assert torch.equal(x.isnan(), y.isnan()) and torch.equal(x.nan_to_num(0.0), y.nan_to_num(0.0))
    assert not torch.isfinite(r32).all()
