"""Key marginal with a pairing plan (large calls with scratch memory) against the same call without scratch, which pairs
neighbours and is compared with fp64 elsewhere: odd numbers of blocks, a partial last block, several batch elements, heads
that keep everything beside sparse ones, lists with holes, also full ones, one and two passes of the plan.  Both exponentiate
the same logits; a key's sum of up to 64 x 401 x 16 weights is taken in fp32 in another order, so sums differ by less
than 1e-5 of the largest."""
import ctypes

import pytest
import torch

DEV = "cuda:0"


class S(ctypes.Structure):
    _fields_ = [("sb", ctypes.c_int64), ("sh", ctypes.c_int64), ("sn", ctypes.c_int64)]


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,N,d,kph,holes", [
    (1, 16, 64 * 400 + 5, 64, [80], True), (1, 16, 64 * 400 + 5, 128, [80, 79], False),
    (2, 17, 64 * 300, 128, [95, 300, 60, 1, 95, 95, 64, 75, 95], True),
    (1, 16, 64 * 450 + 64, 64, [111, 112, 451], True), (1, 12, 64 * 640 + 1, 128, [150], False)])
def test_planned_marginal_is_the_plain_one(B, H, N, d, kph, holes):
    from paper_2512_05754_b200 import binding
    L = binding.lib()
    L.usv_attn_entropy_workspace.restype = L.usv_attn_entropy_lists_workspace.restype = ctypes.c_size_t
    kph = (kph * H)[:H]
    NB, kmax = -(-N // 64), max(kph)
    assert B * NB * sum(k for k in kph if k < NB) >= 500000
    g = torch.Generator(device=DEV).manual_seed(N + d)
    q, k = (torch.randn(B, H, N, d, generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
    lse = 6 + torch.rand(B, H, N, generator=g, device=DEV)
    # lists that overlap with those of blocks far away, as in video
    score = torch.rand(B, H, 16, NB, generator=g, device=DEV)[:, :, torch.randint(16, (NB,), generator=g, device=DEV)]
    score = score + 0.2 * torch.rand(B, H, NB, NB, generator=g, device=DEV)
    sel = torch.full((B, H, NB, kmax), -1, dtype=torch.int32, device=DEV)
    for h in range(H):
        sel[:, h, :, :kph[h]] = score[:, h].topk(kph[h], -1).indices.sort(-1).values.int()
    if holes:
        sel[:, :, ::3, kmax // 2] = -1
        sel[:, :, 1::5, 0] = -1
    s = S(*q.stride()[:3])
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    n = L.usv_attn_entropy_lists_workspace(B, H, N, (ctypes.c_int32 * H)(*kph))
    assert 256 < n <= L.usv_attn_entropy_workspace(B, H, N, kmax)
    ws = torch.zeros(n, dtype=torch.uint8, device=DEV)
    out = []
    for room in (n - 1, n):
        marg, ent = torch.full((B, N), -1.0, device=DEV), torch.full((B,), -1.0, device=DEV)
        ws[4:256].fill_(7)
        before = L.usv_kernel_launches()
        rc = L.usv_attn_entropy_ws(B, H, N, d, p(q), ctypes.byref(s), p(k), ctypes.byref(s), p(sel), (ctypes.c_int32 * H)(*kph),
                                   kmax, p(lse), ctypes.c_float(0.0), p(marg), p(ent), p(ws), ctypes.c_size_t(room),
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0 and (L.usv_kernel_launches() - before > 2) == (room == n)
        torch.cuda.synchronize()
        assert int(ws[:4].view(torch.int32)) == 0 and bool((ws[4:256] == 7).all())   # the attention's counts stay
        out.append((marg, ent))
    assert torch.equal(out[0][0] == 0, out[1][0] == 0)
    assert (out[0][0] - out[1][0]).abs().max() <= 1e-5 * out[0][0].max()
    assert (out[0][1] - out[1][1]).abs().max() <= 1e-5 * out[0][1].abs().max()


@pytest.mark.gpu
def test_calls_without_a_plan_ask_for_no_room():
    """Lists that a plan does not pay for, although one head keeps everything, take nothing beyond the header from a stream's buffer."""
    import paper_2512_05754_b200 as usv
    from paper_2512_05754_b200 import binding
    H, NB = 2, 300
    g = torch.Generator(device=DEV).manual_seed(5)
    q, k = (torch.randn(1, H, 64 * NB, 64, generator=g, device=DEV).to(torch.bfloat16) for _ in range(2))
    sel = torch.arange(NB, device=DEV, dtype=torch.int32).expand(1, H, NB, NB).contiguous()
    with torch.cuda.stream(torch.cuda.Stream()):
        marg, _ = usv.attn_entropy(q, k, sel, [NB, 10], torch.full((1, H, 64 * NB), 6.0, device=DEV))
        torch.cuda.synchronize()
        assert binding._workspace(torch.device(DEV), 0).numel() == 256
    assert bool((marg > 0).all())
