"""Attention of heads that keep every key block at head width 128, where the kernel on pairs of SMs can go wrong: block
counts that leave one, two or three of an item's four query blocks without rows, an odd number of key blocks (half of the
last tile is no keys), partial last blocks, more items than clusters and fewer, several batch elements, token-major views, calls
that mix full heads with sparse ones, rows that the fixed softmax reference cannot hold; and the calls that the rules leave to other
kernels (items of one tile, items with idle halves, little work).  Every case says which kernels it has to run on.  The reference is
attention in PyTorch fp64 on the same bf16 values.  Bounds as for the other tcgen05 attention kernel: 2e-2 absolute on the fp32 output and
3e-3 relative in the 2-norm for white noise (weights rounded to bf16), 4e-3 on the log-sum-exp (sums of rounded weights)."""
import pytest
import torch

from parity_utils import attention_path

DEV = "cuda:0"


def _reference(q, k, v, sel, kph):
    B, H, N, d = q.shape
    NB = -(-N // 64)
    o, lse = torch.empty(B, H, N, d, dtype=torch.float64, device=DEV), torch.empty(B, H, N, dtype=torch.float64, device=DEV)
    for b in range(B):
        for h in range(H):
            s = (q[b, h].double() @ k[b, h].double().t()) * d ** -0.5
            if kph[h] < NB:
                m = torch.zeros(NB, NB, dtype=torch.bool, device=DEV).scatter_(1, sel[b, h, :, :kph[h]].long(), True)
                s.masked_fill_(~m.repeat_interleave(64, 0).repeat_interleave(64, 1)[:N, :N], -torch.inf)
            lse[b, h] = torch.logsumexp(s, -1)
            o[b, h] = (s - lse[b, h][:, None]).exp() @ v[b, h].double()
    return o, lse


def _lists(B, H, NB, kph, g):
    sel = torch.full((B, H, NB, max(kph)), -1, dtype=torch.int32, device=DEV)
    for h in range(H):
        sel[:, h, :, :kph[h]] = torch.rand(B, NB, NB, generator=g, device=DEV).topk(kph[h], -1).indices.sort(-1).values.int()
    return sel


def _check(B, H, N, kph, path, token_major=False, edit=None):
    import paper_2512_05754_b200 as usv
    NB, d = -(-N // 64), 128
    g = torch.Generator(device=DEV).manual_seed(N + H)
    shape = (B, N, H, d) if token_major else (B, H, N, d)
    q, k, v = (torch.randn(shape, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    if token_major:
        q, k, v = (x.permute(0, 2, 1, 3) for x in (q, k, v))
    if edit is not None:
        edit(q, k)
    sel = _lists(B, H, NB, kph, g)
    assert attention_path(lambda: usv.sparse_attn_fwd(q, k, v, sel, kph), B * H * NB) == path
    o, o32, lse = usv.sparse_attn_fwd(q, k, v, sel, kph, return_f32=True, return_lse=True)
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0
    n = usv.sparse_attn_fallbacks()
    ro, rl = _reference(q, k, v, sel, kph)
    err = (o32.double() - ro).abs()
    assert err.max() <= 2e-2 and err.norm() <= 3e-3 * ro.norm()
    assert torch.equal(o.contiguous(), o32.to(torch.bfloat16))
    assert (lse.double() - rl).abs().max() <= 4e-3
    return n


@pytest.mark.gpu
@pytest.mark.parametrize("path,B,H,N,token_major", [
    ("dense", 10, 80, 64 * 3, False), ("dense", 10, 80, 64 * 2 + 5, True), ("dense", 10, 60, 64 * 4 - 9, False), ("dense", 10, 48, 64 * 5, True),
    ("dense", 8, 50, 64 * 5 + 3, False), ("dense", 7, 50, 64 * 7 - 1, False), ("dense", 3, 100, 64 * 8, True), ("dense", 1, 60, 64 * 19 - 7, False),
    ("dense", 2, 24, 64 * 30 + 63, True), ("dense", 1, 2, 64 * 101 + 64, False), ("dense", 1, 1, 64 * 145 + 3, False),
    ("dense", 1, 2, 64 * 150 + 9, False), ("dense", 2, 2, 64 * 104, True),
    ("plan", 20, 60, 65, False), ("plan", 20, 60, 64 * 2, True), ("plan", 3, 80, 64 * 10, False), ("plan", 2, 100, 64 * 12 + 1, False),
    ("no plan", 11, 100, 37, False), ("no plan", 10, 120, 64, True), ("no plan", 9, 60, 65, True), ("no plan", 4, 90, 64 * 3, False),
    ("no plan", 3, 80, 64 * 4 + 1, False), ("no plan", 3, 100, 64 * 5 + 3, True), ("no plan", 4, 75, 64 * 6, False)])
def test_full_heads_against_fp64(path, B, H, N, token_major):
    assert _check(B, H, N, [-(-N // 64)] * H, path, token_major) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("N", [64 * 19 + 11, 64 * 20])
def test_full_heads_beside_sparse_ones(N):
    # 50 full heads of 20 blocks, 2 batch elements: 500 items of four blocks, above six waves of 74 clusters
    kph = [20, 20, 3, 20, 20, 20, 20, 7, 20, 20, 20, 20] * 5
    assert _check(2, 60, N, kph, "plan, dense") == 0


@pytest.mark.gpu
@pytest.mark.parametrize("path,N", [("dense", 64 * 100), ("dense", 64 * 101 + 5), ("no plan", 64 * 40), ("no plan", 64 * 41 + 5)])
def test_rows_out_of_range_go_to_the_exact_kernel(path, N):
    """A row's reference is its maximum over the first key block; here later keys of some rows exceed it by more than 100
    powers of two.  Every query block with such a row is counted once."""
    rows = [3, 70, 100, 64 * 7 + 1]

    def edit(q, k):
        for r in rows:
            q[0, 1, r] = 6.0                  # logits with the key below: 6 * 6 * 128 / sqrt(128) = 407, its own block's sums are small
        k[0, 1, 64 * 5 + 2] = 6.0
    assert _check(1, 3, N, [-(-N // 64)] * 3, path, edit=edit) == 3
