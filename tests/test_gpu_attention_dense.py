"""Attention of heads that keep every key block at head width 128, where the kernel on pairs of SMs can go wrong: block
counts that leave one, two or three of an item's four query blocks without rows, an odd number of key blocks (half of the
last tile is no keys), partial last blocks, more items than clusters and fewer, several batch elements, token-major views, calls
that mix full heads with sparse ones, rows that the fixed softmax reference cannot hold, lists of as many entries as there are
key blocks with holes (-1, which every kernel skips); and the calls that the rules leave to other
kernels (items of one tile, emptier waves, little work).  Every case says which kernels it has to run on.  The reference is
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
            l = sel[b, h, :, :kph[h]].long()
            m = torch.zeros(NB, NB + 1, dtype=torch.bool, device=DEV).scatter_(1, torch.where(l < 0, NB, l), True)[:, :NB]
            if not m.all():
                s.masked_fill_(~m.repeat_interleave(64, 0).repeat_interleave(64, 1)[:N, :N], -torch.inf)
            lse[b, h] = torch.logsumexp(s, -1)
            o[b, h] = torch.softmax(s, -1).nan_to_num(0.0) @ v[b, h].double()
            lse[b, h][lse[b, h] == -torch.inf] = 0.0          # (no key at all: zeros)
    return o, lse


def _lists(B, H, NB, kph, g):
    sel = torch.full((B, H, NB, max(kph)), -1, dtype=torch.int32, device=DEV)
    for h in range(H):
        sel[:, h, :, :kph[h]] = torch.rand(B, NB, NB, generator=g, device=DEV).topk(kph[h], -1).indices.sort(-1).values.int()
    return sel


def _check(B, H, N, kph, path, token_major=False, edit=None, d=128, holes=None):
    import paper_2512_05754_b200 as usv
    NB = -(-N // 64)
    g = torch.Generator(device=DEV).manual_seed(N + H)
    shape = (B, N, H, d) if token_major else (B, H, N, d)
    q, k, v = (torch.randn(shape, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    if token_major:
        q, k, v = (x.permute(0, 2, 1, 3) for x in (q, k, v))
    if edit is not None:
        edit(q, k)
    sel = _lists(B, H, NB, kph, g)
    if holes is not None:
        holes(sel)
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
    ("dense", 1, 2, 64 * 150 + 9, False), ("dense", 2, 2, 64 * 104, True), ("dense", 1, 12, 64 * 29 + 1, False), ("no plan", 1, 12, 64 * 28, False),
    ("dense", 3, 70, 64 * 7 - 3, True),
    ("plan", 20, 60, 65, False), ("plan", 20, 60, 64 * 2, True), ("plan", 4, 100, 64 * 10, False), ("plan", 1, 100, 64 * 12 + 1, False), ("plan", 1, 16, 64 * 53 - 1, False), ("dense", 1, 7, 64 * 85, True),
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
@pytest.mark.parametrize("path,N", [("dense", 64 * 100), ("dense", 64 * 101 + 5), ("no plan", 64 * 40), ("no plan", 64 * 41 + 5), ("dense", 64 * 60)])
def test_rows_out_of_range_go_to_the_exact_kernel(path, N):
    """A row's reference is its maximum over the first key block; here later keys of some rows exceed it by more than 100
    powers of two.  Every query block with such a row is counted once."""
    rows = [3, 70, 100, 64 * 7 + 1]

    def edit(q, k):
        for r in rows:
            q[0, 1, r] = 6.0                  # logits with the key below: 6 * 6 * 128 / sqrt(128) = 407, its own block's sums are small
        k[0, 1, 64 * 5 + 2] = 6.0
    assert _check(1, 3, N, [-(-N // 64)] * 3, path, edit=edit) == 3


@pytest.mark.gpu
@pytest.mark.parametrize("path,d,B,H,N,kph", [
    ("dense", 128, 1, 3, 64 * 100 + 7, [101]), ("dense", 128, 10, 80, 64 * 3, [3]), ("dense", 128, 2, 24, 64 * 30 + 63, [31]),
    ("plan, dense", 128, 2, 60, 64 * 20, [20, 20, 3, 20, 20, 20, 20, 7, 20, 20, 20, 20]), ("plan", 128, 4, 100, 64 * 10, [10]),
    ("plan", 128, 1, 12, 64 * 60 - 5, [60, 20, 20]), ("plan", 64, 1, 4, 64 * 103 + 1, [104]), ("plan", 64, 1, 10, 64 * 300, [300, 10]),
    ("no plan", 128, 1, 3, 64 * 40, [40]), ("no plan", 64, 1, 3, 64 * 33 - 1, [33])])
def test_holes_in_full_lists(path, d, B, H, N, kph):
    """A block without its first, its last and an inner entry, one with a single key block and one with none, in the first head and
    in the last full one.  On the dense kernel they go to the exact one; the others read their lists, and only the rows that share an
    item but see no key go there."""
    NB = -(-N // 64)
    kph = (kph * H)[:H]
    heads = [0, max(h for h in range(H) if kph[h] == NB)]

    def holes(sel):
        for h in heads:
            sel[-1, h, 0, 0] = -1
            sel[-1, h, NB - 1, NB - 1] = -1
            sel[-1, h, 1, 1] = -1
            if NB > 3:
                sel[-1, h, NB // 2, :NB - 1] = -1
                sel[-1, h, NB // 2 + 1] = -1
    n = _check(B, H, N, kph, path, d=d, holes=holes)
    assert n == len(set(heads)) * ((5 if NB > 3 else 3) if "dense" in path else 1)


@pytest.mark.gpu
def test_holes_in_full_lists_with_the_unmerge_folded_in():
    import paper_2512_05754_b200 as usv
    H, N, n_full = 3, 64 * 101, 64 * 120
    g = torch.Generator(device=DEV).manual_seed(2)
    q, k, v = (torch.randn(1, H, N, 128, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    sel = torch.arange(101, device=DEV, dtype=torch.int32).expand(1, H, 101, 101).clone()
    sel[0, 1, 7, 50:] = -1
    sel[0, 2, 8] = -1
    pos = torch.cat([torch.arange(N, device=DEV), torch.randint(N, (n_full - N,), generator=g, device=DEV)]).int()[None]
    y = usv.sparse_attn_fwd_unmerge(q, k, v, sel, [101] * H, usv.unmerge_map(pos, N), n_full)
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0
    o, _ = _reference(q, k, v, sel, [101] * H)
    ref = o.permute(0, 2, 1, 3).reshape(1, N, H * 128)[:, pos[0].long()]
    assert (y.double() - ref).abs().max() <= 2e-2 and (y.double() - ref).norm() <= 5e-3 * ref.norm()   # (bf16 output: 2^-9 more)
