"""The tcgen05 attention kernel where its head-width-64 form, and the hand-over of non-finite rows
to the exact kernel, can go wrong; against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import usv_inputs as ui
from parity_utils import attention_path, attn_errors

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MAX_ABS, REL_L2, REL_L2_BF16 = 2e-2, 1e-3, 2.5e-3


@pytest.fixture(scope="module")
def usv():
    import paper_2512_05754_b200 as m
    return m


# an odd number of query blocks and a partial last block on either side of the longest list of small calls (10 entries); more
# query blocks than those with short lists; union lists beyond a ring slot (512 entries); more work than runs without a plan
@pytest.mark.parametrize("path,B,H,grid,kph", [
    ("one kernel", 1, 1, (3, 9, 25), [9]), ("no plan", 1, 1, (3, 12, 25), [11]), ("no plan", 2, 3, (5, 31, 33), [3, 1, 8]),
    ("plan", 1, 1, (9, 62, 66), [515]), ("plan", 1, 8, (10, 32, 32), [30, 29, 40])])
def test_head_width_64(usv, path, B, H, grid, kph):
    kph = (kph * H)[:H]
    wl = ui.Workload("d64_edges", 170 + len(kph), B, H, 64, grid, (100,))
    N, NB = wl.N, wl.NB
    q, k, v = ui.make_qkv(wl, layout="bnhd")
    rng = np.random.default_rng(NB)
    sel = np.full((B, H, NB, max(kph)), -1, dtype=np.int32)
    for b in range(B):
        for h in range(H):
            for i in range(NB):
                sel[b, h, i, :kph[h]] = np.sort(rng.choice(NB, size=kph[h], replace=False))
    args = (q.to(DEV), k.to(DEV), v.to(DEV), torch.from_numpy(sel).to(DEV), kph, N)
    assert attention_path(lambda: usv.sparse_attn_fwd(*args), B * H * NB) == path
    o, o32, lse = usv.sparse_attn_fwd(*args, return_f32=True, return_lse=True)
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0 and usv.sparse_attn_fallbacks() == 0
    o_ref, lse_ref = oracle.sparse_attn(q, k, v, N, sel, kph)
    o_ref = o_ref.reshape(B, H, NB * 64, 64)[:, :, :N]
    mx, rl2 = attn_errors(o32.cpu().numpy(), o_ref)
    _, rl2b = attn_errors(o.float().cpu().numpy(), o_ref)
    assert mx <= MAX_ABS and rl2 <= REL_L2 and rl2b <= REL_L2_BF16, (mx, rl2, rl2b)
    assert np.abs(lse.cpu().numpy() - lse_ref.reshape(B, H, NB * 64)[:, :, :N]).max() <= 2e-3


# small calls, which keep query blocks apart, items of neighbours, and items of a plan, which pairs the one block with another list
# with the one that is left of those with the same
@pytest.mark.parametrize("path,H,NB,K,with_inf", [("one kernel", 1, 12, 9, slice(1, None, 2)), ("no plan", 1, 14, 11, slice(1, None, 2)),
                                                  ("no plan", 2, 80, 15, slice(7, 8)), ("plan", 4, 120, 80, slice(1, 2))])
def test_an_infinity_reaches_only_the_query_blocks_that_selected_it(usv, path, H, NB, K, with_inf):
    """Two query blocks share an item; one alone selects a block with an infinity in V.
    Its own rows are not finite, its partner's equal the result without that block."""
    N, d = 64 * NB, 64
    g = torch.Generator().manual_seed(d)
    q, k, v = (torch.randn(1, H, N, d, generator=g).to(torch.bfloat16) for _ in range(3))
    v[:, 0, 64 * (NB - 1) + 5, 3] = float("inf")
    sel = torch.arange(K, dtype=torch.int32).expand(1, H, NB, K).clone()
    sel[0, 0, with_inf, K - 1] = NB - 1
    args = (q.to(DEV), k.to(DEV), v.to(DEV), sel.to(DEV), [K] * H)
    assert attention_path(lambda: usv.sparse_attn_fwd(*args), H * NB) == path
    o = usv.sparse_attn_fwd(*args).float().cpu()[0].reshape(H, NB, 64, d)
    if path != "one kernel":
        assert usv.sparse_attn_fallbacks() == 2 * len(range(NB)[with_inf])        # they did share items, and were recomputed
    exact = usv.sparse_attn_fwd(*args, impl=1).float().cpu()[0].reshape(H, NB, 64, d)
    hit = torch.zeros(H, NB, dtype=torch.bool)
    hit[0, with_inf] = True
    assert torch.isfinite(o[~hit]).all()
    assert not torch.isfinite(o[hit][..., 3]).any()
    assert (o[~hit] - exact[~hit]).abs().max() <= MAX_ABS


# the kernel of small calls, without a plan, with one; some with logits nine times the size
@pytest.mark.parametrize("path,B,H,grid,k,amp", [
    ("one kernel", 1, 2, (4, 20, 24), 6, 1.0), ("no plan", 2, 3, (5, 31, 33), 20, 1.0), ("one kernel", 1, 1, (3, 9, 25), 5, 1.0),
    ("no plan", 1, 4, (6, 32, 32), 30, 3.0), ("plan", 1, 8, (10, 32, 32), 30, 3.0)])
def test_log_sum_exp_is_fp32_exact(usv, path, B, H, grid, k, amp):
    """The log-sum-exp comes from unrounded weights.  Bound: logits in base 2 of up to 100 carry an fp32 rounding of
    100 x 2^-24 = 6e-6 each from the product and from the reference, exp2 2^-22 and the sum of up to 1920 weights in
    four chains 480 x 2^-24 = 2.9e-5 if every rounding went the same way; seen: 1.2e-5."""
    wl = ui.Workload("d64_lse", 230 + k, B, H, 64, grid, (100,))
    N, NB = wl.N, wl.NB
    q, kk, v = ui.make_qkv(wl)
    q, kk = (q.float() * amp).to(torch.bfloat16), (kk.float() * amp).to(torch.bfloat16)
    sel = np.sort(np.argsort(np.random.default_rng(k).random((B, H, NB, NB)), axis=-1)[..., :k].astype(np.int32), axis=-1)
    args = (q.to(DEV), kk.to(DEV), v.to(DEV), torch.from_numpy(sel).to(DEV), [k] * H)
    assert attention_path(lambda: usv.sparse_attn_fwd(*args, return_lse=True), B * H * NB) == path
    _, lse = usv.sparse_attn_fwd(*args, return_lse=True)
    assert usv.workspace_status() == 0
    _, ref = oracle.sparse_attn(q, kk, v, N, sel, [k] * H)
    assert np.abs(lse.cpu().numpy() - ref.reshape(B, H, NB * 64)[:, :, :N]).max() <= 4e-5


@pytest.mark.parametrize("d", [64, 128])
def test_repeated_calls_give_the_same_bits(usv, d):
    """Several items a CTA, drawn in another order every time: the partial row sums are still added in one order."""
    H, NB, k = 4, 400, 90
    g = torch.Generator().manual_seed(d)
    q, kk, v = (torch.randn(1, H, 64 * NB, d, generator=g).to(torch.bfloat16).to(DEV) for _ in range(3))
    sel = torch.rand(1, H, NB, NB, generator=g).topk(k, -1).indices.sort(-1).values.to(torch.int32).to(DEV)
    first = usv.sparse_attn_fwd(q, kk, v, sel, [k] * H, return_f32=True, return_lse=True)
    for _ in range(4):
        again = usv.sparse_attn_fwd(q, kk, v, sel, [k] * H, return_f32=True, return_lse=True)
        assert all(torch.equal(a, b) for a, b in zip(first, again))


# one kept block and four on either side of the lines to the mma.sync kernel, a few beyond
@pytest.mark.parametrize("H,NB,k", [(2, 1, 1), (4, 450, 1), (4, 451, 1), (4, 751, 2), (4, 96, 4), (4, 97, 4), (4, 96, 5), (3, 5, 5)])
def test_lines_to_the_kernel_of_short_lists(usv, H, NB, k):
    N = 64 * NB - 9
    g = torch.Generator().manual_seed(NB + k)
    q, kk, v = (torch.randn(1, H, N, 64, generator=g).to(torch.bfloat16) for _ in range(3))
    sel = np.sort(np.argsort(np.random.default_rng(NB).random((1, H, NB, NB)), axis=-1)[..., :k].astype(np.int32), axis=-1)
    o, o32, lse = usv.sparse_attn_fwd(q.to(DEV), kk.to(DEV), v.to(DEV), torch.from_numpy(sel).to(DEV), [k] * H, return_f32=True,
                                      return_lse=True)
    assert usv.workspace_status() == 0 and usv.sparse_attn_fallbacks() == 0
    o_ref, lse_ref = oracle.sparse_attn(q, kk, v, N, sel, [k] * H)
    mx, rl2 = attn_errors(o32.cpu().numpy(), o_ref.reshape(1, H, NB * 64, 64)[:, :, :N])
    # bf16 weights are off by up to 2^-9 of themselves each; values without a common part do not average that away
    assert mx <= MAX_ABS and rl2 <= 2.0 ** -9, (mx, rl2)
    assert np.abs(lse.cpu().numpy() - lse_ref.reshape(1, H, NB * 64)[:, :, :N]).max() <= 2e-5
