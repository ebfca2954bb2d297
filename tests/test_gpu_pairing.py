"""Calls whose query blocks are put in list order before they are paired: every query block is computed
exactly once whatever the lists look like.  Against the fp64 oracle on sampled blocks and the
mma.sync kernel, which pairs nothing, on all of them."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import attn_errors, gather_qblocks

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
MAX_ABS, REL_L2_WHITE_NOISE_V = 2e-2, 3e-3


@pytest.fixture(scope="module")
def usv():
    import paper_2512_05754_b200 as m
    return m


# 401 blocks: a last chunk of 17; a full list beside sparse ones; odd counts, a partial last block,
# head width 64; the longest sequence of the tcgen05 kernel
@pytest.mark.parametrize("B,H,N,d,kph", [(1, 24, 401 * 64, 128, [220, 401] * 12), (2, 12, 641 * 64 - 50, 64, [70, 12, 120] * 4),
                                         (1, 1, 4096 * 64 - 1, 128, [250])])
def test_every_query_block_once(usv, B, H, N, d, kph):
    NB, kmax = (N + 63) // 64, max(kph)
    g = torch.Generator(device=DEV).manual_seed(NB)
    q, k, v = (torch.randn(B, H, N, d, generator=g, device=DEV).to(torch.bfloat16) for _ in range(3))
    rng = np.random.default_rng(NB)
    sel = np.full((B, H, NB, kmax), -1, dtype=np.int32)
    for b in range(B):
        for h in range(H):
            kk = kph[h]
            if kk == NB:
                sel[b, h] = np.arange(NB)
                continue
            # families of similar lists, far apart in index
            base = np.array([np.sort(rng.choice(NB, size=kk, replace=False)) for _ in range(NB // 7)])
            sel[b, h, :, :kk] = base[rng.integers(0, NB // 7, size=NB)]
            swap = rng.integers(0, NB, size=NB)
            for i in range(0, NB, 3):
                if swap[i] not in sel[b, h, i, :kk]:
                    sel[b, h, i, kk // 2] = swap[i]
                    sel[b, h, i, :kk] = np.sort(sel[b, h, i, :kk])
            sel[b, h, 5] = -1                                 # a block without keys
            sel[b, h, NB - 3, 1:] = -1                        # holes for all but one entry
            sel[b, h, 40:300] = sel[b, h, 40]                 # more equal lists than a chunk holds
    args = (q, k, v, torch.from_numpy(sel).to(DEV), kph)
    o, o32, lse = usv.sparse_attn_fwd(*args, return_f32=True, return_lse=True, out_f32=torch.full((B, H, N, d), 7e9, device=DEV),
                                      out_lse=torch.full((B, H, N), 7e9, device=DEV))
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0
    assert usv.sparse_attn_fallbacks() <= B * H               # at most the blocks without keys
    _, e32, elxe = usv.sparse_attn_fwd(*args, return_f32=True, return_lse=True, impl=1)
    # both kernels carry the rounding of the weights to bf16 (white-noise V: 1.4e-3 each against the oracle)
    assert ((o32 - e32).double().norm() / e32.double().norm()).item() <= REL_L2_WHITE_NOISE_V
    assert (o32 - e32).abs().max().item() <= MAX_ABS
    assert (lse - elxe).abs().max().item() <= 2e-3
    work = [(b, h, i) for b in range(B) for h in range(H) if kph[h] < NB for i in (0, 5, 41, 299, NB - 3, NB - 1)][:24]
    o_ref, _ = oracle.sparse_attn(q.cpu(), k.cpu(), v.cpu(), N, sel, kph, qb_list=work)
    mx, rl2 = attn_errors(gather_qblocks(o32, work, N), o_ref)
    assert mx <= MAX_ABS and rl2 <= REL_L2_WHITE_NOISE_V, (mx, rl2)
