"""Lists of merged sources per destination at the sizes where they change form: up to four sources in
the destination's own slots, a chain up to 32, a pass over the plan beyond; from a fresh plan, from a
stored one and through the plan cache, against the oracle's merge of the same plan."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import bf16_ulp_distance, bits

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def usv():
    import paper_2512_05754_b200 as m
    return m


@pytest.mark.parametrize("C", [72, 776])
def test_list_lengths(usv, C):
    grid, part = (2, 12, 16), (1, 1, 2)                      # 192 sources, 192 destinations
    B, N = 2, 384
    dst = np.nonzero(oracle.destination_mask(grid, part))[0]
    src = np.nonzero(~oracle.destination_mask(grid, part))[0]
    g = torch.Generator().manual_seed(C)
    metric = torch.randn(B, N, 2, 64, generator=g)
    want = np.full((B, N), -1)
    for b in range(B):
        rest = list(np.random.default_rng(b).permutation(src))
        for t, n in enumerate([1, 2, 3, 4, 5, 6, 31, 32, 33, 60]):
            for _ in range(n):
                i = rest.pop()
                metric[b, i] = metric[b, dst[7 * t + b]]
                want[b, i] = dst[7 * t + b]
    x = torch.randn(B, N, C, generator=g).to(torch.bfloat16)
    r = int((want[0] >= 0).sum())
    xm, plan = usv.token_merge(x.to(DEV), metric.to(torch.bfloat16).to(DEV), grid, part, r)
    dst_of, pos = plan.dst_of.cpu().numpy(), plan.pos.cpu().numpy()
    assert np.array_equal(dst_of, want)
    ref = oracle.round_to_bf16(oracle.merge_apply(x, dst_of, pos, N - r))
    assert bf16_ulp_distance(bits(xm), ref).max() <= 1       # the fp64 mean rounds once, the fp32 one twice
    stored, _ = usv.token_merge(x.to(DEV), None, grid, part, r, plan=plan)
    assert torch.equal(stored, xm) and torch.equal(usv.token_merge_apply(x.to(DEV), plan), xm)
