"""The merge plan of few sources in one kernel: source counts around the keys a thread holds and past the largest, all tied confidences,
one source merged and all but one, several batch elements.  Integer outputs identical to the oracle's outside the near-tie band,
cosines within 2e-6."""
import pytest
import torch

from parity_utils import check_merge_plan

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("distinct", [0, 3])
@pytest.mark.parametrize("grid,nA", [((1, 2, 2), 2), ((1, 3, 22), 33), ((2, 32, 32), 1024), ((1, 41, 50), 1025), ((4, 32, 32), 2048),
                                     ((1, 3, 1366), 2049), ((6, 32, 32), 3072), ((1, 7, 878), 3073)])
def test_plan_of_few_sources(grid, nA, distinct):
    import paper_2512_05754_b200 as usv
    N, part, win, B = grid[0] * grid[1] * grid[2], (1, 1, 2), (1, 1, 1), 2
    assert N // 2 == nA
    g = torch.Generator().manual_seed(N + distinct)
    x = torch.randn((B, N, 64), generator=g).to(torch.bfloat16)
    metric = torch.randn((B, N, 1, 64), generator=g).to(torch.bfloat16)
    if distinct:     # equal rows: confidences and destinations tie
        metric = metric[:, torch.randint(distinct, (N,), generator=g)].contiguous()
    for r in {1, nA // 2, nA - 1}:
        _, plan = usv.token_merge(x.to(DEV), metric.to(DEV), grid, part, r, debug=True, window=win)
        torch.cuda.synchronize()
        pg = {k: getattr(plan, k).cpu().numpy() for k in ("dst_of", "pos", "u", "jstar")}
        check_merge_plan(pg, metric, grid, part, r, window=win)
