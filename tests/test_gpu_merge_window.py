"""Matching inside a window, at the sizes where the kernel changes its way: rows of three destinations (30 candidates at a time, so a
second group, and a part of one), rows of two at the grid's edges, one column of blocks, CTAs that go through several sources, and the
own block alone.  Chosen destinations identical to the oracle's outside the near-tie band, cosines within 2e-6."""
import pytest
import torch

from parity_utils import check_merge_plan

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("grid,part,win,dm,B", [
    ((7, 9, 8), (1, 1, 2), (2, 1, 1), 128, 2),       # 12 to 45 candidates
    ((9, 11, 6), (1, 2, 2), (4, 2, 1), 64, 1),       # up to 135, five groups
    ((5, 8, 4), (1, 1, 2), (1, 1, 1), 128, 1),       # two columns of blocks
    ((5, 8, 2), (1, 1, 2), (1, 1, 1), 64, 1),        # one
    ((17, 30, 36), (1, 1, 2), (0, 0, 1), 128, 2),    # one row of three; several sources a warp
    ((17, 30, 36), (2, 2, 2), (1, 1, 1), 64, 1),
    ((17, 30, 36), (2, 2, 2), (0, 0, 0), 64, 2),     # the own block alone, several sources a warp
    ((17, 30, 36), (2, 2, 2), (0, 0, 0), 128, 1),
])
def test_window(grid, part, win, dm, B):
    import paper_2512_05754_b200 as usv
    N = grid[0] * grid[1] * grid[2]
    g = torch.Generator().manual_seed(N + dm)
    x = torch.randn((B, N, 64), generator=g).to(torch.bfloat16)
    metric = torch.randn((B, N, 2, dm), generator=g).to(torch.bfloat16)
    r = N // 4
    _, plan = usv.token_merge(x.to(DEV), metric.to(DEV), grid, part, r, debug=True, window=win)
    torch.cuda.synchronize()
    pg = {k: getattr(plan, k).cpu().numpy() for k in ("dst_of", "pos", "u", "jstar")}
    check_merge_plan(pg, metric, grid, part, r, window=win)
