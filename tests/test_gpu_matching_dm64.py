"""The tensor-core matcher at descriptor width 64 where it can go wrong: crowded windows (every source
takes the fp32 scan), exact ties between tiles, odd tile remainders; against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from parity_utils import check_merge_plan

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def usv():
    import paper_2512_05754_b200 as m
    return m


def _plan(usv, metric, grid, part, r):
    N = metric.shape[1]
    x = torch.zeros((metric.shape[0], N, 8), dtype=torch.bfloat16, device=DEV)
    _, plan = usv.token_merge(x, metric.to(DEV), grid, part, r, debug=True)
    torch.cuda.synchronize()
    assert usv.workspace_status() == 0
    pg = dict(dst_of=plan.dst_of.cpu().numpy(), pos=plan.pos.cpu().numpy(), u=plan.u.cpu().numpy(),
              jstar=plan.jstar.cpu().numpy())
    return pg, check_merge_plan(pg, metric, grid, part, r)


# one tile and less, one row beyond a tile, several tiles with a remainder; cut blocks at the edges
@pytest.mark.parametrize("B,grid,part,r", [(1, (1, 5, 7), (1, 2, 2), 9), (2, (2, 3, 43), (1, 1, 2), 100),
                                           (1, (3, 21, 33), (2, 2, 2), 700), (1, (5, 13, 29), (1, 1, 2), 500)])
def test_dm64_sizes(usv, B, grid, part, r):
    N = grid[0] * grid[1] * grid[2]
    g = torch.Generator().manual_seed(N)
    metric = torch.randn(B, N, 3, 64, generator=g).to(torch.bfloat16)
    _plan(usv, metric, grid, part, r)


def test_dm64_crowded_windows_and_exact_ties(usv):
    grid, part, N = (4, 12, 32), (1, 1, 2), 1536
    g = torch.Generator().manual_seed(78)
    proto = torch.randn(5, 2, 64, generator=g)
    metric = proto[torch.randint(0, 5, (N,), generator=g)] + 1e-4 * torch.randn(N, 2, 64, generator=g)
    _plan(usv, metric.unsqueeze(0).to(torch.bfloat16), grid, part, 300)
    # three destinations in different tiles that equal a source: the lowest wins
    metric = torch.randn(N, 2, 64, generator=g)
    dst = np.nonzero(oracle.destination_mask(grid, part))[0]
    cases = {}
    for i, a in enumerate((7, 401, 1201)):
        trio = dst[[17 + 40 * i, 148 + 40 * i, 407 + 40 * i]]
        for j in trio:
            metric[j] = metric[a]
        cases[a] = int(trio.min())
    pg, stats = _plan(usv, metric.unsqueeze(0).to(torch.bfloat16), grid, part, 768)
    assert stats["jstar_differ"] == 0
    for a, j in cases.items():
        assert pg["jstar"][0, a] == j and abs(pg["u"][0, a] - 1.0) < 1e-6
