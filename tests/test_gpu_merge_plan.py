"""The merge plan in one kernel, by one CTA and by a cluster of eight: source counts around the keys a thread holds and past the largest, all tied confidences,
one source merged and all but one, several batch elements.  Integer outputs identical to the oracle's outside the near-tie band,
cosines within 2e-6; large plans against a stable sort of the
confidences, all equal."""
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


@pytest.mark.gpu
@pytest.mark.parametrize("distinct", [0, 5])
@pytest.mark.parametrize("nA", [12288, 12289, 16384, 16385, 32769, 40961, 65536, 90112, 131072, 131073])
def test_plan_of_many_sources(nA, distinct):
    import paper_2512_05754_b200 as usv
    N, B = 2 * nA, 2
    g = torch.Generator(device=DEV).manual_seed(nA)
    x = torch.zeros((B, N, 8), dtype=torch.bfloat16, device=DEV)
    metric = torch.randn((B, N, 1, 64), generator=g, device=DEV).to(torch.bfloat16)
    if distinct:
        metric = metric[:, torch.randint(distinct, (N,), generator=g, device=DEV)].contiguous()
    for r in (1, nA // 3, nA - 1):
        _, plan = usv.token_merge(x, metric, (nA, 1, 2), (1, 1, 2), r, debug=True, window=(0, 0, 0))   # odd tokens are the sources
        src = torch.arange(1, N, 2, device=DEV)
        assert (plan.jstar[:, 1::2] == src - 1).all()
        order = torch.sort(plan.u[:, 1::2], dim=1, descending=True, stable=True).indices[:, :r]
        merged = torch.zeros((B, nA), dtype=torch.bool, device=DEV).scatter_(1, order, True)
        place = torch.where(merged, nA - r + src // 2, torch.cumsum(~merged, 1) - 1)
        assert torch.equal(plan.dst_of[:, 1::2], torch.where(merged, src - 1, -1).int()) and (plan.dst_of[:, 0::2] == -1).all()
        assert torch.equal(plan.pos[:, 1::2], place.int())
        assert torch.equal(plan.pos[:, 0::2], (nA - r + src // 2).int().expand(B, nA))
