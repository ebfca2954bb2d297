"""Top-k selection of short rows, where every score is ranked against all the others: one score, either side of 32 and 64, one to all
kept and a longer output, rows that do not fill a CTA, ties, infinities and NaN (between the negative and the other scores, as in
the longer forms).  Reference: a stable sort."""
import pytest
import torch

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,NBq,NBk", [(1, 1, 1, 1), (1, 3, 7, 5), (2, 4, 32, 32), (1, 5, 33, 33), (1, 2, 64, 64), (1, 3, 500, 64),
                                         (1, 3, 501, 63), (2, 7, 65, 65)])
def test_short_rows(B, H, NBq, NBk):
    import paper_2512_05754_b200 as usv
    g = torch.Generator(device=DEV).manual_seed(NBq * NBk)
    s = torch.randn(B, H, NBq, NBk, generator=g, device=DEV)
    s[:, :, 1::4] = s[:, :, 1::4].round()                       # ties
    s[:, :, 2::8] = 0.0
    s[:, :, 2::16, ::2] = -0.0
    s[:, :, 3::5, NBk // 2] = float("inf")
    s[:, :, 3::5, :NBk // 3] = float("-inf")
    s[:, :, 5::6, NBk // 3] = float("nan")
    kph = [max(1, min(NBk, v)) for v in (1, NBk, NBk // 2, NBk - 1, 7, 2, 33)][:H]
    sel = usv.select_blocks(s, kph, kmax=NBk + 3).cpu()
    key = torch.where(s.isnan(), -1.2e-38, s + 0.0).cpu()         # no score lies between -1.2e-38 and 0
    for h in range(H):
        ref = key[:, h].sort(dim=-1, descending=True, stable=True).indices[..., :kph[h]].sort(-1).values
        assert torch.equal(sel[:, h, :, :kph[h]].long(), ref)
        assert (sel[:, h, :, kph[h]:] == -1).all()
