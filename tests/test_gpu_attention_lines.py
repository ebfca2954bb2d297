"""Attention calls on either side of the limits up to which they run without a pairing plan (key blocks kept over all query
blocks, and query blocks, at either head width), as in test_gpu_attention_direct: holes, blocks without keys, rows handed to the exact
kernel, against the mma.sync kernel, with the bounds stated there."""
import pytest
import test_gpu_attention_direct as direct
import torch

from parity_utils import attention_path


@pytest.mark.gpu
@pytest.mark.parametrize("d,B,H,NB,kph,cut", [
    (64, 1, 9, 200, [20] * 9, 3), (64, 1, 9, 200, [21] + [20] * 8, 0), (64, 1, 12, 200, [10] * 12, 1), (64, 2, 6, 201, [9] * 6, 0),
    (128, 1, 10, 170, [12, 11] * 5, 0), (128, 1, 10, 170, [12] * 10, 5), (128, 1, 23, 100, [5, 6] * 11 + [8], 0),
    (128, 1, 23, 101, [5] * 23, 2), (128, 2, 40, 33, [2] * 40, 1)])
def test_lines(d, B, H, NB, kph, cut):
    direct.test_small_calls(d, B, H, NB, kph, cut)


# short and long lists, whole and nearly empty last waves of items (on 148 SMs); full lists
@pytest.mark.gpu
@pytest.mark.parametrize("path,d,H,NB,k", [
    ("no plan", 64, 12, 150, 20), ("no plan", 64, 8, 90, 36), ("plan", 64, 4, 150, 53), ("no plan", 64, 4, 140, 53), ("no plan", 64, 4, 150, 40), ("plan", 64, 2, 180, 90),
    ("no plan", 64, 1, 250, 125), ("plan", 64, 12, 30, 30), ("no plan", 64, 12, 28, 28), ("no plan", 64, 12, 30, 29), ("no plan", 128, 12, 30, 29),
    ("plan", 128, 100, 13, 13), ("no plan", 128, 60, 12, 12), ("plan", 128, 6, 120, 30)])
def test_paths(path, d, H, NB, k):
    import paper_2512_05754_b200 as usv
    g = torch.Generator(device="cuda:0").manual_seed(NB)
    q, kk, v = (torch.randn(1, H, 64 * NB, d, generator=g, device="cuda:0").to(torch.bfloat16) for _ in range(3))
    sel = torch.rand(1, H, NB, NB, generator=g, device="cuda:0").topk(k, -1).indices.sort(-1).values.int()
    assert attention_path(lambda: usv.sparse_attn_fwd(q, kk, v, sel, [k] * H), H * NB) == path
