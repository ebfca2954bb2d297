"""Attention calls on either side of the limits up to which they run without a pairing plan (key blocks kept over all query
blocks, and query blocks, at either head width), as in test_gpu_attention_direct: holes, blocks without keys, rows handed to the exact
kernel, against the mma.sync kernel, with the bounds stated there."""
import pytest
import test_gpu_attention_direct as direct


@pytest.mark.gpu
@pytest.mark.parametrize("d,B,H,NB,kph,cut", [
    (64, 1, 9, 200, [20] * 9, 3), (64, 1, 9, 200, [21] + [20] * 8, 0), (64, 1, 12, 200, [10] * 12, 1), (64, 2, 6, 201, [9] * 6, 0),
    (128, 1, 10, 170, [12, 11] * 5, 0), (128, 1, 10, 170, [12] * 10, 5), (128, 1, 23, 100, [5, 6] * 11 + [8], 0),
    (128, 1, 23, 101, [5] * 23, 2), (128, 2, 40, 33, [2] * 40, 1)])
def test_lines(d, B, H, NB, kph, cut):
    direct.test_small_calls(d, B, H, NB, kph, cut)
