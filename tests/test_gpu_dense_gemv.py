"""GPU parity of spark_dense_gemv: row counts, widths and token counts at the edges of the kernels' tiles."""
import numpy as np
import pytest
import torch

from paper_2506_06644_b200 import binding as S
from paper_2506_06644_b200 import synth

pytestmark = pytest.mark.gpu


# one piece of a tile per block (few tiles), a single chunk, ragged widths and rows, whole tiles per block (290 tiles), equal
# parts that cut tiles (157 tiles)
@pytest.mark.parametrize("B,n_in,n_out", [(5, 64, 1), (5, 72, 127), (16, 1000, 129), (17, 2304, 4096), (64, 200, 3001), (33, 512, 20001),
                                          (64, 64, 37000), (8, 128, 37120), (1, 1000, 3001), (4, 2048, 300), (2, 72, 129), (3, 1000, 20001), (4, 64, 37120)])
@pytest.mark.parametrize("add", ["none", "other", "alias"])
def test_projection_against_float64(B, n_in, n_out, add):
    W_bits = synth.f32_to_bf16_bits(synth.normal_f32((n_out, n_in), 3, 1, n_in ** -0.5))
    W = synth.bf16_bits_to_f32(W_bits).astype(np.float64)
    x = synth.normal_f32((B, n_in), 3, 2)
    base = synth.normal_f32((B, n_out), 3, 3)
    ctx = S.SparkContext(0, max_batch=B, max_d=n_in)
    Wg, xg = torch.from_numpy(W_bits.view(np.int16)).cuda().view(torch.bfloat16), torch.from_numpy(x).cuda()
    y = torch.from_numpy(base).cuda() if add == "alias" else torch.full((B, n_out), float("nan"), device="cuda")
    y_add = {"none": None, "other": torch.from_numpy(base).cuda(), "alias": y}[add]
    S.spark_dense_gemv(ctx, xg, B, Wg, S.SPARK_BF16, n_in, n_out, y_add, y)
    assert ctx.device_status() == S.SPARK_OK
    ref = x.astype(np.float64) @ W.T + (0 if add == "none" else base.astype(np.float64))
    # the inputs enter as two bf16 terms (2^-17 of each value at most; up to four tokens: three terms, 2^-24), the fp32 accumulator
    # drops up to 2^-23 of the sum of magnitudes at each of its n_in / 16 steps
    bound = ((2.0 ** -17 if B > 4 else 2.0 ** -24) + (n_in / 16 + 4) * 2.0 ** -23) * (np.abs(x).astype(np.float64) @ np.abs(W).T + np.abs(ref)) + 1e-12
    assert np.all(np.abs(y.cpu().numpy() - ref) <= bound)
    ctx.close()
