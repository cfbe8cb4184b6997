"""GPU parity of spark_prefill over spans of a prompt (more than 64 tokens through a layer at once) against token-by-token decoding
in the oracle: token counts at the edges of the 128-token tiles, several spans, every head grouping, partial operand boxes."""
import numpy as np
import pytest
import torch

from oracle import spark_oracle as O
from paper_2506_06644_b200 import binding as S
from paper_2506_06644_b200 import synth
from tests import parity
from tests.test_gpu_layer import bf16_dev

pytestmark = pytest.mark.gpu


def shape(d=256, d_ff=1024, r_ff=128, k_ff=82, n_q=4, n_kv=2, hd=64, r_attn=32, k_attn=16):
    return synth.LayerShape(d=d, d_ff=d_ff, r_ff=r_ff, k_ff=k_ff, n_q=n_q, n_kv=n_kv, hd=hd, r_attn=r_attn, k_attn=k_attn, n_layers=1, vocab=512)


@pytest.mark.parametrize("sh,N,L0,window,flags,max_batch", [
    (shape(), 65, 0, 0, 0, 64),                                                    # the smallest span
    (shape(), 128, 30, 0, 0, 64),                                                  # one full token tile
    (shape(), 129, 5, 50, 0, 64),                                                  # one token in the second tile; local window
    (shape(), 600, 3, 0, 0, 16),                                                   # more than the small workspace holds at once
    (shape(n_q=8, n_kv=1, hd=128, r_attn=64), 150, 20, 0, S.SPARK_GELU_ERF, 64),   # eight heads share a KV head: sixteen tokens a sub-chunk
    (shape(n_q=4, n_kv=4, hd=96, r_attn=32), 200, 0, 100, 0, 64),                  # one head per KV head, unequal parts, partial value boxes
    (shape(n_q=8, n_kv=2, hd=256, r_attn=128, k_attn=300), 140, 2, 0, 0, 64),      # k_attn beyond the window: nothing is thresholded
    (shape(d=200, d_ff=1000, r_ff=72, k_ff=1000), 90, 0, 0, 0, 64),                # ragged widths, every neuron active
])
def test_span_equals_token_by_token_decoding(sh, N, L0, window, flags, max_batch):
    cap = L0 + N + 3
    ctx = S.SparkContext(0, max_batch=max_batch, max_dff=sh.d_ff, max_cap=cap, n_q=sh.n_q, hd=sh.hd, max_d=sh.d)
    lw = synth.layer_weights(sh, 31, 0)
    kv = synth.attn_inputs(1, sh.n_q, sh.n_kv, sh.hd, sh.r_attn, cap, [max(L0, 1)], "bf16", seed=32)
    h0 = synth.normal_f32((N, sh.d), 33, 60)
    dev = dict(norm1=torch.from_numpy(lw.norm1).cuda(), norm2=torch.from_numpy(lw.norm2).cuda(), Wqkv=bf16_dev(lw.Wqkv_bits),
               Wo=bf16_dev(lw.Wo_bits), K1t=bf16_dev(lw.K1t_bits), K2t=bf16_dev(lw.K2t_bits), Vt=bf16_dev(lw.Vt_bits))
    cache = dict(k1c=bf16_dev(kv.k1c_bits[0]), k2c=bf16_dev(kv.k2c_bits[0]), vc=bf16_dev(kv.vc_bits[0]))
    cfg = dict(d=sh.d, d_ff=sh.d_ff, r_ff=sh.r_ff, k_ff=sh.k_ff, n_q=sh.n_q, n_kv=sh.n_kv, hd=sh.hd, r_attn=sh.r_attn, k_attn=sh.k_attn,
               window=window, cap=cap, rms_eps=1e-6, rope_base=10000.0, flags=S.SPARK_SHARED_CACHE | flags)
    h = torch.from_numpy(h0).cuda()
    S.spark_prefill(ctx, [S.make_layer(dev, cfg, cache)], h, L0, chunk=64)
    assert ctx.device_status() == S.SPARK_OK
    ctx.close()
    got = h.cpu().numpy()

    W = {"norm1": lw.norm1, "norm2": lw.norm2, "Wqkv": synth.bf16_bits_to_f32(lw.Wqkv_bits), "Wo": synth.bf16_bits_to_f32(lw.Wo_bits),
         "K1t": synth.bf16_bits_to_f32(lw.K1t_bits), "K2t": synth.bf16_bits_to_f32(lw.K2t_bits), "Vt": synth.bf16_bits_to_f32(lw.Vt_bits)}
    kc = np.concatenate([kv.k1c[0], kv.k2c[0]], axis=-1).astype(np.float64)
    vc = kv.vc[0].astype(np.float64)
    k1g, k2g, vg = (cache[k].float().cpu().numpy().astype(np.float64) for k in ("k1c", "k2c", "vc"))
    for t in range(N):
        n = L0 + t + 1
        kin, vin = kc.copy(), vc.copy()
        kw = dict(n_q=sh.n_q, n_kv=sh.n_kv, hd=sh.hd, r_attn=sh.r_attn, k_attn=sh.k_attn, r_ff=sh.r_ff, k_ff=sh.k_ff, gelu_form="erf" if flags else "tanh")
        best = np.inf
        # a cached token within rounding distance of an attention threshold may fall on either side of it
        for ref in parity.layer_refs_within_band(O, h0[t].astype(np.float64), W, kin, vin, n, window, **kw):
            best = min(best, np.abs(got[t] - ref["h"]).max() / parity.rms(ref["h"]))
            if best <= parity.OUT_TOL["bf16"]:
                break
        assert best <= parity.OUT_TOL["bf16"], (t, best)
        # the stored rows are the oracle's up to one bf16 step; later tokens see the stored ones
        new = np.concatenate([k1g[:, n - 1], k2g[:, n - 1]], axis=-1)
        assert np.all(np.abs(new - kin[:, n - 1]) <= 2.0 ** -7 * np.abs(kin[:, n - 1]) + 1e-4)
        assert np.all(np.abs(vg[:, n - 1] - vin[:, n - 1]) <= 2.0 ** -7 * np.abs(vin[:, n - 1]) + 1e-4)
        kc[:, n - 1], vc[:, n - 1] = new, vg[:, n - 1]
