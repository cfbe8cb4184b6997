"""GPU parity: spark_attn_decode through the C ABI against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import spark_oracle as O
from paper_2506_06644_b200 import binding as S
from paper_2506_06644_b200 import synth
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = S.SparkContext(0, max_batch=8, max_cap=32768, n_q=16, hd=256)
    yield c
    assert c.device_status() == S.SPARK_OK
    c.close()


def to_dev(a: synth.AttnInputs):
    if a.kvdtype == "bf16":
        f = lambda bits: torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
        return f(a.k1c_bits), f(a.k2c_bits), f(a.vc_bits)
    return tuple(torch.from_numpy(x).cuda() for x in (a.k1c, a.k2c, a.vc))


def run_attn(ctx, a: synth.AttnInputs, k_attn, window=0, flags=0, idx_cap=None, dev=None, want_idx=True):
    B = a.q.shape[0]
    k1c, k2c, vc = dev if dev is not None else to_dev(a)
    q = torch.from_numpy(a.q).cuda()
    cl = torch.from_numpy(a.ctx_len).cuda()
    o = torch.full((B, a.n_q, a.hd), float("nan"), device="cuda")
    idx_cap = idx_cap or int(a.ctx_len.max())
    theta = torch.full((B, a.n_q), 9.0, device="cuda")
    count = torch.full((B, a.n_q), -3, dtype=torch.int32, device="cuda") if want_idx else None
    idx = torch.full((B, a.n_q, idx_cap), -1, dtype=torch.int32, device="cuda") if want_idx else None
    S.spark_attn_decode(ctx, q, k1c, k2c, vc, S.SPARK_BF16 if a.kvdtype == "bf16" else S.SPARK_F32, B, a.n_q, a.n_kv,
                        a.hd, a.r, a.cap, cl, window, k_attn, flags, o, theta, count, idx, idx_cap)
    torch.cuda.synchronize()
    return (o.cpu().numpy(), theta.cpu().numpy(), count.cpu().numpy() if want_idx else None,
            idx.cpu().numpy() if want_idx else None)


def compare(a: synth.AttnInputs, out, k_attn, window=0, seqs=None, heads=None):
    o, theta, count, idx = out
    worst = 0.0
    for b in (range(a.q.shape[0]) if seqs is None else seqs):
        n = int(a.ctx_len[b])
        kc = np.concatenate([a.k1c[b], a.k2c[b]], axis=-1)
        ref = O.spark_attention(a.q[b], kc, a.vc[b], n, k_attn, a.r, window)
        lo = 0 if window <= 0 else max(0, n - window)
        override = None
        for h in (range(a.n_q) if heads is None else heads):
            g = h // (a.n_q // a.n_kv)
            s = a.k1c[b, g, lo:n].astype(np.float64) @ a.q[b, h, : a.r].astype(np.float64)
            _, std = O.mean_std(s) if s.size > 1 else (0.0, 1.0)
            std = std if std > 0 else 1.0
            parity.check_theta(theta[b, h], ref["theta"][h], std, f"seq {b} head {h}")
            got = idx[b, h, : count[b, h]]
            assert np.all(idx[b, h, count[b, h]:] == -1)
            assert got.size == 0 or got.min() >= lo
            diff = parity.check_set(got - lo, ref["mask"][h, lo:n], s, ref["theta"][h], std, f"seq {b} head {h}")
            if diff.size:        # the hard threshold is discontinuous: re-evaluate with the GPU's set
                if override is None:
                    override = ref["mask"].copy()
                override[h] = False
                override[h, got] = True
        if override is not None:
            ref = O.spark_attention(a.q[b], kc, a.vc[b], n, k_attn, a.r, window, mask_override=override)
        sel = slice(None) if heads is None else list(heads)
        worst = max(worst, parity.check_output(o[b][sel], ref["o"][sel], a.kvdtype, f"seq {b}"))
    return worst


@pytest.mark.parametrize("ctx_len", [4096, 16384])
def test_gemma2_attention_shape_bf16(ctx, ctx_len):
    # 8 query heads, 4 KV heads, head_dim 256, predictor slice 128, k_attn 256, one sequence
    a = synth.attn_inputs(1, 8, 4, 256, 128, ctx_len, [ctx_len], "bf16", seed=0)
    dev = to_dev(a)
    out = run_attn(ctx, a, 256, dev=dev)
    err = compare(a, out, 256)
    assert err < 5e-3
    sd = {4096: 10.3, 16384: 13.0}[ctx_len]
    assert np.all(np.abs(out[2] - 256) < 6 * sd + 1)
    dense = run_attn(ctx, a, 256, flags=S.SPARK_DENSE_LOADS, dev=dev)
    np.testing.assert_allclose(dense[0], out[0], rtol=0, atol=1e-5 * parity.rms(out[0]))
    assert np.array_equal(dense[2], out[2])
    for b in range(1):
        for h in range(8):
            assert sorted(dense[3][b, h, : dense[2][b, h]]) == sorted(out[3][b, h, : out[2][b, h]])
    plain = run_attn(ctx, a, 256, dev=dev, want_idx=False)
    np.testing.assert_allclose(plain[0], out[0], rtol=0, atol=1e-5 * parity.rms(out[0]))


def test_batch_of_eight_mixed_lengths(ctx):
    lens = [4096, 1, 300, 2049, 4000, 257, 1023, 77]
    a = synth.attn_inputs(8, 8, 4, 256, 128, 4096, lens, "bf16", seed=1)
    out = run_attn(ctx, a, 256)
    compare(a, out, 256)
    # contexts of at most k_attn tokens are attended to densely
    assert out[2][1].tolist() == [1] * 8 and out[2][7].tolist() == [77] * 8
    assert np.all(np.isneginf(out[1][1])) and np.all(np.isneginf(out[1][7]))


def test_full_size_32k_batch8_sampled(ctx):
    """ctx 32768, batch 8 (the largest attention workload): two sequences and three heads are
    checked against the oracle; counts are checked everywhere."""
    a = synth.attn_inputs(8, 8, 4, 256, 128, 32768, [32768] * 8, "bf16", seed=2)
    out = run_attn(ctx, a, 256, idx_cap=1024)
    compare(a, out, 256, seqs=[0, 5], heads=[0, 3, 6])
    assert np.all(np.abs(out[2] - 256) < 6 * 14.0 + 1)


@pytest.mark.parametrize("kv", ["f32", "bf16"])
@pytest.mark.parametrize("n_q,n_kv,hd,r,cap,lens,k_attn,window", [
    (4, 2, 64, 32, 512, [500, 37], 16, 0),
    (4, 4, 64, 32, 300, [300, 299, 150], 40, 100),        # local window, one query head per KV head
    (8, 1, 128, 64, 1000, [999], 64, 0),                  # eight query heads share one KV head
    (16, 8, 256, 128, 700, [650, 700], 256, 512),
    (2, 2, 32, 16, 64, [5, 64, 1, 33], 8, 0),
    (4, 2, 96, 32, 9000, [9000], 100, 4096),              # head_dim 96: unequal halves, window < context
])
def test_shapes_windows_and_groups(ctx, kv, n_q, n_kv, hd, r, cap, lens, k_attn, window):
    a = synth.attn_inputs(len(lens), n_q, n_kv, hd, r, cap, lens, kv, seed=cap)
    out = run_attn(ctx, a, k_attn, window=window)
    compare(a, out, k_attn, window=window)
    if window:
        for b, n in enumerate(lens):
            for h in range(n_q):
                got = out[3][b, h, : out[2][b, h]]
                assert got.size == 0 or got.min() >= max(0, n - window)


def test_special_cases_against_library_attention(ctx):
    # q[r:] = 0 makes every gate ln 2: the result is ln 2 x softmax attention restricted to the selected set
    a = synth.attn_inputs(1, 4, 2, 64, 32, 400, [400], "f32", seed=5)
    a.q[:, :, 32:] = 0.0
    o, theta, count, idx = run_attn(ctx, a, 24)
    for h in range(4):
        g = h // 2
        sel = np.sort(idx[0, h, : count[0, h]])
        tq = torch.from_numpy(a.q[0, h, :32]).double()[None, None, None]
        tk = torch.from_numpy(a.k1c[0, g, sel]).double()[None, None]
        tv = torch.from_numpy(a.vc[0, g, sel]).double()[None, None]
        ref = torch.nn.functional.scaled_dot_product_attention(tq, tk, tv, scale=1.0)[0, 0, 0].numpy() * np.log(2.0)
        parity.check_output(o[0, h], ref, "f32", f"head {h}")


def test_unselected_rows_are_never_read(ctx):
    a = synth.attn_inputs(2, 4, 2, 64, 32, 2048, [2048, 1500], "bf16", seed=6)
    base = run_attn(ctx, a, 64)
    keep = np.zeros((2, 2, 2048), dtype=bool)
    for b in range(2):
        for h in range(4):
            keep[b, h // 2, base[3][b, h, : base[2][b, h]]] = True
    a.k2c_bits[~keep] = 0x7FC0                 # NaN patterns in every unselected row
    a.vc_bits[~keep] = 0x7FC0
    poisoned = run_attn(ctx, a, 64)
    np.testing.assert_allclose(poisoned[0], base[0], rtol=0, atol=1e-5 * parity.rms(base[0]))


def test_empty_selection_gives_zero(ctx):
    hd, r, n = 32, 16, 1024
    a = synth.attn_inputs(1, 1, 1, hd, r, n, [n], "f32", seed=7)
    a.k1c[:] = 0.0
    a.k1c[0, 0, :, 0] = np.linspace(-1, 1, n)
    a.q[:] = 0.0
    a.q[0, 0, 0] = 1.0
    o, theta, count, idx = run_attn(ctx, a, 20)
    assert count[0, 0] == 0 and np.all(o == 0.0) and abs(theta[0, 0] - 1.1931251) < 2e-5


def test_index_list_overflow_is_reported(ctx):
    a = synth.attn_inputs(1, 2, 2, 64, 32, 2000, [2000], "f32", seed=8)
    out = run_attn(ctx, a, 200, idx_cap=50)
    assert np.all(out[2] > 50)
    assert ctx.device_status() == S.SPARK_ERR_OVERFLOW
    assert ctx.device_status() == S.SPARK_OK


def test_argument_errors(ctx):
    a = synth.attn_inputs(1, 4, 2, 64, 32, 128, [100], "f32", seed=9)
    k1c, k2c, vc = to_dev(a)
    q = torch.from_numpy(a.q).cuda()
    cl = torch.from_numpy(a.ctx_len).cuda()
    o = torch.empty((1, 4, 64), device="cuda")

    def call(**kw):
        v = dict(n_q=4, n_kv=2, hd=64, r=32, k=16, window=0)
        v.update(kw)
        S.spark_attn_decode(ctx, q, k1c, k2c, vc, S.SPARK_F32, 1, v["n_q"], v["n_kv"], v["hd"], v["r"], 128, cl,
                            v["window"], v["k"], 0, o, None, None, None, 0)

    for bad, code in ((dict(k=0), 1), (dict(n_kv=3), 1), (dict(r=0), 1), (dict(r=64), 1), (dict(window=-1), 1),
                      (dict(r=36), 2), (dict(n_q=6, n_kv=2), 2)):
        with pytest.raises(S.SparkError) as e:
            call(**bad)
        assert e.value.status == code, bad
    call()
    torch.cuda.synchronize()


@pytest.mark.parametrize("B,n_q,n_kv,hd,r,cap,k_attn", [(3, 4, 2, 256, 128, 32768, 256), (80, 4, 2, 64, 32, 120, 20), (5, 8, 1, 64, 32, 2500, 100), (160, 2, 2, 64, 32, 9, 3)])
def test_blocks_that_span_segments(B, n_q, n_kv, hd, r, cap, k_attn):
    # the flat cut: blocks with two pieces, half of the warps each (long and short ones, one and more warps per head), and with more than two
    lens = [max(1, cap - (7 * b) % max(1, (2 * cap) // 3)) for b in range(B)]
    a = synth.attn_inputs(B, n_q, n_kv, hd, r, cap, lens, "bf16", seed=B)
    c = S.SparkContext(0, max_batch=B, max_cap=cap, n_q=n_q, hd=hd)
    compare(a, run_attn(c, a, k_attn), k_attn, seqs=range(0, B, max(1, B // 12)))
    assert c.device_status() == S.SPARK_OK
    c.close()
