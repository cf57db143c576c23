"""Per-kernel parity: each C-ABI kernel call against the matching oracle sub-step on the
same seeded inputs (small and odd shapes spanning several tiles and ragged tails)."""
import math

import numpy as np
import pytest
import torch

import synth
from oracle import marche_oracle as orc
from helpers import (TOL, assert_close, dev, host, idx_dev, make_model, max_abs, rel_l2)

pytestmark = pytest.mark.gpu


def model_for(dtype, D, H, F, S, B, L=1):
    """dtype "f32", "bf16" (bf16 cache, fp16 projection operands) or "bf16b" (bf16 throughout)."""
    cfg = synth.CONFIGS["tiny"].replace(L=L, E=0, D=D, H=H, F=F, S=S, B=B, dtype="f32" if dtype == "f32" else "bf16",
                                        n_buffer=0)
    blocks = synth.make_weights(cfg)
    return cfg, blocks, make_model(cfg, blocks, operand="bf16" if dtype == "bf16b" else "f16")


def tdt(dtype):
    """element type of q/k/v and the K/V cache"""
    return torch.float32 if dtype == "f32" else torch.bfloat16


def adt(dtype):
    """element type of the projections' operands: weight matrices and the activations that feed them"""
    return {"f32": torch.float32, "bf16": torch.float16, "bf16b": torch.bfloat16}[dtype]


def quant_a(a, dtype):
    """What the device holds for a projection operand."""
    a = np.asarray(a, np.float32)
    if dtype == "bf16":
        return a.astype(np.float16).astype(np.float64)
    return synth.round_to_bf16(a).astype(np.float64) if dtype == "bf16b" else a.astype(np.float64)


def quant(a, dtype):
    """What the device holds for q/k/v and cache entries."""
    return np.asarray(a, np.float32).astype(np.float64) if dtype == "f32" else synth.round_to_bf16(a).astype(np.float64)


LOW = ("bf16", "bf16b")        # the 16-bit contexts


# ------------------------------------------------------------------ K1 gather + LayerNorm
@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
@pytest.mark.parametrize("D,H", [(256, 4), (768, 12), (1024, 16), (1280, 16)])
@pytest.mark.parametrize("n", [1, 2, 41, 68])
def test_gather_layernorm(dtype, D, H, n):
    S, B = 68, 3
    cfg, blocks, m = model_for(dtype, D, H, 128, S, B)
    rng = np.random.default_rng(n + D)
    hidden = rng.standard_normal((B, S, D)).astype(np.float32)
    hidden[0] += 100.0                                   # large mean: variance cancellation
    patterns = [np.stack([rng.permutation(S)[:n] for _ in range(B)]),
                np.tile(np.arange(S - 1, S - 1 - n, -1), (B, 1))]
    g, be = blocks[0]["ln1_g"], blocks[0]["ln1_b"]
    for idx in patterns:
        x_out = torch.full((B * n, D), -7.0, device="cuda")
        u_out = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
        m.gather_layernorm(dev(hidden), idx_dev(idx), n, dev(g), dev(be), x_out, u_out)
        X = np.stack([hidden[b, idx[b]] for b in range(B)]).reshape(B * n, D)
        assert np.array_equal(x_out.cpu().numpy(), X)                       # the gather is a copy: exact
        want = orc.layer_norm(X.astype(np.float64), g.astype(np.float64), be.astype(np.float64), cfg.ln_eps)
        assert_close(host(u_out), want, dtype, "LN", scale=1.0 if dtype in LOW else 10.0)
    # identity index (idx NULL), no compact copy
    u_out = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
    m.gather_layernorm(dev(hidden), None, n, dev(g), dev(be), None, u_out)
    want = orc.layer_norm(hidden[:, :n].reshape(B * n, D).astype(np.float64), g.astype(np.float64),
                          be.astype(np.float64), cfg.ln_eps)
    assert_close(host(u_out), want, dtype, "LN identity", scale=1.0 if dtype in LOW else 10.0)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("D", [256, 2048])
def test_gather_layernorm_of_parameters_just_gathered(dtype, D):
    """gamma and beta come from the call right before (rows picked from a table): few rows, whose launch is set up while
    that call still runs, must not read them before it has written them."""
    S, B, n = 320, 2, 41
    cfg, blocks, m = model_for(dtype, D, D // 64, 128, S, B)
    gen = torch.Generator(device="cuda").manual_seed(D)
    table, x = torch.randn(B, S, D, generator=gen, device="cuda"), torch.randn(B, S, D, generator=gen, device="cuda")
    xn = torch.nn.functional.layer_norm(x[:, :n].double(), (D,), eps=cfg.ln_eps).reshape(B * n, D)
    picked = torch.zeros(B, S, D, device="cuda")
    u = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
    for t in range(8):
        order = torch.randperm(S, generator=gen, device="cuda").to(torch.int32).expand(B, S).contiguous()
        m.gather_rows(table, order, picked)
        m.gather_layernorm(x, None, n, picked[1, S - 2], picked[1, S - 1], None, u)
        want = xn * table[1, order[0, S - 2]].double() + table[1, order[0, S - 1]].double()
        assert (u.double() - want).abs().max() <= (2e-2 if dtype in LOW else 1e-4)     # |want| < 32: half an fp16 step 8e-3


# ------------------------------------------------------------------ K2 projections
@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
@pytest.mark.parametrize("M", [1, 24, 62, 129, 300])
@pytest.mark.parametrize("N,K", [(768, 256), (256, 256), (1024, 256), (256, 1024), (384, 128), (128, 320)])
def test_linear_all_epilogues(dtype, M, N, K):
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(M * 7 + N + K)
    a = rng.standard_normal((M, K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    aq, wq = quant_a(a, dtype), quant_a(w, dtype)
    acc = orc.linear(aq, wq, bias.astype(np.float64))
    a_d, w_d, b_d = dev(a, adt(dtype)), dev(w, adt(dtype)), dev(bias)
    ma, rl = TOL[dtype]
    # bias
    out = torch.zeros(M, N, dtype=tdt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 0, out)
    assert rel_l2(host(out), acc) <= (4e-3 if dtype in LOW else 1e-6)
    assert max_abs(host(out), acc) <= (3e-2 if dtype in LOW else 1e-4)
    # bias + residual (fp32 read-modify-write)
    res = rng.standard_normal((M, N)).astype(np.float32)
    out = dev(res)
    m.linear(a_d, w_d, b_d, 1, out)
    assert max_abs(host(out), acc + res) <= 1e-4 * max(1.0, math.sqrt(K / 256))
    # bias + GELU
    out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 2, out)
    want = orc.gelu(acc)
    assert rel_l2(host(out), want) <= (4e-3 if dtype in LOW else 1e-6)
    assert max_abs(host(out), want) <= (3e-2 if dtype in LOW else 1e-4)


@pytest.mark.parametrize("dtype", ["bf16", "bf16b"])
def test_gelu_epilogue_over_the_whole_input_range(dtype):
    """The GELU of the tensor-core epilogue (a polynomial for erf, saturating beyond |x| = 3 sqrt 2) against the
    oracle's erf GELU on a dense grid: a selection matrix as the weight and the grid as bias make the accumulator
    equal the grid value exactly, so the only differences are the approximation and the 16-bit rounding of the
    result.  Grid: -12 .. 12 in steps of 1/512 (covers the fitted range, the clamp point and the saturated tails),
    plus large magnitudes up to the fp16 maximum."""
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    M, N, K = 128, 12288 + 128, 64
    grid = np.concatenate([np.arange(-12.0, 12.0, 1.0 / 512.0),
                           np.array([-65000.0, -1000.0, -100.0, -13.0, 13.0, 100.0, 1000.0, 60000.0]),
                           np.zeros(120)]).astype(np.float32)
    assert grid.shape[0] == N
    a = np.zeros((M, K), np.float32)                                    # accumulator = bias exactly
    w = np.zeros((N, K), np.float32)
    out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
    m.linear(dev(a, adt(dtype)), dev(w, adt(dtype)), dev(grid), 2, out)
    torch.cuda.synchronize()
    got = host(out)
    assert (got == got[0:1]).all()                                      # every row the same function of the bias
    want = orc.gelu(grid.astype(np.float64))
    if dtype == "bf16":                                                 # fp16 result: saturates at 65504
        want = np.clip(want, -65504.0, 65504.0)
    eps = 2.0 ** -11 if dtype == "bf16" else 2.0 ** -8                  # half an ulp, relative
    err = np.abs(got[0] - want)
    bound = eps * np.abs(want) + 1.0e-4                                 # rounding + the approximation (<= 4.8e-5)
    worst = int(np.argmax(err - bound))
    assert (err <= bound).all(), "x = %g: got %g, want %g" % (grid[worst], got[0][worst], want[worst])
    assert (got[0][grid <= -13.0] == 0).all() and np.isfinite(got).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
def test_linear_strided_input_and_row_guard(dtype):
    """a is a column slice of a wider matrix (lda > K); rows >= M of `out` stay untouched."""
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(5)
    M, N, K = 70, 256, 256
    wide = rng.standard_normal((M, 3 * K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    wide_d = dev(wide, adt(dtype))
    out = torch.full((M + 60, N), 5.0, dtype=tdt(dtype), device="cuda")
    m.linear(wide_d[:, K:2 * K], dev(w, adt(dtype)), dev(bias), 0, out, M=M, lda=3 * K)
    want = orc.linear(quant_a(wide[:, K:2 * K], dtype), quant_a(w, dtype), bias.astype(np.float64))
    assert rel_l2(host(out[:M]), want) <= (4e-3 if dtype in LOW else 1e-6)
    assert (host(out[M:]) == 5.0).all()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
@pytest.mark.parametrize("gemm_kernel", [0, 1, 2])
def test_linear_of_no_rows(dtype, gemm_kernel):
    """M = 0 is a valid call that enqueues nothing, whichever kernel would run."""
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    m.set_tuning(gemm_kernel=gemm_kernel)
    a, w, bias = torch.zeros(8, 256, dtype=adt(dtype), device="cuda"), torch.zeros(512, 256, dtype=adt(dtype), device="cuda"), torch.zeros(512, device="cuda")
    for epi, t in ((0, tdt(dtype)), (1, torch.float32), (2, adt(dtype))):
        out = torch.full((8, 512), 5.0, dtype=t, device="cuda")
        m.linear(a, w, bias, epi, out, M=0)
        assert (out == 5.0).all()


# ------------------------------------------------------------------ K5 scatter
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n", [1, 7, 41])
def test_scatter_kv_and_untouched_rows(dtype, n):
    S, B, D = 68, 3, 256
    cfg, blocks, m = model_for(dtype, D, 4, 128, S, B)
    rng = np.random.default_rng(n)
    qkv = dev(rng.standard_normal((B * n, 3 * D)).astype(np.float32), tdt(dtype))
    cache = dev(rng.standard_normal((2, B, S, D)).astype(np.float32), tdt(dtype))
    before = cache.clone()
    idx = np.stack([rng.permutation(S)[:n] for _ in range(B)]).astype(np.int32)
    m.scatter_kv(qkv[:, D:], qkv[:, 2 * D:], 3 * D, idx_dev(idx), n, cache)
    torch.cuda.synchronize()
    want = before.clone()
    q3 = qkv.view(B, n, 3 * D)
    for b in range(B):
        want[0, b, torch.as_tensor(idx[b], dtype=torch.long)] = q3[b, :, D:2 * D]
        want[1, b, torch.as_tensor(idx[b], dtype=torch.long)] = q3[b, :, 2 * D:]
    assert torch.equal(cache, want)                                     # byte-identical everywhere


def test_scatter_rows_and_build_active():
    S, B, D = 68, 3, 256
    cfg, blocks, m = model_for("f32", D, 4, 128, S, B)
    rng = np.random.default_rng(0)
    rows = dev(rng.standard_normal((B, 5, D)).astype(np.float32))
    idx = np.stack([rng.permutation(S)[:5] for _ in range(B)]).astype(np.int32)
    dst = torch.full((B, S, D), 3.0, device="cuda")
    m.scatter_rows(rows, idx_dev(idx), dst)
    want = torch.full((B, S, D), 3.0, device="cuda")
    for b in range(B):
        want[b, torch.as_tensor(idx[b], dtype=torch.long)] = rows[b]
    assert torch.equal(dst, want)
    G, N, R = idx[:, :2], idx[:, 2:3], idx[:, 3:]
    act = torch.zeros(B, 5, dtype=torch.int32, device="cuda")
    m.build_active(idx_dev(G), idx_dev(N), idx_dev(R), 2, act)
    assert np.array_equal(act.cpu().numpy(), orc.active_set(G, N, R))
    act2 = torch.zeros(B, 2, dtype=torch.int32, device="cuda")
    m.build_active(idx_dev(G), None, None, 0, act2)
    assert np.array_equal(act2.cpu().numpy(), G)


# ------------------------------------------------------------------ K3 attention (+ scores)
@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
@pytest.mark.parametrize("S", [68, 320])
@pytest.mark.parametrize("dh,H", [(64, 4), (80, 2)])
@pytest.mark.parametrize("n,nG", [(1, 1), (2, 0), (12, 7), (41, 25), (77, 77)])
def test_attention_and_score_partials(dtype, S, dh, H, n, nG):
    if n > S:
        pytest.skip("n > S")
    B, D = 2, dh * H
    if D % 128:
        H = {64: 4, 80: 8}[dh]
        D = dh * H
    cfg, blocks, m = model_for(dtype, D, H, 128, S, B)
    rng = np.random.default_rng(S + n + dh)
    gain = 3.0                                                       # logits of order a few units
    q = (rng.standard_normal((B * n, 3 * D)) * gain).astype(np.float32)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    flags = np.zeros((B, n), dtype=np.uint8)
    for b in range(B):
        flags[b, rng.permutation(n)[:nG]] = 1
    q_d = dev(q, tdt(dtype))
    o = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
    partial = torch.full((B, H, S), -1.0, device="cuda")
    m.attention(q_d, 3 * D, n, dev(cache, tdt(dtype)), dev(flags), partial, o)
    qq, cc = quant(q, dtype), quant(cache, dtype)
    want_o = np.zeros((B * n, D))
    want_p = np.zeros((B, H, S))
    for b in range(B):
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            z, p = orc.softmax_attention(qq[b * n:(b + 1) * n, c], cc[0, b][:, c], cc[1, b][:, c])
            want_o[b * n:(b + 1) * n, c] = z
            want_p[b, h] = p[flags[b].astype(bool)].sum(axis=0)
    got_o, got_p = host(o), host(partial)
    assert rel_l2(got_o, want_o) <= (8e-3 if dtype in LOW else 1e-5)
    assert max_abs(got_o, want_o) <= (3e-2 if dtype in LOW else 1e-4)
    assert max_abs(got_p, want_p) <= (2e-2 if dtype in LOW else 1e-5) * max(1, nG) / 8 + 1e-6
    assert np.allclose(got_p.sum(-1), nG, rtol=(5e-3 if dtype in LOW else 1e-5), atol=1e-6)   # each row sums to 1
    # scores off: partial buffer untouched
    partial2 = torch.full((B, H, S), -1.0, device="cuda")
    m.attention(q_d, 3 * D, n, dev(cache, tdt(dtype)), None, partial2, o)
    assert (partial2 == -1.0).all()


@pytest.mark.parametrize("S", [68, 320, 1088])
@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("n,nG", [(1, 1), (12, 7), (41, 5), (77, 0), (130, 25)])
def test_two_segment_attention_equals_scatter_then_attend(S, dh, H, n, nG):
    """The two-segment kernel (Eq. 6-10 + write-back) against the oracle's plain attention over
    the updated cache, and bit-exact cache contents against marche_scatter_kv."""
    if n > S:
        pytest.skip("n > S")
    B, D = 2, dh * H
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    rng = np.random.default_rng(S + n + dh)
    qkv = (rng.standard_normal((B * n, 3 * D)) * np.array([3.0] * D + [1.0] * 2 * D)).astype(np.float32)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    idx = np.stack([rng.permutation(S)[:n] for _ in range(B)]).astype(np.int32)
    flags = np.zeros((B, n), dtype=np.uint8)
    for b in range(B):
        flags[b, rng.permutation(n)[:nG]] = 1
    qkv_d = dev(qkv, torch.bfloat16)
    cache_a, cache_b = dev(cache, torch.bfloat16), dev(cache, torch.bfloat16)
    o_a = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
    p_a = torch.full((B, H, S), -1.0, device="cuda")
    m.attention_two_segment(qkv_d, 3 * D, n, idx_dev(idx), cache_a, dev(flags), p_a, o_a)
    m.scatter_kv(qkv_d[:, D:], qkv_d[:, 2 * D:], 3 * D, idx_dev(idx), n, cache_b)
    torch.cuda.synchronize()
    assert m.device_status() == 0
    assert torch.equal(cache_a, cache_b)                               # write-back: byte-identical
    qq, cc = quant(qkv, "bf16"), host(cache_b)
    want_o, want_p = np.zeros((B * n, D)), np.zeros((B, H, S))
    for b in range(B):
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            z, p = orc.softmax_attention(qq[b * n:(b + 1) * n, c], cc[0, b][:, c], cc[1, b][:, c])
            want_o[b * n:(b + 1) * n, c] = z
            want_p[b, h] = p[flags[b].astype(bool)].sum(axis=0)
    assert rel_l2(host(o_a), want_o) <= 8e-3 and max_abs(host(o_a), want_o) <= 3e-2
    assert max_abs(host(p_a), want_p) <= 2e-2 * max(1, nG) / 8 + 1e-6
    assert np.allclose(host(p_a).sum(-1), nG, rtol=5e-3, atol=1e-6)


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16b"])
def test_attention_uniform_and_peaked(dtype):
    S, B, H, dh, n = 68, 2, 4, 64, 5
    D = H * dh
    cfg, blocks, m = model_for(dtype, D, H, 128, S, B)
    rng = np.random.default_rng(1)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    flags = np.ones((B, n), dtype=np.uint8)
    # q = 0 -> uniform weights: o = mean of V, partial = n / S
    o = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
    partial = torch.zeros(B, H, S, device="cuda")
    m.attention(torch.zeros(B * n, D, dtype=tdt(dtype), device="cuda"), D, n, dev(cache, tdt(dtype)), dev(flags),
                partial, o)
    vm = quant(cache, dtype)[1].mean(axis=1)
    assert max_abs(host(o).reshape(B, n, D), np.repeat(vm[:, None], n, 1)) <= (4e-3 if dtype in LOW else 1e-5)
    assert np.allclose(host(partial), n / S, rtol=1e-3 if dtype in LOW else 1e-5)
    # q = 64 * k_t -> one-hot on key t: o = V[t]; no inf/nan
    tsel = rng.integers(0, S, size=(B, n))
    kq = quant(cache, dtype)
    q = np.stack([kq[0, b, tsel[b]] for b in range(B)]).reshape(B * n, D) * 64.0
    m.attention(dev(q.astype(np.float32), tdt(dtype)), D, n, dev(cache, tdt(dtype)), dev(flags), partial, o)
    got = host(o).reshape(B, n, D)
    assert np.isfinite(got).all()
    for b in range(B):
        assert max_abs(got[b], kq[1, b, tsel[b]]) <= (2e-2 if dtype in LOW else 1e-4)
    assert np.allclose(host(partial).sum(-1), n, rtol=1e-3)


# ------------------------------------------------------------------ K4 top-k (bit-exact)
@pytest.mark.parametrize("S,k", [(5, 2), (68, 7), (320, 32), (320, 0), (320, 311), (1088, 109), (1088, 1), (2048, 205),
                                 (2048, 2043), (33, 28)])
def test_select_refresh_bit_exact(S, k):
    B = 4
    cfg, blocks, m = model_for("f32", 128, 2, 128, S, B)
    rng = np.random.default_rng(S * 3 + k)
    n_new, n_excl = (2, 3) if S > 5 else (1, 1)
    kinds = [rng.random((B, S)), np.ones((B, S)), rng.integers(0, 3, (B, S)).astype(float),
             rng.random((B, S)) * 1e-42, np.exp(rng.uniform(-80, 10, (B, S))), np.zeros((B, S))]
    kinds[5][:, ::2] = -0.0
    mask = torch.empty(B * S, dtype=torch.uint8, device="cuda")
    for sc in kinds:
        sc = sc.astype(np.float32)
        perm = np.stack([rng.permutation(S) for _ in range(B)]).astype(np.int32)
        for new, excl in ((perm[:, :n_new], perm[:, n_new:n_new + n_excl]), (perm[:, :n_new], None),
                          (np.tile(np.arange(n_new, dtype=np.int32), (B, 1)), np.tile(np.arange(S - n_excl, S, dtype=np.int32), (B, 1)))):
            kk = min(k, S - n_new - (0 if excl is None else n_excl))
            out = torch.full((B, max(kk, 1)), -1, dtype=torch.int32, device="cuda")
            m.select_refresh(dev(sc), idx_dev(new), None if excl is None else idx_dev(excl), kk, out, mask)
            want = orc.select_refresh(sc, new, excl, kk)
            if kk:
                assert np.array_equal(out.cpu().numpy(), want)
            else:
                assert (out.cpu().numpy() == -1).all()


@pytest.mark.parametrize("policy,name", [(0, "high"), (1, "low"), (2, "random")])
def test_select_refresh_policies_bit_exact(policy, name):
    B, S, k = 5, 320, 32
    cfg, blocks, m = model_for("f32", 128, 2, 128, S, B)
    rng = np.random.default_rng(policy)
    mask = torch.empty(B * S, dtype=torch.uint8, device="cuda")
    for sc in (rng.random((B, S)), rng.integers(0, 4, (B, S)).astype(float), np.zeros((B, S))):
        sc = sc.astype(np.float32)
        perm = np.stack([rng.permutation(S) for _ in range(B)]).astype(np.int32)
        new, excl = perm[:, :4], perm[:, 4:9]
        out = torch.full((B, k), -1, dtype=torch.int32, device="cuda")
        m.select_refresh_policy(dev(sc), idx_dev(new), idx_dev(excl), k, policy, 1234, out, mask)
        assert np.array_equal(out.cpu().numpy(), orc.select_refresh(sc, new, excl, k, policy=name, seed=1234))


@pytest.mark.parametrize("S,k", [(33, 9), (320, 32), (1088, 700)])
def test_select_refresh_many_samples_bit_exact(S, k):
    """More samples than run at once (a crowded bin of one score goes straight to the indices): scores of few values, of one, and
    of a few spread ones in one crowded bin; distinct ones."""
    B = 800
    cfg, blocks, m = model_for("f32", 128, 2, 128, S, B)
    rng = np.random.default_rng(S + k)
    mask = torch.empty(B * S, dtype=torch.uint8, device="cuda")
    perm = np.stack([rng.permutation(S) for _ in range(B)]).astype(np.int32)
    new, excl = perm[:, :3], perm[:, 3:7]
    near = 1.0 + rng.integers(0, 40, (B, S)) * 2.0 ** -23
    near[:, 0], near[:, 1] = 1e-30, 1e30
    for sc in (rng.integers(0, 3, (B, S)), np.ones((B, S)), near, rng.random((B, S))):
        sc = sc.astype(np.float32)
        out = torch.full((B, k), -1, dtype=torch.int32, device="cuda")
        m.select_refresh(dev(sc), idx_dev(new), idx_dev(excl), k, out, mask)
        assert np.array_equal(out.cpu().numpy(), orc.select_refresh(sc, new, excl, k))


@pytest.mark.parametrize("F,S,B", [(2048, 300, 64), (4096, 320, 64), (3072, 330, 100)])
def test_fc2_shared_tiles_equal_whole_tiles(F, S, B):
    """75, 80 and 129 tiles of 256 x 256 dealt to the CTA pairs in whole tiles or in ranges of 5/4, 9/8 and 7/4 tiles (74
    pairs), where a pair completes what its neighbour began.  Everything before fc2 is the same launch; the sums of K
    terms of order 1/16 differ by sqrt(K) 2^-24 at most, the additions to |hidden| < 8 by half a step, 2.4e-7, each."""
    cfg, blocks, m = model_for("bf16", 256, 4, F, S, B)
    hidden = torch.randn(B, S, 256, device="cuda", generator=torch.Generator(device="cuda").manual_seed(S))
    cache, ws = m.alloc_cache(), m.alloc_workspace(S)
    new = idx_dev(np.tile(np.arange(4, dtype=np.int32), (B, 1)))
    refresh = torch.zeros(B * S, dtype=torch.int32, device="cuda")
    m.set_tuning(gemm_kernel=2)
    outs = []
    for stream_k in (0, 1, 1):
        m.set_tuning(stream_k=stream_k)
        outs.append(torch.full((B, S, 256), 5.0, device="cuda"))
        m.full_step(hidden, cache, new, None, 0.1, outs[-1], refresh, ws)
    m.check_status()
    assert outs[0].abs().max() < 8.0 and (outs[0] - hidden).abs().max() > 0.01
    assert (outs[1] - outs[0]).abs().max() <= 1e-5
    assert torch.equal(outs[1], outs[2])                                 # bit-reproducible


def test_validate_indices():
    from paper_2506_12035_b200.binding import MarcheError
    S, B = 68, 2
    cfg, blocks, m = model_for("f32", 128, 2, 128, S, B)
    act = np.array([[1, 2, 3, 4], [5, 6, 7, 8]], np.int32)
    new = act[:, :2]
    excl = np.array([[9], [10]], np.int32)
    m.validate_indices(idx_dev(act), idx_dev(new), idx_dev(excl))
    for bad_act, bad_new, bad_excl in [
        (np.array([[1, 2, 3, 3], [5, 6, 7, 8]], np.int32), new, excl),            # duplicate
        (np.array([[1, 2, 3, 68], [5, 6, 7, 8]], np.int32), new, excl),           # out of range
        (act, np.array([[1, 9], [5, 6]], np.int32), None),                         # new not in active
        (act, new, np.array([[2], [10]], np.int32)),                               # exclude overlaps new
    ]:
        with pytest.raises(MarcheError) as e:
            m.validate_indices(idx_dev(bad_act), idx_dev(bad_new), None if bad_excl is None else idx_dev(bad_excl))
        assert e.value.code == -5


@pytest.mark.parametrize("dtype", ["bf16", "bf16b"])
@pytest.mark.parametrize("M,N,K", [(1, 128, 4096), (9, 640, 2560), (7, 256, 320), (127, 512, 448), (129, 512, 448),
                                   (40, 3072, 1024), (128, 1024, 1024), (257, 384, 128), (640, 4096, 1024),
                                   (8, 4096, 1024), (161, 384, 192), (390, 1024, 4096), (521, 1280, 5120)])
def test_linear_few_rows_split_k(dtype, M, N, K):
    """Row counts at the edges of the A tile, every tile width and cluster size of the split-K kernel, K ranges that do
    not divide evenly (5, 7, 40 blocks over 4, 4, 8 CTAs).  Products of unit size: |acc + bias| stays below 8, where
    half a bf16 step is 0.016 (limit 0.02 with the fp32 sum), and an fp32 sum of K terms errs by sqrt(K) 2^-24.
    (Asked for by name: up to 32 rows run on another kernel by themselves.)"""
    from paper_2506_12035_b200 import binding
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    m.set_tuning(gemm_kernel=binding.GEMM_SINGLE)
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((M, K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) / math.sqrt(K)).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    acc = orc.linear(quant_a(a, dtype), quant_a(w, dtype), bias.astype(np.float64))
    assert np.abs(acc).max() < 8.0
    a_d, w_d, b_d = dev(a, adt(dtype)), dev(w, adt(dtype)), dev(bias)
    out = torch.full((M + 3, N), 5.0, dtype=tdt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 0, out, M=M)
    assert max_abs(host(out[:M]), acc) <= 2e-2 and (host(out[M:]) == 5.0).all()
    res = rng.standard_normal((M, N)).astype(np.float32)
    first = None
    for _ in range(2):                                                   # bit-reproducible
        out = dev(res)
        m.linear(a_d, w_d, b_d, 1, out)
        assert max_abs(host(out), acc + res) <= 2e-5
        assert first is None or torch.equal(out, first)
        first = out
    out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 2, out)
    assert max_abs(host(out), orc.gelu(acc)) <= 2e-2
    assert m.device_status() == 0


@pytest.mark.parametrize("M,N,K", [(4800, 1024, 256), (9000, 768, 128), (5248, 3072, 192), (19100, 256, 128)])
def test_linear_many_tiles_all_epilogues(M, N, K):
    """Shapes with more output tiles than CTA pairs and a partial last round, where the pair GEMM
    cuts the left-over tiles into column slices (and, for the residual epilogue with long K, uses
    stream-K): every element against the oracle's product."""
    dtype = "bf16"
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((M, K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    aq, wq = quant_a(a, dtype), quant_a(w, dtype)
    acc = orc.linear(aq, wq, bias.astype(np.float64))
    a_d, w_d, b_d = dev(a, adt(dtype)), dev(w, adt(dtype)), dev(bias)
    out = torch.zeros(M + 3, N, dtype=tdt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 0, out, M=M)
    assert max_abs(host(out[:M]), acc) <= 3e-2 and rel_l2(host(out[:M]), acc) <= 4e-3
    assert (host(out[M:]) == 0).all()                                    # rows beyond M untouched
    res = rng.standard_normal((M, N)).astype(np.float32)
    out = dev(res)
    m.linear(a_d, w_d, b_d, 1, out)
    assert max_abs(host(out), acc + res) <= 1e-4 * max(1.0, math.sqrt(K / 256))
    out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 2, out)
    want = orc.gelu(acc)
    assert max_abs(host(out), want) <= 3e-2 and rel_l2(host(out), want) <= 4e-3
    assert m.device_status() == 0


@pytest.mark.parametrize("D,F", [(768, 3072), (1024, 4096), (1280, 5120)])
@pytest.mark.parametrize("M", [256, 4352, 5760, 10176])
def test_projection_shapes_of_the_configs(D, F, M):
    """The four projections of a block at the row counts of the benchmark configurations (K = 1280 and
    5120 loop counts included); 384 sampled rows of each output against the oracle's product."""
    dtype = "bf16"
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(D + M)
    rows = np.unique(np.concatenate([[0, M - 1], rng.integers(0, M, 382)]))
    for (N, K, epi) in ((3 * D, D, 0), (D, D, 1), (F, D, 2), (D, F, 1)):
        a = rng.standard_normal((M, K)).astype(np.float32)
        w = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
        bias = (rng.standard_normal(N) * 0.02).astype(np.float32)
        acc = orc.linear(quant_a(a[rows], dtype), quant_a(w, dtype), bias.astype(np.float64))
        a_d, w_d, b_d = dev(a, adt(dtype)), dev(w, adt(dtype)), dev(bias)
        if epi == 0:
            out = torch.zeros(M, N, dtype=tdt(dtype), device="cuda")
            want = acc
        elif epi == 1:
            res = rng.standard_normal((M, N)).astype(np.float32)
            out = dev(res)
            want = acc + res[rows]
        else:
            out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
            want = orc.gelu(acc)
        m.linear(a_d, w_d, b_d, epi, out)
        got = host(out)[rows]
        lim = 1e-4 * max(1.0, math.sqrt(K / 256)) if epi == 1 else 3e-2
        assert max_abs(got, want) <= lim, (N, K, epi, max_abs(got, want))
        if epi != 1:
            assert rel_l2(got, want) <= 4e-3
    assert m.device_status() == 0


@pytest.mark.parametrize("S", [320, 1088])
@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("n,nG", [(159, 25), (320, 320), (97, 1)])
def test_attention_many_rows(S, dh, H, n, nG):
    """Active sets beyond one query tile, every query scoring in one case.  With scores: the two-pass tcgen05 kernel
    (head_dim 64) and mma.sync with seven consumer warps (80); without: the single-pass tcgen05 kernel for both."""
    dtype = "bf16"
    B, D = 2, dh * H
    cfg, blocks, m = model_for(dtype, D, H, 128, S, B)
    rng = np.random.default_rng(S + n + dh)
    q = (rng.standard_normal((B * n, 3 * D)) * 3.0).astype(np.float32)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    flags = np.zeros((B, n), dtype=np.uint8)
    for b in range(B):
        flags[b, rng.permutation(n)[:nG]] = 1
    o = torch.zeros(B * n, D, dtype=adt(dtype), device="cuda")
    partial = torch.full((B, H, S), -1.0, device="cuda")
    m.attention(dev(q, tdt(dtype)), 3 * D, n, dev(cache, tdt(dtype)), dev(flags), partial, o)
    qq, cc = quant(q, dtype), quant(cache, dtype)
    want_o = np.zeros((B * n, D))
    want_p = np.zeros((B, H, S))
    for b in range(B):
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            z, p = orc.softmax_attention(qq[b * n:(b + 1) * n, c], cc[0, b][:, c], cc[1, b][:, c])
            want_o[b * n:(b + 1) * n, c] = z
            want_p[b, h] = p[flags[b].astype(bool)].sum(axis=0)
    got_o, got_p = host(o), host(partial)
    assert rel_l2(got_o, want_o) <= 8e-3 and max_abs(got_o, want_o) <= 3e-2
    assert max_abs(got_p, want_p) <= 2e-2 * max(1, nG) / 8 + 1e-6
    assert np.allclose(got_p.sum(-1), nG, rtol=5e-3, atol=1e-6)
    o2 = torch.zeros_like(o)
    m.attention(dev(q, tdt(dtype)), 3 * D, n, dev(cache, tdt(dtype)), None, None, o2)       # plain flavour
    assert rel_l2(host(o2), want_o) <= 8e-3 and max_abs(host(o2), want_o) <= 3e-2
    assert m.device_status() == 0


@pytest.mark.parametrize("operand", ["bf16", "bf16b"])
@pytest.mark.parametrize("dh", [64, 80])
@pytest.mark.parametrize("B,H,S,n", [(2, 4, 68, 1), (3, 4, 257, 7), (2, 8, 320, 16), (2, 8, 320, 17), (5, 4, 64, 32),
                                     (80, 16, 200, 5), (140, 8, 130, 20)])
def test_attention_small_sets_persistent(operand, dh, B, H, S, n):
    """The persistent mma.sync launch, which the plain attention takes at up to 32 query rows where the keys are not split (it
    is asked for here, since few items would be): one and two consumer warps, both head sizes, ragged key tiles, fewer
    items than resident CTAs and several items per CTA (1280 and 1120 items), where a CTA's loads run ahead into its next
    item."""
    from paper_2506_12035_b200 import binding
    if dh == 80:
        H = (H + 7) // 8 * 8                                # the model width must be a multiple of 128
    D = H * dh
    if operand == "bf16b" and B > 5:
        pytest.skip("one operand type is enough for the large shapes")
    cfg, blocks, m = model_for(operand, D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_MMA)
    rng = np.random.default_rng(7 * B + H + S + n + dh)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    q = (rng.standard_normal((B * n, D)) * 2.0).astype(np.float32)
    o = torch.zeros(B * n, D, dtype=adt(operand), device="cuda")
    m.attention(dev(q, torch.bfloat16), D, n, dev(cache, torch.bfloat16), None, None, o)
    torch.cuda.synchronize()
    assert m.device_status() == 0
    got = host(o).reshape(B, n, D)
    assert np.isfinite(got).all()
    qq, cc = quant(q, "bf16").reshape(B, n, D), quant(cache, "bf16")
    for b in sorted(set([0, 1, B // 2, B - 2, B - 1])):
        want = np.zeros((n, D))
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            want[:, c], _ = orc.softmax_attention(qq[b][:, c], cc[0, b][:, c], cc[1, b][:, c])
        assert rel_l2(got[b], want) <= 8e-3 and max_abs(got[b], want) <= 3e-2, \
            "b=%d: max-abs %.3g rel-L2 %.3g" % (b, max_abs(got[b], want), rel_l2(got[b], want))


@pytest.mark.parametrize("dh", [64, 80])
@pytest.mark.parametrize("S,n", [(33, 30), (64, 32), (100, 30), (164, 17), (192, 30), (192, 16)])
def test_attention_persistent_rows_of_every_item(dh, S, n):
    """2048 items, several per CTA, whose one to three key tiles fit the ring, so that an item's query rows are on their way
    while the one before is computed: every row of every item, and the same bits in every launch.  Weights are bf16 (2^-9
    each, of both signs over S keys, values below 6) and the output fp16: 3e-2 as in the other attention tests."""
    from paper_2506_12035_b200 import binding
    B, H = 128, 16
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_MMA)
    gen = torch.Generator(device="cuda").manual_seed(S + n + dh)
    q = (torch.randn(B * n, D, generator=gen, device="cuda") * 2.0).to(torch.bfloat16)
    cache = torch.randn(2, B, S, D, generator=gen, device="cuda").to(torch.bfloat16)
    heads = lambda t: t.view(B, -1, H, dh).transpose(1, 2).double()
    want = torch.softmax(heads(q) @ heads(cache[0]).transpose(2, 3) / math.sqrt(dh), -1) @ heads(cache[1])
    first = None
    for _ in range(20):
        o = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
        m.attention(q, D, n, cache, None, None, o)
        assert first is None or torch.equal(o, first)
        first = o
    assert (heads(first) - want).abs().max() <= 3e-2 and m.device_status() == 0


@pytest.mark.parametrize("operand", ["bf16", "bf16b"])
@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n,nG", [(2, 68, 33, 33), (3, 257, 41, 5), (30, 320, 48, 9), (2, 320, 49, 0), (2, 1088, 64, 20), (2, 130, 97, 97),
                                      (2, 320, 120, 3)])
def test_attention_mma_sync_one_cta_per_item(operand, dh, H, B, S, n, nG):
    """The mma.sync kernel with one CTA per item, asked for by name: three to seven consumer warps and a second query tile, ragged
    keys, plain and with scores.  Bounds as in the tests above."""
    from paper_2506_12035_b200 import binding
    D = H * dh
    cfg, blocks, m = model_for(operand, D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_MMA)
    rng = np.random.default_rng(B + S + n + dh)
    cache, q = rng.standard_normal((2, B, S, D)).astype(np.float32), (rng.standard_normal((B * n, D)) * 3.0).astype(np.float32)
    flags = np.zeros((B, n), dtype=np.uint8)
    for b in range(B):
        flags[b, rng.permutation(n)[:nG]] = 1
    partial = torch.full((B, H, S), -1.0, device="cuda")
    outs = []
    for f in (flags, None):
        outs.append(torch.zeros(B * n, D, dtype=adt(operand), device="cuda"))
        m.attention(dev(q, torch.bfloat16), D, n, dev(cache, torch.bfloat16), None if f is None else dev(f), partial, outs[-1])
    assert m.device_status() == 0
    qq, cc, got_p = quant(q, "bf16").reshape(B, n, D), quant(cache, "bf16"), host(partial)
    for b in sorted({0, B // 2, B - 1}):
        want = np.zeros((n, D))
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            want[:, c], p = orc.softmax_attention(qq[b][:, c], cc[0, b][:, c], cc[1, b][:, c])
            assert max_abs(got_p[b, h], p[flags[b].astype(bool)].sum(axis=0)) <= 2e-2 * max(1, nG) / 8 + 1e-6
        for o in outs:
            got = host(o).reshape(B, n, D)[b]
            assert rel_l2(got, want) <= 8e-3 and max_abs(got, want) <= 3e-2


@pytest.mark.parametrize("operand", ["bf16", "bf16b"])
@pytest.mark.parametrize("B,H,S,n", [(2, 4, 68, 5), (2, 4, 128, 128), (3, 4, 320, 41), (40, 4, 320, 41), (2, 4, 320, 129),
                                     (2, 4, 320, 320), (100, 4, 320, 77), (2, 16, 1088, 122), (2, 16, 1088, 159),
                                     (1, 4, 1088, 1088), (2, 4, 2048, 300), (37, 8, 300, 257)])
def test_attention_single_pass_tcgen05(operand, B, H, S, n):
    """The single-pass tcgen05 kernel (weights kept in tensor memory, persistent over (sample, head) items) on
    its own: one, two and more query tiles, one key tile up to sixteen with ragged tails, more items than SMs,
    and logits whose row maximum keeps growing from tile to tile (the lazy rescaling of the accumulator)."""
    from paper_2506_12035_b200 import binding
    dh = 64
    D = H * dh
    if operand == "bf16b" and B * H * n * S > 3e6:
        pytest.skip("one operand type is enough for the large shapes")
    cfg, blocks, m = model_for(operand, D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_TCGEN05)
    rng = np.random.default_rng(B + H + S + n)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    # (i) ordinary logits; (ii) logits that grow with the key index: every tile raises the row maximum by
    # far more than 2^8, so each tile rescales the accumulator; (iii) one-hot rows on a late key
    q_rand = (rng.standard_normal((B * n, D)) * 3.0).astype(np.float32)
    ramp = np.linspace(0.0, 40.0, S, dtype=np.float32)
    cache_ramp = cache.copy()
    cache_ramp[0, :, :, 0::dh] = ramp[None, :, None]                   # first channel of every head's keys
    q_ramp = q_rand.copy()
    q_ramp[:, 0::dh] = 16.0                                            # logit contribution 16 * ramp / 8 = 0 .. 80
    kq = quant(cache, "bf16")
    tsel = rng.integers(max(0, S - 40), S, size=(B, n))
    q_hot = np.stack([kq[0, b, tsel[b]] for b in range(B)]).reshape(B * n, D).astype(np.float32) * 64.0
    sample_b = sorted(set([0, B // 2, B - 1]))
    for name, q, cch in (("random", q_rand, cache), ("ramp", q_ramp, cache_ramp), ("one-hot", q_hot, cache)):
        o = torch.zeros(B * n, D, dtype=adt(operand), device="cuda")
        m.attention(dev(q, torch.bfloat16), D, n, dev(cch, torch.bfloat16), None, None, o)
        torch.cuda.synchronize()
        assert m.device_status() == 0
        got = host(o).reshape(B, n, D)
        assert np.isfinite(got).all(), name
        qq, cc = quant(q, "bf16").reshape(B, n, D), quant(cch, "bf16")
        for b in sample_b:
            want = np.zeros((n, D))
            for h in range(H):
                c = slice(h * dh, (h + 1) * dh)
                want[:, c], _ = orc.softmax_attention(qq[b][:, c], cc[0, b][:, c], cc[1, b][:, c])
            assert rel_l2(got[b], want) <= 8e-3 and max_abs(got[b], want) <= 3e-2, \
                "%s b=%d: max-abs %.3g rel-L2 %.3g" % (name, b, max_abs(got[b], want), rel_l2(got[b], want))


@pytest.mark.parametrize("M,N,K", [(31, 64, 16), (33, 128, 144), (136, 1024, 256), (136, 256, 1024), (700, 192, 400),
                                   (1776, 1024, 256), (2100, 640, 272)])
def test_linear_f32_tiles_and_k_slices(M, N, K):
    """The fp32 projection kernel: both tile sizes, one to four K slices, ragged rows, K chunks of fewer than 128 and a
    wider row stride from an unaligned start.  Products of unit size: an fp32 sum of K terms errs by about sqrt(K) 2^-24 < 2e-6."""
    cfg, blocks, m = model_for("f32", 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(M + N + K)
    for lda, skip in ((K, 0), (K + 4, 1)):
        a = rng.standard_normal((M, lda)).astype(np.float32)
        w = (rng.standard_normal((N, K)) / math.sqrt(K)).astype(np.float32)
        bias, res = rng.standard_normal(N).astype(np.float32), rng.standard_normal((M, N)).astype(np.float32)
        acc = orc.linear(a[:, :K].astype(np.float64), w.astype(np.float64), bias.astype(np.float64))
        a_d = torch.empty(M * lda + skip, device="cuda")[skip:].copy_(dev(a).view(-1))
        w_d, b_d = dev(w), dev(bias)
        for epi, start, want in ((0, np.full((M, N), 5.0, np.float32), acc), (1, res, acc + res), (2, res, orc.gelu(acc))):
            out = torch.full((M + 3, N), 5.0, device="cuda")
            out[:M] = dev(start)
            m.linear(a_d, w_d, b_d, epi, out, M=M, lda=lda)
            assert max_abs(host(out[:M]), want) <= 1e-5 and (host(out[M:]) == 5.0).all()


@pytest.mark.parametrize("B,H,S,dh,n,nG", [(1, 2, 1, 64, 1, 1), (2, 4, 64, 64, 16, 3), (2, 4, 65, 32, 17, 17), (12, 4, 148, 64, 148, 5),
                                           (1, 2, 2048, 128, 40, 11), (1, 8, 320, 16, 130, 0), (80, 8, 68, 16, 33, 9)])
def test_attention_f32_query_clusters(B, H, S, dh, n, nG):
    """The fp32 attention: one to eight CTAs per item, one to many 16-query tiles, ragged keys, both ring depths, scores
    added over the cluster.  Weights sum to one, so an output errs by a few 2^-24 times the largest value (5)."""
    cfg, blocks, m = model_for("f32", H * dh, H, 128, S, B)
    rng = np.random.default_rng(B + S + n)
    q = (rng.standard_normal((B * n, H * dh)) * 2.0).astype(np.float32)
    cache = rng.standard_normal((2, B, S, H * dh)).astype(np.float32)
    flags = np.zeros((B, n), dtype=np.uint8)
    flags[:, rng.permutation(n)[:nG]] = 1
    o, partial = torch.zeros(B * n, H * dh, device="cuda"), torch.full((B, H, S), -1.0, device="cuda")
    m.attention(dev(q), H * dh, n, dev(cache), dev(flags), partial, o)
    got_o, got_p = host(o).reshape(B, n, H * dh), host(partial)
    for b in sorted({0, B // 2, B - 1}):
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            z, p = orc.softmax_attention(q[b * n:(b + 1) * n, c].astype(np.float64), cache[0, b][:, c].astype(np.float64),
                                         cache[1, b][:, c].astype(np.float64))
            assert max_abs(got_o[b][:, c], z) <= 2e-5
            assert max_abs(got_p[b, h], p[flags[b].astype(bool)].sum(axis=0)) <= 1e-5


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n", [(1, 1, 1), (2, 64, 16), (1, 65, 17), (2, 320, 41), (2, 320, 64), (1, 1088, 48), (1, 2048, 33),
                                   (3, 577, 5)])
def test_attention_keys_split_over_a_cluster(dh, H, B, S, n):
    """One to eight CTAs per item (one without a cluster), one to four key tiles per CTA and one to four query warps,
    logits that grow along the keys (the ranks' maxima far apart) and one-hot rows; bit-reproducible.  So few items always
    take this kernel."""
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    rng = np.random.default_rng(B + S + n + dh)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    cache_ramp = cache.copy()
    cache_ramp[0, :, :, 0::dh] = np.linspace(0.0, 40.0, S, dtype=np.float32)[None, :, None]
    q = (rng.standard_normal((B * n, D)) * 3.0).astype(np.float32)
    q_ramp = q.copy()
    q_ramp[:, 0::dh] = 16.0
    q_hot = np.stack([quant(cache, "bf16")[0, b, rng.integers(0, S, size=n)] for b in range(B)]).reshape(B * n, D).astype(np.float32) * 64.0
    for qq, cc in ((q, cache), (q_ramp, cache_ramp), (q_hot, cache)):
        outs = []
        for _ in range(2):
            o = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
            m.attention(dev(qq, torch.bfloat16), D, n, dev(cc, torch.bfloat16), None, None, o)
            outs.append(o)
        assert torch.equal(outs[0], outs[1]) and m.device_status() == 0
        qq, cc = quant(qq, "bf16"), quant(cc, "bf16")
        want = np.zeros((B * n, D))
        for b in range(B):
            for h in range(H):
                c = slice(h * dh, (h + 1) * dh)
                want[b * n:(b + 1) * n, c], _ = orc.softmax_attention(qq[b * n:(b + 1) * n, c], cc[0, b][:, c], cc[1, b][:, c])
        assert rel_l2(host(outs[0]), want) <= 8e-3 and max_abs(host(outs[0]), want) <= 3e-2


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n,nG", [(1, 1, 1, 1), (2, 64, 16, 16), (2, 65, 17, 17), (3, 320, 32, 5), (2, 1088, 32, 31), (1, 1200, 20, 0)])
def test_attention_scores_of_the_generating_rows(dh, H, B, S, n, nG):
    """The kernel that scores the flagged rows alone: none, one group of 16 (four warps share the tiles) and two, one to
    nineteen key tiles; weights in fp32 from bf16 logits, so a score errs by the logits' rounding as in the attention."""
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    rng = np.random.default_rng(B + S + n + dh)
    q, cache = (rng.standard_normal((B * n, D)) * 3.0).astype(np.float32), rng.standard_normal((2, B, S, D)).astype(np.float32)
    flags = np.zeros((B, n), dtype=np.uint8)
    for b in range(B):
        flags[b, rng.permutation(n)[:nG]] = 1
    got = []
    for _ in range(2):
        o, partial = torch.zeros(B * n, D, dtype=torch.float16, device="cuda"), torch.full((B, H, S), -1.0, device="cuda")
        m.attention(dev(q, torch.bfloat16), D, n, dev(cache, torch.bfloat16), dev(flags), partial, o)
        got.append(partial)
    assert torch.equal(got[0], got[1]) and m.device_status() == 0
    qq, cc = quant(q, "bf16"), quant(cache, "bf16")
    want = np.zeros((B, H, S))
    for b in range(B):
        for h in range(H):
            c = slice(h * dh, (h + 1) * dh)
            _, p = orc.softmax_attention(qq[b * n:(b + 1) * n, c], cc[0, b][:, c], cc[1, b][:, c])
            want[b, h] = p[flags[b].astype(bool)].sum(axis=0)
    assert max_abs(host(got[0]), want) <= 2e-4 * max(1, nG) and np.allclose(host(got[0]).sum(-1), nG, rtol=1e-4, atol=1e-6)


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n", [(1, 1, 1), (2, 65, 33), (3, 320, 70), (2, 128, 128), (60, 130, 129), (2, 1088, 150), (25, 577, 300)])
def test_attention_single_pass_streams(dh, H, B, S, n):
    """The single-pass tcgen05 kernel at both head sizes: query tiles on one to four lane quarters (alone and behind full
    ones), fewer and more units than run at once, ragged keys, row maxima that keep growing."""
    from paper_2506_12035_b200 import binding
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_TCGEN05)
    rng = np.random.default_rng(B + S + n + dh)
    cache = rng.standard_normal((2, B, S, D)).astype(np.float32)
    q = (rng.standard_normal((B * n, D)) * 3.0).astype(np.float32)
    ramp, q_ramp = cache.copy(), q.copy()
    ramp[0, :, :, dh - 1::dh] = np.linspace(0.0, 40.0, S, dtype=np.float32)[None, :, None]
    q_ramp[:, dh - 1::dh] = 16.0
    for qq, cc in ((q, cache), (q_ramp, ramp)):
        o = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
        m.attention(dev(qq, torch.bfloat16), D, n, dev(cc, torch.bfloat16), None, None, o)
        assert m.device_status() == 0
        got, qq, cc = host(o).reshape(B, n, D), quant(qq, "bf16").reshape(B, n, D), quant(cc, "bf16")
        for b in sorted({0, B // 2, B - 1}):
            want = np.zeros((n, D))
            for h in range(H):
                c = slice(h * dh, (h + 1) * dh)
                want[:, c], _ = orc.softmax_attention(qq[b][:, c], cc[0, b][:, c], cc[1, b][:, c])
            assert rel_l2(got[b], want) <= 8e-3 and max_abs(got[b], want) <= 3e-2


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n", [(40, 64, 20), (40, 65, 33), (38, 320, 70), (75, 130, 97), (40, 577, 128), (38, 200, 150)])
def test_attention_single_pass_streams_of_many_units(dh, H, B, S, n):
    """More units than SMs (152 to 600): the streams of a CTA work side by side, with query tiles on one to four lane quarters.
    (With fewer units head_dim 64 runs CTAs of one stream.)  Bounds as in the test above."""
    from paper_2506_12035_b200 import binding
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_TCGEN05)
    gen = torch.Generator(device="cuda").manual_seed(B + S + n + dh)
    cache = torch.randn(2, B, S, D, generator=gen, device="cuda")
    q = torch.randn(B * n, D, generator=gen, device="cuda") * 3.0
    ramp, q_ramp = cache.clone(), q.clone()
    ramp[0, :, :, dh - 1::dh] = torch.linspace(0.0, 40.0, S, device="cuda")[None, :, None]
    q_ramp[:, dh - 1::dh] = 16.0
    heads = lambda t: t.view(B, -1, H, dh).transpose(1, 2).double()
    for qq, cc in ((q.to(torch.bfloat16), cache.to(torch.bfloat16)), (q_ramp.to(torch.bfloat16), ramp.to(torch.bfloat16))):
        o = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
        m.attention(qq, D, n, cc, None, None, o)
        assert m.device_status() == 0
        want = torch.softmax(heads(qq) @ heads(cc[0]).transpose(2, 3) / math.sqrt(dh), -1) @ heads(cc[1])
        assert (heads(o) - want).norm() <= 8e-3 * want.norm() and (heads(o) - want).abs().max() <= 3e-2


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n,nG", [(2, 129, 16, 1), (3, 192, 7, 7), (2, 320, 48, 16), (2, 1088, 151, 21), (3, 577, 130, 32), (2, 320, 320, 2),
                                      (1, 2048, 40, 3), (40, 200, 300, 17)])
def test_scores_of_a_few_among_many_rows(dh, H, B, S, n, nG):
    """The scoring block of a one-block step, whose generating rows (one or two groups of 16) lie anywhere among the active
    ones, in the kernel that scores them alone where the rule takes it, and in the attention itself: against the oracle on the
    step's own q and keys.  Per head as in the test above; the scores are sums over the heads."""
    from paper_2506_12035_b200 import binding
    D = H * dh
    if n > S:
        n = S
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    rng = np.random.default_rng(B + S + n + dh)
    hidden = dev(rng.standard_normal((B, S, D)).astype(np.float32))
    act = np.stack([rng.permutation(S)[:n] for _ in range(B)]).astype(np.int32)
    new = np.stack([a[rng.permutation(n)[:nG]] for a in act]).astype(np.int32)
    cache, ws, out = m.alloc_cache(), m.alloc_workspace(S), torch.zeros(B, S, D, device="cuda")
    scores = torch.zeros(B, S, device="cuda")
    m.init_cache(cache)
    m.full_step(hidden, cache, idx_dev(new), None, 0.0, out, None, ws)
    # q of the active rows, by the calls the step makes
    u = torch.zeros(B * n, D, dtype=torch.float16, device="cuda")
    qkv = torch.zeros(B * n, 3 * D, dtype=torch.bfloat16, device="cuda")
    w = m.weights[0]
    m.gather_layernorm(hidden, idx_dev(act), n, w["ln1_g"], w["ln1_b"], None, u)
    m.linear(u, w["w_qkv"], w["b_qkv"], 0, qkv)
    for kernel in (binding.ATTENTION_AUTO, binding.ATTENTION_TCGEN05_TWO_PASS):
        m.set_tuning(attention_kernel=kernel)
        m.step(hidden, cache, idx_dev(act), idx_dev(new), None, 0.0, out, None, ws)
        m.get_scores(ws, scores)
        got, q, k = host(scores), host(qkv).reshape(B, n, 3 * D), host(cache[0, 0])
        for b in sorted({0, B // 2, B - 1}):
            rows = np.isin(act[b], new[b])
            want = np.zeros(S)
            for h in range(H):
                c = slice(h * dh, (h + 1) * dh)
                _, p = orc.softmax_attention(q[b][rows][:, c], k[b][:, c], k[b][:, c])
                want += p.sum(axis=0)
            assert max_abs(got[b], want) <= 2e-4 * H * nG and abs(got[b].sum() - H * nG) <= 1e-4 * H * nG
    assert m.device_status() == 0


@pytest.mark.parametrize("dh,H", [(64, 4), (80, 8)])
@pytest.mark.parametrize("B,S,n", [(111, 128, 128), (112, 100, 65), (148, 130, 128), (149, 33, 33), (75, 257, 257), (50, 300, 300), (23, 577, 577),
                                   (16, 1100, 1100)])
def test_attention_single_pass_streams_deal_units(dh, H, B, S, n):
    """Around one unit per stream (444 units of three streams, 592 of four) and over several turns, with 1 to 9 query tiles per
    item: every unit is taken once, whole and by one stream.  Bounds as in the two tests of these streams above."""
    from paper_2506_12035_b200 import binding
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    m.set_tuning(attention_kernel=binding.ATTENTION_TCGEN05)
    gen = torch.Generator(device="cuda").manual_seed(B + S + n + dh)
    cache = torch.randn(2, B, S, D, generator=gen, device="cuda").to(torch.bfloat16)
    q = (torch.randn(B * n, D, generator=gen, device="cuda") * 3.0).to(torch.bfloat16)
    o = torch.full((B * n + 1, D), 7.0, dtype=torch.float16, device="cuda")
    m.attention(q, D, n, cache, None, None, o[:-1])
    assert m.device_status() == 0 and (o[-1] == 7.0).all()
    heads = lambda t: t.view(B, -1, H, dh).transpose(1, 2).float()
    want = torch.softmax(heads(q) @ heads(cache[0]).transpose(2, 3) / math.sqrt(dh), -1) @ heads(cache[1])
    assert (heads(o[:-1]) - want).norm() <= 8e-3 * want.norm() and (heads(o[:-1]) - want).abs().max() <= 3e-2


@pytest.mark.parametrize("dtype", ["bf16", "bf16b"])
@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (3, 384, 128), (7, 2304, 768), (15, 128, 2048), (16, 640, 2112), (16, 1024, 4096), (17, 768, 768),
                                   (31, 384, 1088), (32, 768, 3072)])
def test_linear_of_a_handful_of_rows(dtype, M, N, K):
    """Up to 32 rows, whole K per CTA and K split over pairs of CTAs, K blocks that do not divide evenly among warps and CTAs:
    against the oracle's product, rows beyond M untouched, and the same bits every time.  (fp32 sums of K products of unit
    scale, then one rounding of the output; residual outputs stay fp32.)"""
    cfg, blocks, m = model_for(dtype, 256, 4, 1024, 68, 2)
    rng = np.random.default_rng(M + N + K)
    a = rng.standard_normal((M, K)).astype(np.float32)
    w = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    bias = rng.standard_normal(N).astype(np.float32)
    acc = orc.linear(quant_a(a, dtype), quant_a(w, dtype), bias.astype(np.float64))
    a_d, w_d, b_d = dev(a, adt(dtype)), dev(w, adt(dtype)), dev(bias)
    scale = math.sqrt(K / 256)
    out = torch.full((M + 2, N), 5.0, dtype=tdt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 0, out, M=M)
    assert max_abs(host(out[:M]), acc) <= 3e-2 * max(1.0, scale) and rel_l2(host(out[:M]), acc) <= 4e-3
    assert (host(out[M:]) == 5.0).all()
    res = rng.standard_normal((M, N)).astype(np.float32)
    first = None
    for _ in range(3):
        out = dev(res)
        m.linear(a_d, w_d, b_d, 1, out)
        assert max_abs(host(out), acc + res) <= 2e-5 * max(1.0, scale)
        assert first is None or torch.equal(out, first)
        first = out
    out = torch.zeros(M, N, dtype=adt(dtype), device="cuda")
    m.linear(a_d, w_d, b_d, 2, out)
    want = orc.gelu(acc)
    assert max_abs(host(out), want) <= 3e-2 * max(1.0, scale) and rel_l2(host(out), want) <= 4e-3
    assert m.device_status() == 0


@pytest.mark.parametrize("operand", ["f16", "bf16"])
@pytest.mark.parametrize("D,H,F,B,n", [(256, 4, 1024, 1, 1), (768, 12, 3072, 2, 8), (768, 12, 3072, 3, 9), (1024, 16, 4096, 1, 15), (1280, 16, 2560, 2, 7),
                                       (2048, 32, 2048, 1, 16)])
def test_few_rows_normalise_in_the_projection(operand, D, H, F, B, n):
    """A step on up to 32 rows whose projections normalise their rows (a mean of ten deviations; gamma 0.5 to 2, beta of unit size):
    what the blocks add to the active rows, and the active tokens' K and V behind a normalising projection, against the oracle,
    against the same step with LayerNorm launches (which a measurement hook asks for), and with the K/V write-back in a launch of
    its own.  Operands are rounded by 2^-11 or 2^-8 of a value, q, k, v by 2^-8: the limits leave a factor of three for what three
    blocks add up.  The oracle without one of the four parameter arrays is more than five limits away."""
    import synth
    from helpers import make_model
    cfg = synth.CONFIGS["mar_b"].replace(L=3, E=0, D=D, H=H, F=F, B=B, S=40, n_buffer=8)
    rng = np.random.default_rng(D + n)
    blocks = synth.make_weights(cfg)
    for blk in blocks:
        for g, b in (("ln1_g", "ln1_b"), ("ln2_g", "ln2_b")):
            blk[g], blk[b] = rng.uniform(0.5, 2.0, D).astype(np.float32), rng.standard_normal(D).astype(np.float32)
    m = make_model(cfg, blocks, operand=operand)
    hidden = (rng.standard_normal((B, cfg.S, D)) + 10.0 * rng.standard_normal((B, cfg.S, 1))).astype(np.float32)
    act = np.stack([rng.permutation(cfg.S)[:n] for _ in range(B)]).astype(np.int32)

    def of_active_rows(out, K, V):                                       # [L][B][S][D] K and V; block 0 has its LayerNorm launch
        return (np.stack([out[b, act[b]] - hidden[b, act[b]] for b in range(B)]),
                np.stack([np.stack([K[1:, b][:, act[b]], V[1:, b][:, act[b]]]) for b in range(B)]))

    def oracle(step_blocks):
        oc, out = orc.KVCache(cfg.L, B, cfg.S, D), np.zeros((B, cfg.S, D))
        kw = dict(n_heads=H, score_layer=cfg.score_layer, ln_eps=cfg.ln_eps)
        orc.full_step(blocks, hidden, oc, act, None, 0.0, out, **kw)
        orc.marche_step(step_blocks, hidden, oc, act, act, None, 0.0, out, **kw)
        return of_active_rows(out, oc.K, oc.V)

    want, limit = oracle(blocks), 1e-2 if operand == "f16" else 2e-2
    for name, neutral, part in (("ln1_g", 1.0, 1), ("ln1_b", 0.0, 1), ("ln2_g", 1.0, 0), ("ln2_b", 0.0, 0)):
        left_out = oracle([blk if l == 0 and part else {**blk, name: np.full(D, neutral)} for l, blk in enumerate(blocks)])
        assert rel_l2(left_out[part], want[part]) > 5 * limit
    got = []
    for hook, fuse in (((), 1), (("gather_layernorm",), 1), ((), 0)):
        m.debug_repeat_classes(hook)
        m.set_tuning(fuse_qkv_scatter=fuse)
        cache, out, ws = m.alloc_cache(), torch.zeros(B, cfg.S, D, device="cuda"), m.alloc_workspace(cfg.S)
        m.init_cache(cache)
        m.full_step(dev(hidden), cache, idx_dev(act), None, 0.0, out, None, ws)
        before = m.launch_count()
        m.step(dev(hidden), cache, idx_dev(act), idx_dev(act), None, 0.0, out, None, ws)
        got.append((*of_active_rows(host(out), host(cache[:, 0]), host(cache[:, 1])), m.launch_count() - before))
        assert all(rel_l2(g, w) <= limit for g, w in zip(got[-1], want)), [rel_l2(g, w) for g, w in zip(got[-1], want)]
    m.debug_repeat_classes(())
    assert got[1][2] - got[0][2] == 2 * cfg.L + 2 * cfg.L - 1              # all but the first are gone, and the hook doubles them
    assert got[2][2] - got[0][2] == cfg.L                                  # the write-back's launches
    assert np.array_equal(got[2][0], got[0][0]) and np.array_equal(got[2][1], got[0][1])
    assert m.device_status() == 0


@pytest.mark.parametrize("dh", [64, 80])
@pytest.mark.parametrize("S", [193, 256, 257, 320])
@pytest.mark.parametrize("n,ld_pad", [(17, 0), (32, 8), (33, 0), (48, 0), (43, 2)])
def test_attention_a_group_of_warps_per_tile(dh, S, n, ld_pad):
    """32 items, two or three groups of query rows over four or five key tiles: one CTA per item, a group of warps per tile, queries by TMA
    (with a row stride of 2 elements more, by loads).  Bounds as in the test of the split over a cluster."""
    H, B = 16, 2
    D = H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    gen = torch.Generator(device="cuda").manual_seed(S + n + dh)
    cache = torch.randn(2, B, S, D, generator=gen, device="cuda").to(torch.bfloat16)
    ld = D + ld_pad
    q = (torch.randn(B * n, ld, generator=gen, device="cuda") * 3.0).to(torch.bfloat16)
    o = torch.full((B * n + 1, D), 7.0, dtype=torch.float16, device="cuda")
    m.attention(q, ld, n, cache, None, None, o[:-1])
    assert m.device_status() == 0 and (o[-1] == 7.0).all()
    heads = lambda t: t.reshape(B, -1, H, dh).transpose(1, 2).float()
    want = torch.softmax(heads(q[:, :D]) @ heads(cache[0]).transpose(2, 3) / math.sqrt(dh), -1) @ heads(cache[1])
    assert (heads(o[:-1]) - want).norm() <= 8e-3 * want.norm() and (heads(o[:-1]) - want).abs().max() <= 3e-2
    again = torch.zeros_like(o)
    m.attention(q, ld, n, cache, None, None, again[:-1])
    assert torch.equal(again[:-1], o[:-1])


@pytest.mark.parametrize("value", [1e20, -3e24])
@pytest.mark.parametrize("D,H,F", [(256, 4, 512), (768, 12, 768), (1280, 16, 1280)])
def test_few_rows_whose_squares_overflow(value, D, H, F):
    """Rows with one value whose squared deviation is beyond fp32: the variance is infinite, the normalised row is beta, in the
    projection as in the LayerNorm launch.  The value stands in another warp's columns for every row (first, last, both sides of a
    slice's end).  Bounds on the later blocks' K and V: beta of unit size rounds the same way on both sides, weights of 0.02."""
    import synth
    from helpers import make_model
    cfg = synth.CONFIGS["mar_b"].replace(L=2, E=0, D=D, H=H, F=F, B=2, S=40, n_buffer=8)
    blocks = synth.make_weights(cfg)
    rng = np.random.default_rng(D)
    for blk in blocks:
        blk["ln1_b"], blk["ln2_b"] = (rng.standard_normal(D).astype(np.float32) for _ in range(2))
    m = make_model(cfg, blocks)
    hidden_np = rng.standard_normal((cfg.B, cfg.S, D)).astype(np.float32)
    cols = [0, 31, 32, D // 2 - 1, D // 2, D - 33, D - 32, D - 1]
    act = np.stack([rng.permutation(cfg.S)[:8] for _ in range(cfg.B)])
    for b in range(cfg.B):
        hidden_np[b, act[b], cols] = value
    hidden, act_d = dev(hidden_np), idx_dev(act)
    got = []
    for hook in ((), ("gather_layernorm",)):
        m.debug_repeat_classes(hook)
        cache, out, ws = m.alloc_cache(), torch.zeros(cfg.B, cfg.S, D, device="cuda"), m.alloc_workspace(cfg.S)
        m.init_cache(cache)
        m.full_step(hidden, cache, act_d, None, 0.0, out, None, ws)
        m.step(hidden, cache, act_d, act_d, None, 0.0, out, None, ws)
        kv = host(cache[1])                                              # [2][B][S][D] of the block behind a normalising projection
        got.append(np.stack([kv[:, b, act[b]] for b in range(cfg.B)]))
    m.debug_repeat_classes(())
    assert np.isfinite(got[1]).all() and np.abs(got[1]).max() > 0.1
    assert max_abs(got[0], got[1]) <= 2.0 ** -7 * np.abs(got[1]).max()   # one bf16 step
    assert m.device_status() == 0


@pytest.mark.parametrize("items,S,n", [(1024, 512, 33), (1024, 577, 128), (448, 512, 129), (448, 700, 256), (800, 896, 160), (460, 1088, 260)])
def test_attention_four_streams_over_several_rounds(items, S, n):
    """Four streams per CTA, whose weights share the logits' columns, over two rounds and more, one to three query tiles per item, every
    unit taken once.  Bounds as in the test above."""
    H, dh = 4, 64
    B, D = items // H, H * dh
    cfg, blocks, m = model_for("bf16", D, H, 128, S, B)
    gen = torch.Generator(device="cuda").manual_seed(B + S + n)
    cache = torch.randn(2, B, S, D, generator=gen, device="cuda").to(torch.bfloat16)
    q = (torch.randn(B * n, D, generator=gen, device="cuda") * 3.0).to(torch.bfloat16)
    o = torch.full((B * n + 1, D), 7.0, dtype=torch.float16, device="cuda")
    m.attention(q, D, n, cache, None, None, o[:-1])
    assert m.device_status() == 0 and (o[-1] == 7.0).all()
    heads = lambda t: t.view(-1, t.shape[-2], H, dh).transpose(1, 2).float()
    for b in range(0, B, 16):                                            # (the logits of all samples would be gigabytes)
        q_b, k_b, v_b = q.view(B, n, D)[b:b + 16], cache[0, b:b + 16], cache[1, b:b + 16]
        want = torch.softmax(heads(q_b) @ heads(k_b).transpose(2, 3) / math.sqrt(dh), -1) @ heads(v_b)
        got = heads(o[:-1].view(B, n, D)[b:b + 16])
        assert (got - want).norm() <= 8e-3 * want.norm() and (got - want).abs().max() <= 3e-2
