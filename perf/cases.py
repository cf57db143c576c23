"""Workloads of the framework: what a program that decodes MAR-shaped images has the library do.

A case is one call (or one generation) on one stack shape.  Its fields:

  kind      "step"        marche_build_active + marche_step, the cache-aware decoding step
            "full"        marche_full_step, the initial refresh and the full-recompute baseline
            "in_step"     marche_step_in_step_selection, the paper's own schedule (active budget 64)
            "two_stage"   marche_mar_step, encoder on the known tokens and cache-aware decoder
            "host"        marche_step_host, inputs from pinned host memory and results back to it
            "generation"  Generation.run, every step of a decoding run
            "graph"       the same run recorded once by Generation.capture and replayed
            "select"      marche_select_refresh on relevance scores the caller has
  model     width, depth and heads (SHAPES)      grid, buffer   tokens: grid x grid image tokens + buffer tokens
  batch     batch rows                           operand        type of the projections' operands: f16, bf16, f32
  steps, t  length of the decoding run and the step the call belongs to (cosine schedule)
  ratio     share of the tokens that is refreshed from the cache at every step
"""
from __future__ import annotations

import math

import torch

from paper_2506_12035_b200.binding import Marche, upload_mar_weights, upload_weights
from paper_2506_12035_b200.generation import Generation

# model: blocks, encoder blocks, width, heads, MLP width
SHAPES = {
    "tiny": (4, 2, 256, 4, 1024),
    "mar_b": (24, 12, 768, 12, 3072),
    "mar_l": (32, 16, 1024, 16, 4096),
    "mar_h": (40, 20, 1280, 16, 5120),
}
BUDGET = 64          # active tokens of the in-step schedule


def _case(name, kind, model, grid, buffer, batch, operand, steps, t, ratio):
    return dict(name=name, kind=kind, model=model, grid=grid, buffer=buffer, batch=batch, operand=operand, steps=steps,
                t=t, ratio=ratio)


def listed():
    return [
        # the refresh selection alone, the smallest call of the path
        _case("hires_select", "select", "mar_b", 32, 64, 64, "f16", 64, 40, 0.10),
        # a debugging-size fp32 run, eight short steps: launches and their latency are all there is
        _case("tiny_f32_generation", "generation", "tiny", 8, 4, 2, "f32", 8, 0, 0.10),
        # one image (two rows, classifier-free guidance) without refresh, the whole run as one CUDA graph
        _case("mar_b_one_image_graph", "graph", "mar_b", 16, 64, 2, "f16", 64, 0, 0.0),
        # one image again, step by step from the host: the latency an interactive caller sees
        _case("mar_l_one_image_step", "step", "mar_l", 16, 64, 2, "f16", 64, 40, 0.10),
        # a handful of images on an odd grid, all operands bf16
        _case("mar_b_ragged_step", "step", "mar_b", 15, 64, 10, "bf16", 64, 50, 0.10),
        # the benchmark batch: 64 images with guidance, mid run
        _case("mar_l_step", "step", "mar_l", 16, 64, 128, "f16", 64, 32, 0.10),
        # every token of the benchmark batch: first step of a run, and the baseline's every step
        _case("mar_l_full_step", "full", "mar_l", 16, 64, 128, "f16", 64, 0, 0.10),
        # the widest and deepest stack, head_dim 80
        _case("mar_h_step", "step", "mar_h", 16, 64, 128, "f16", 64, 32, 0.10),
        # 32 x 32 image tokens: long sequences, more than a hundred active rows per sample
        _case("hires_step", "step", "mar_l", 32, 64, 64, "f16", 64, 40, 0.10),
        # the paper's schedule: the first blocks on every token, selection inside the step
        _case("mar_b_in_step", "in_step", "mar_b", 16, 64, 16, "f16", 64, 31, 0.0),
        # encoder on the known tokens, decoder cache-aware
        _case("mar_l_two_stage", "two_stage", "mar_l", 16, 64, 32, "f16", 64, 40, 0.0),
        # a sampler that lives on the host drives the step through pinned buffers
        _case("mar_b_host_step", "host", "mar_b", 16, 64, 64, "f16", 64, 45, 0.10),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 4 + ["full", "in_step", "two_stage", "host", "generation", "graph", "select"])
    if kind == "generation":
        return _free(kind, "tiny", rng.randint(6, 12), 4, rng.randint(1, 12), "f32", 8, 0, rng.choice([0.05, 0.10, 0.20]))
    model = rng.choice(["mar_b", "mar_l", "mar_l", "mar_h"])
    grid = int(round(math.exp(rng.uniform(math.log(10), math.log(32)))))
    batch = int(round(math.exp(rng.uniform(0.0, math.log(128)))))
    operand = rng.choice(["f16", "f16", "bf16"])
    ratio = rng.choice([0.0, 0.05, 0.10, 0.10, 0.20])
    steps, t = 64, rng.randint(1, 63)
    if kind == "full":
        t = 0
    if kind == "graph":
        ratio, t = 0.0, 0
    if kind == "select":
        model, operand, ratio = "mar_b", "f16", max(ratio, 0.05)
    case = _free(kind, model, grid, 64, batch, operand, steps, t, ratio)
    # no dearer than the largest listed case (the full step of the benchmark batch)
    most = max(_seconds(c) for c in listed())
    while _seconds(case) > most and case["batch"] > 1:
        case["batch"] = case["batch"] * 3 // 4
    return case


def _free(*args):
    case = _case("", *args)
    del case["name"]
    return case


# ------------------------------------------------------------------------------------- sizes of a case
def _tokens(case):
    return case["grid"] ** 2 + case["buffer"]


def _counts(n_img, steps):
    """Tokens generated at each step: cosine schedule, at least one per step."""
    counts, masked = [], n_img
    for t in range(steps):
        left = 0 if t == steps - 1 else max(1, min(int(n_img * math.cos(math.pi / 2 * (t + 1) / steps)), masked - 1))
        counts.append(masked - left)
        masked = left
    return counts


def _refreshed(case, n_cand):
    return min(int(math.floor(case["ratio"] * _tokens(case) + 0.5)), n_cand)


def _sizes(case, t):
    """(tokens of step t, of the step before, of the step after, refreshed tokens) of one sample."""
    c = _counts(case["grid"] ** 2, case["steps"])
    new, prev, nxt = c[t], c[t - 1] if t > 0 else 0, c[t + 1] if t + 1 < len(c) else 0
    if case["kind"] in ("in_step", "two_stage"):
        return new, prev, nxt, max(0, min(BUDGET, _tokens(case)) - new - prev)
    return new, prev, nxt, _refreshed(case, _tokens(case) - new - prev)


def _blocks_work(case, n_blocks, rows, keys):
    """Bytes and flops of n_blocks blocks on `rows` rows per sample that attend to `keys` cached rows."""
    _, _, D, _, F = SHAPES[case["model"]]
    eb = 4 if case["operand"] == "f32" else 2
    B = case["batch"]
    weights = (4 * D * D + 2 * D * F) * eb
    cache = 2 * B * (keys + rows) * D * eb
    flops = 2 * B * rows * (4 * D * D + 2 * D * F) + 4 * B * rows * keys * D
    return n_blocks * (weights + cache), n_blocks * flops


def _step_work(case, t, full):
    S, B, D = _tokens(case), case["batch"], SHAPES[case["model"]][2]
    L = SHAPES[case["model"]][0]
    new, prev, _, k = _sizes(case, t)
    rows = S if full else new + prev + k
    b, f = _blocks_work(case, L, rows, S)
    return b + 2 * B * rows * D * 4 + 4 * B * (rows + k), f


def work(case):
    L, E, D, _, _ = SHAPES[case["model"]]
    S, B, t = _tokens(case), case["batch"], case["t"]
    new, prev, _, k = _sizes(case, t)
    if case["kind"] == "select":
        return {"bytes": B * (S * 4 + (new + _sizes(case, t)[2] + k) * 4), "flops": 0}
    if case["kind"] in ("generation", "graph"):
        parts = [_step_work(case, i, i == 0) for i in range(case["steps"])]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif case["kind"] == "in_step":
        (b0, f0), (b1, f1) = _blocks_work(case, E + 2, S, S), _blocks_work(case, L - E - 2, new + prev + k, S)
        b, f = b0 + b1 + 4 * B * D * (S + new + prev + k), f0 + f1
    elif case["kind"] == "two_stage":
        known = case["buffer"] + sum(_counts(case["grid"] ** 2, case["steps"])[:t])
        (be, fe), (b0, f0), (b1, f1) = (_blocks_work(case, E, known, known), _blocks_work(case, 2, S, S),
                                        _blocks_work(case, L - E - 2, new + prev + k, S))
        b, f = be + b0 + b1 + 4 * B * D * (known + new + prev + k), fe + f0 + f1 + 2 * B * known * D * D
    else:
        b, f = _step_work(case, t, case["kind"] == "full")
        if case["kind"] == "host":
            b += 2 * 4 * B * D * (new + prev)
    return {"bytes": b, "flops": f}


def _seconds(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / (1.4e15 if case["operand"] != "f32" else 5e13))


def tolerance(case):
    # Measured between the attention and projection kernels that the context can choose from, and for fp32 against the
    # same run in 64 bits; about four times the largest difference seen.
    if case["kind"] == "select":
        return "exact"
    if case["operand"] == "f32":
        return {"rel": 5e-6, "max": 1e-4}
    # The schedules that select inside the step may swap two tokens of nearly equal score: such a row is another row.
    swapped = case["kind"] in ("in_step", "two_stage")
    if case["operand"] == "f16":
        return {"rel": 6e-3, "max": 0.5 if swapped else 0.04}
    return {"rel": 1.8e-2, "max": 0.5 if swapped else 0.15}


# ------------------------------------------------------------------------------------- inputs and calls
def _weights(case, gen):
    L, _, D, _, F = SHAPES[case["model"]]

    def normal(*shape, mean=0.0, std=0.02):
        return torch.randn(*shape, generator=gen, device="cuda") * std + mean

    blocks = []
    for _ in range(L):
        w = dict(ln1_g=normal(D, mean=1.0), ln1_b=normal(D), w_qkv=normal(3 * D, D), b_qkv=normal(3 * D),
                 w_o=normal(D, D), b_o=normal(D), ln2_g=normal(D, mean=1.0), ln2_b=normal(D),
                 w_fc1=normal(F, D), b_fc1=normal(F), w_fc2=normal(D, F), b_fc2=normal(D))
        # the queries of a head share a direction, as in a trained stack: some tokens matter to all of them
        w["b_qkv"][:D] = normal(D, std=1.5)
        blocks.append(w)
    return blocks


def _mar_weights(case, gen):
    D, S = SHAPES[case["model"]][2], _tokens(case)

    def normal(*shape, mean=0.0, std=0.02):
        return torch.randn(*shape, generator=gen, device="cuda") * std + mean

    return dict(enc_norm_g=normal(D, mean=1.0), enc_norm_b=normal(D), w_dec_embed=normal(D, D, std=D ** -0.5),
                b_dec_embed=normal(D), mask_token=normal(D, std=1.0), dec_pos=normal(S, D, std=1.0),
                dec_norm_g=normal(D, mean=1.0), dec_norm_b=normal(D))


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    L, E, D, H, F = SHAPES[case["model"]]
    S, B, t, kind = _tokens(case), case["batch"], case["t"], case["kind"]
    dtype = "f32" if case["operand"] == "f32" else "bf16"
    m = Marche(L=L, E=E, D=D, H=H, F=F, S=S, B=B, dtype=dtype, n_buffer=case["buffer"],
               weights=upload_weights(_weights(case, gen), dtype, operand=case["operand"]))
    hidden = torch.randn(B, S, D, generator=gen, device="cuda")
    # every sample generates its image tokens in an order of its own; rows b and b + B/2 are one image under guidance
    images = B if B % 2 else B // 2
    order = torch.argsort(torch.rand(images, case["grid"] ** 2, generator=gen, device="cuda"), dim=1) + case["buffer"]
    order = order.repeat(B // images, 1).to(torch.int32)
    counts = _counts(case["grid"] ** 2, case["steps"])

    if kind in ("generation", "graph"):
        sets = list(torch.split(order, counts, dim=1))
        rows = [torch.randn(B, c, D, generator=gen, device="cuda") for c in counts]
        run = Generation(m, sets, case["ratio"], rows)
        s = dict(kind=kind, run=run, hidden=hidden)
        if kind == "graph":
            s["graph"] = run.capture(hidden)
        return s

    new, prev, nxt, k = _sizes(case, t)
    at = sum(counts[:t])
    G = order[:, at:at + new].contiguous()
    N = order[:, at - prev:at].contiguous() if prev else None
    X = order[:, at + new:at + new + nxt].contiguous() if nxt else None
    k_next = _refreshed(case, S - new - nxt)
    s = dict(kind=kind, m=m, ratio=case["ratio"], G=G, N=N, X=X, k=k, scores=torch.zeros(B, S, device="cuda"),
             refresh=torch.zeros(B, k_next, dtype=torch.int32, device="cuda"))
    if kind == "select":
        # sums of softmax weights over heads and new tokens: positive, spread over about a factor of ten
        s["scores"].normal_(0.0, 0.6, generator=gen).exp_()
        s["mask"] = torch.empty(B * S, dtype=torch.uint8, device="cuda")
        return s
    s.update(hidden=hidden, cache=m.alloc_cache(), out=torch.zeros(B, S, D, device="cuda"), ws=m.alloc_workspace(S))
    if kind == "full":
        m.init_cache(s["cache"])
        return s
    if kind == "two_stage":
        m.set_mar_weights(upload_mar_weights(_mar_weights(case, gen), dtype, operand=case["operand"]))
        known = torch.arange(case["buffer"], dtype=torch.int32, device="cuda").expand(B, -1)
        s["known"] = torch.cat([known, torch.sort(order[:, :at], dim=1).values], dim=1).contiguous()
    # the step before this one has filled the cache and the outputs
    m.init_cache(s["cache"])
    if kind == "two_stage":
        before = s["known"][:, :s["known"].shape[1] - prev].contiguous() if prev else s["known"]
        m.mar_step(True, hidden, before, s["cache"], N, None, 0, None, s["out"], None, None, s["ws"])
    else:
        m.full_step(hidden, s["cache"], N, G, 0.0, s["out"], None, s["ws"])
    sampled = torch.randn(B, prev, D, generator=gen, device="cuda")
    if kind in ("in_step", "two_stage"):
        s["active"] = torch.zeros(B, new + prev + k, dtype=torch.int32, device="cuda")
        s["refresh"] = torch.zeros(B, k, dtype=torch.int32, device="cuda")
    else:
        # the refresh set the step before has chosen: any tokens but the new and the previous ones
        key = torch.rand(B, S, generator=gen, device="cuda")
        key.scatter_(1, torch.cat([G, N], dim=1).long(), -1.0)
        s["R"] = torch.sort(torch.topk(key, k, dim=1).indices, dim=1).values.to(torch.int32).contiguous() if k else None
        s["active"] = torch.zeros(B, new + prev + k, dtype=torch.int32, device="cuda")
    if kind == "host":
        def pin(x):
            return None if x is None else x.cpu().pin_memory()
        s.update(h_rows=pin(sampled), h_N=pin(N), h_G=pin(G), h_X=pin(X), most=max(new, prev, nxt),
                 h_out=torch.zeros(B, new, D).pin_memory(), h_refresh=torch.zeros(B, k_next, dtype=torch.int32).pin_memory())
        s["staging"] = torch.empty(m.staging_bytes(s["most"]), dtype=torch.uint8, device="cuda")
    else:
        m.scatter_rows(sampled, N, hidden)       # the sampler's rows replace the previous tokens
    return s


def run(s):
    kind = s["kind"]
    if kind == "generation":
        s["run"].run(s["hidden"])
        return s["run"].hidden_out, s["run"].cache, s["run"].hidden
    if kind == "graph":
        s["graph"].replay()
        return s["run"].hidden_out, s["run"].cache, s["run"].hidden
    m, ratio = s["m"], s["ratio"]
    if kind == "select":
        m.select_refresh(s["scores"], s["G"], s["X"], s["refresh"].shape[1], s["refresh"], s["mask"])
        return s["refresh"]
    # What a step computes: hidden rows, cache and relevance scores.  The refreshed tokens follow from the scores (the
    # "select" case returns them); their ascending list is left out here, since one swap of a near-tie shifts the rest.
    if kind == "step":
        m.build_active(s["G"], s["N"], s["R"], s["k"], s["active"])
        m.step(s["hidden"], s["cache"], s["active"], s["G"], s["X"], ratio, s["out"], s["refresh"], s["ws"])
    elif kind == "full":
        m.full_step(s["hidden"], s["cache"], s["G"], s["X"], ratio, s["out"], s["refresh"], s["ws"])
    elif kind == "in_step":
        m.step_in_step_selection(s["hidden"], s["cache"], s["G"], s["N"], s["k"], None, s["out"], s["refresh"],
                                 s["active"], s["ws"])
    elif kind == "two_stage":
        m.mar_step(False, s["hidden"], s["known"], s["cache"], s["G"], s["N"], s["k"], None, s["out"], s["refresh"],
                   s["active"], s["ws"])
    else:
        m.step_host(False, s["hidden"], s["cache"], s["h_rows"], s["h_N"], s["h_G"], s["h_X"], s["R"], s["k"], ratio,
                    s["out"], s["refresh"], s["h_out"], s["h_refresh"], s["most"], s["staging"], s["ws"])
        torch.cuda.current_stream().synchronize()     # the caller's sampler reads the rows on the host
        return s["h_out"], s["out"], s["cache"], s["hidden"]
    m.get_scores(s["ws"], s["scores"])
    return s["out"], s["cache"], s["scores"]
