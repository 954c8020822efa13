"""The work whose speed is watched: passes of the packed Pairformer-style block through the calls a user's program makes.

listed()   the cases that stand for the range; draw() gives more of the same ranges.
prepare()  weights, layout, workspace and inputs on the device: what a program holds before it calls.
run()      one pass: new tokens are copied into the (in place updated) token buffer, then the block or stack runs.
work()     bytes and flops a pass cannot do without; tolerance() what two correct implementations may differ by.

Kinds of pass
  stack       runner.PairStack on pair lengths.  mode "cached": forward_cached, a length signature that comes back;
              "launched": forward, every call issued by the host; "fresh": a new Layout for every batch, then forward.
  token       runner.PairStack of the single-ragged special case (token attention and pooled mean).
  pairformer  the whole block through binding: broadcast, both triangle updates, row and column attention, transition,
              pair-biased single attention, mean and token update; from the second block on the broadcast is
              accumulated onto the pair state (a persistent pair stream).
  rect        rectangular pairs: broadcast from row and column tokens, transition, mean over the columns, token update.
"""
import math

import torch

from paper_2609_30379_b200 import binding as nt
from paper_2609_30379_b200 import runner
from paper_2609_30379_b200 import workloads as wl

EPS = runner.LN_EPS

# widths (c_s, c_z, c_h, H, d) of the configurations in workloads.py
WIDE = dict(c_s=384, c_z=128, c_h=128, H=4, d=32)      # cfg2, cfg3
NARROW = dict(c_s=256, c_z=64, c_h=64, H=4, d=16)      # cfg5
TINY = dict(c_s=32, c_z=16, c_h=16, H=2, d=8)          # cfg1
TOKEN = dict(c_s=768, c_z=768, c_h=0, H=12, d=64)      # cfg4


def _text(lengths):
    return " ".join(str(int(n)) for n in lengths)


def _ints(text):
    return tuple(int(n) for n in text.split())


def _case(kind, dtype, lengths, widths, blocks=1, **more):
    return dict(kind=kind, dtype=dtype, lengths=_text(lengths), blocks=blocks, **widths, **more)


def listed():
    cfgs = wl.CONFIGS
    named = {
        # the correctness block of a test suite or a notebook: launches and host time are all there is
        "tiny_f32": _case("stack", "f32", cfgs["cfg1"].lengths, TINY, mode="launched"),
        # single precision in earnest (validation runs, numerics comparisons) on short samples
        "ordinary_f32": _case("stack", "f32", (110, 24, 71, 37, 96, 64), NARROW, mode="launched"),
        # a few short samples, never seen together before: layout built and every kernel launched from the host
        "small_fresh": _case("stack", "bf16", (18, 61, 7, 33), WIDE, blocks=4, mode="fresh"),
        # near-uniform lengths whose signature comes back (the benchmark's workload), replayed as a graph
        "uniform_stack": _case("stack", "bf16", cfgs["cfg2"].lengths, WIDE, blocks=4, mode="cached"),
        # lengths that vary by a factor of 16 in one batch, launched by the host as a new batch would be
        "varied_stack": _case("stack", "bf16", cfgs["cfg3"].lengths, WIDE, blocks=4, mode="launched"),
        # the largest pair states: samples of up to 2048 tokens
        "large_stack": _case("stack", "bf16", cfgs["cfg5"].lengths, NARROW, blocks=2, mode="launched"),
        # sentence-length token batches: attention over the token axis and a pooled mean
        "token_batch": _case("token", "bf16", cfgs["cfg4"].lengths, TOKEN),
        # three short sequences of one request: the smallest token call
        "token_small": _case("token", "bf16", (23, 61, 5), TOKEN),
        # one whole block (every sub-layer) on near-uniform lengths
        "pairformer_uniform": _case("pairformer", "bf16", cfgs["cfg2"].lengths, WIDE),
        # two whole blocks with a persistent pair stream on a ragged batch, short and long samples mixed
        "pairformer_ragged": _case("pairformer", "bf16", (131, 37, 401, 88, 243, 59, 310, 180), WIDE, blocks=2),
        # one long sample alone, the ordinary shape of a prediction served by itself
        "pairformer_long": _case("pairformer", "bf16", (977,), WIDE),
        # rectangular pairs of the benchmark's rectangular workload: rows 130-221, columns 148-224
        "rect_block": _case("rect", "bf16", (135, 201, 180, 216, 130, 172, 221, 158), WIDE,
                            columns=_text((224, 161, 148, 203, 187, 219, 170, 152))),
    }
    return [dict(case, name=name) for name, case in named.items()]


def _draw_lengths(rng, most_tokens, longest, exponent, most):
    """B lengths, near-uniform or spread over their logarithm, with sum N^exponent bounded by `most`."""
    B = int(round(math.exp(rng.uniform(0.0, math.log(24.5)))))
    top = math.exp(rng.uniform(math.log(8.0), math.log(longest)))
    low = top * rng.choice((0.9, 0.5, 0.06))
    n = [max(1, int(round(math.exp(rng.uniform(math.log(low), math.log(top)))))) for _ in range(B)]
    while len(n) > 1 and (sum(v ** exponent for v in n) > most or sum(n) > most_tokens):
        n.pop()
    return tuple(n)


def draw(rng):
    kind = rng.choice(("stack", "stack", "stack", "f32", "token", "pairformer", "pairformer", "rect"))
    if kind == "token":
        return _case("token", "bf16", _draw_lengths(rng, 9000, 512, 2, 3e6), TOKEN)
    if kind == "f32":
        widths = rng.choice((TINY, NARROW))
        return _case("stack", "f32", _draw_lengths(rng, 1000, 130, 2, 4e4), widths, mode="launched")
    widths = rng.choice((WIDE, WIDE, NARROW))
    if kind == "rect":
        rows = _draw_lengths(rng, 6000, 400, 2, 8e5)
        return _case("rect", "bf16", rows, widths,
                     columns=_text(max(1, int(round(n * rng.uniform(0.6, 1.6)))) for n in rows))
    lengths = _draw_lengths(rng, 8000, 1100, 3, 1.5e9)
    if kind == "pairformer":
        return _case("pairformer", "bf16", lengths, widths, blocks=rng.choice((1, 2)))
    return _case("stack", "bf16", lengths, widths, blocks=rng.choice((1, 2, 4)),
                 mode=rng.choice(("cached", "launched", "fresh")))


# ---------------------------------------------------------------------------------------------------------------
def _config(case, seed, blocks):
    return wl.Config("case", case["dtype"], _ints(case["lengths"]), case["c_s"], case["c_z"], case["c_h"], case["H"],
                     case["d"], blocks, seed=1 + 2 * seed, kind="token" if case["kind"] == "token" else "pair")


def _bytes_buffer(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("stack", "token"):
        cfg = _config(case, seed, case["blocks"])
        host = wl.make_inputs(cfg)
        stack = runner.PairStack(cfg, cfg.lengths, host["blocks"])
        x0 = runner.to_device(host["x"], stack.dtype)
        return dict(case=case, stack=stack, lengths=cfg.lengths, x0=x0, x=torch.empty_like(x0))
    if kind == "rect":
        return _prepare_rect(case, seed)
    return _prepare_pairformer(case, seed)


def _prepare_pairformer(case, seed):
    # two sets of block weights each: the second set's triangle and attention weights serve the incoming / column forms
    n = case["blocks"]
    cfg = _config(case, seed, 2 * n)
    host = wl.make_inputs(cfg)
    bf = torch.bfloat16
    W = runner.upload_weights(host["blocks"], bf)
    for w in W:
        for key in ("trimul", "attn"):
            buf = _bytes_buffer(nt.NT_PREPARED_WEIGHTS_BYTES)
            if key == "trimul":
                nt.nt_prepare_trimul_weights(w[key], buf)
            else:
                nt.nt_prepare_attn_weights(w[key], cfg.H, cfg.d, buf)
            w[key]["prepared"] = buf
    blocks = []
    for k in range(n):
        one, two = W[2 * k], W[2 * k + 1]
        up = lambda d: {name: runner.to_device(a, bf) for name, a in d.items()}  # noqa: E731
        blocks.append(dict(broadcast=one["broadcast"], tri_out=one["trimul"], tri_in=two["trimul"], row=one["attn"],
                           col=two["attn"], transition=up(wl.make_transition_weights(cfg, k)),
                           single=up(wl.make_single_attn_weights(cfg, k)), reduce=one["reduce"]))
    L = nt.Layout(cfg.lengths)
    dims = (cfg.c_s, cfg.c_z, cfg.c_h, cfg.H, cfg.d)
    ws = max(nt.nt_workspace_bytes(nt.NT_OP_BLOCK, nt.NT_BF16, nt.NT_ORDER_PAIR_IJC, L.lengths_h, dims),
             nt.nt_transition_workspace_bytes(bf, cfg.c_z, 4 * cfg.c_z, L.T2),
             nt.nt_single_attn_workspace_bytes(bf, cfg.lengths, cfg.c_s, cfg.H, cfg.d))
    x0 = runner.to_device(host["x"], bf)
    return dict(case=case, cfg=cfg, L=L, blocks=blocks, x0=x0, x=torch.empty_like(x0),
                z=torch.empty((L.T2, cfg.c_z), dtype=bf, device="cuda"),
                m=torch.empty((L.T1, cfg.c_z), dtype=bf, device="cuda"), ws=_bytes_buffer(ws))


def _prepare_rect(case, seed):
    cfg = _config(case, seed, 1)
    bf = torch.bfloat16
    host = wl.make_inputs(cfg)
    L = nt.RectLayout(cfg.lengths, _ints(case["columns"]))
    w = runner.upload_weights(host["blocks"], bf)[0]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x0 = runner.to_device(host["x"], bf)
    ws = max(nt.nt_rect_broadcast_workspace_bytes(L, cfg.c_z), nt.nt_transition_workspace_bytes(bf, cfg.c_z, 4 * cfg.c_z, L.T2))
    return dict(case=case, L=L, b=w["broadcast"], W_r=w["reduce"]["W_r"], x0=x0, x=torch.empty_like(x0),
                transition={k: runner.to_device(a, bf) for k, a in wl.make_transition_weights(cfg).items()},
                y=torch.randn((L.T1m, cfg.c_s), generator=gen, device="cuda").to(bf),
                z=torch.empty((L.T2, cfg.c_z), dtype=bf, device="cuda"),
                m=torch.empty((L.T1n, cfg.c_z), dtype=bf, device="cuda"), ws=_bytes_buffer(ws))


# ---------------------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    x = state["x"]
    x.copy_(state["x0"])
    if case["kind"] == "stack":
        stack = state["stack"]
        if case["mode"] == "cached":
            return stack.forward_cached(x)
        if case["mode"] == "fresh":
            stack.L = nt.Layout(state["lengths"])
        return stack.forward(x)
    if case["kind"] == "token":
        return state["stack"].forward(x)
    if case["kind"] == "rect":
        b, L, z, m, ws = state["b"], state["L"], state["z"], state["m"], state["ws"]
        nt.nt_rect_pair_broadcast(L, x, state["y"], b["W_a"], b["W_b"], b["ln_gamma"], b["ln_beta"], EPS, z, ws)
        nt.nt_pair_transition(state["transition"], EPS, z, ws, L.status)
        nt.nt_segment_reduce(nt.NT_REDUCE_MEAN, L.row_splits, z, m, L.status)
        nt.nt_token_update(m, state["W_r"], x)
        return x, z
    cfg, L, z, m, ws = state["cfg"], state["L"], state["z"], state["m"], state["ws"]
    for k, w in enumerate(state["blocks"]):
        b = w["broadcast"]
        broadcast = nt.nt_pair_broadcast_add if k else nt.nt_pair_broadcast
        broadcast(L, x, b["W_a"], b["W_b"], b["ln_gamma"], b["ln_beta"], EPS, z, ws)
        nt.nt_tri_mul_out(L, w["tri_out"], EPS, z, ws)
        nt.nt_tri_mul_in(L, w["tri_in"], EPS, z, ws)
        nt.nt_row_attn_pairbias(L, nt.NT_ORDER_PAIR_IJC, w["row"], cfg.H, cfg.d, EPS, z, ws)
        nt.nt_col_attn_pairbias(L, w["col"], cfg.H, cfg.d, EPS, z, ws)
        nt.nt_pair_transition(w["transition"], EPS, z, ws, L.status)
        nt.nt_single_attn_pairbias(L, w["single"], cfg.H, cfg.d, EPS, x, z, ws)
        nt.nt_segment_reduce(nt.NT_REDUCE_MEAN, L.row_splits, z, m, L.status)
        nt.nt_token_update(m, w["reduce"]["W_r"], x)
    return x, z


# ---------------------------------------------------------------------------------------------------------------
def work(case):
    n = _ints(case["lengths"])
    c_s, c, c_h, Hd = case["c_s"], case["c_z"], case["c_h"], case["H"] * case["d"]
    H, blocks, e = case["H"], case["blocks"], 4 if case["dtype"] == "f32" else 2
    T1, T2, N3 = sum(n), sum(v * v for v in n), sum(v ** 3 for v in n)
    if case["kind"] == "token":
        weights = 4 * Hd * c
        flops = 2 * T1 * c * Hd * 4 + 4 * T2 * Hd
        return dict(bytes=e * (2 * T1 * c + len(n) * c + weights), flops=flops)
    broadcast, update = 4 * T1 * c_s * c, 2 * T1 * c * c_s
    w_broadcast, w_update = 2 * c * c_s, c * c_s
    hidden = 4 * c
    transition, w_transition = 6 * T2 * c * hidden, 3 * c * hidden
    if case["kind"] == "rect":
        cols = _ints(case["columns"])
        T1m, T2 = sum(cols), sum(a * b for a, b in zip(n, cols))
        flops = 2 * (T1 + T1m) * c_s * c + 6 * T2 * c * hidden + T2 * c + update
        return dict(bytes=e * (2 * T1 * c_s + T1m * c_s + T2 * c + w_broadcast + w_transition + w_update), flops=flops)
    # one direction of the triangle update: gated projections, contraction, gate and output projection
    tri = 2 * T2 * c * 4 * c_h + 2 * N3 * c_h + 2 * T2 * (c + c_h) * c
    w_tri = 4 * c_h * c + c * c + c * c_h
    # one pair attention: q, k, v, bias, gate, scores and weighted sum, output projection
    attn = 2 * T2 * c * (4 * Hd + H) + 4 * N3 * Hd + 2 * T2 * Hd * c
    w_attn = (5 * Hd + H) * c
    one = broadcast + tri + attn + T2 * c + update
    w_one = w_broadcast + w_tri + w_attn + w_update
    if case["kind"] == "pairformer":
        single = 2 * T1 * c_s * 5 * Hd + 2 * T2 * c * H + 4 * T2 * Hd
        one += tri + attn + transition + single
        w_one += w_tri + w_attn + w_transition + 5 * Hd * c_s + H * c
    return dict(bytes=e * (2 * T1 * c_s + T2 * c + blocks * w_one), flops=blocks * one)


def tolerance(case):
    # float32 storage and sums; bf16 storage of state and intermediates between the calls, float32 sums
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
