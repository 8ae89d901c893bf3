"""The library's work as a scoring service has it do it, case by case.

A case is one call (or the short fixed sequence of calls) that a user's program
makes through the public binding, on inputs drawn from a seed.  The kinds:

  linear     one int4 linear layer, plain or with the fused epilogue
             (w4a16.linear, w4a16.linear_fused);
  stack      the linear layers of one decoder layer in order, as a captured
             graph or launched from the host (w4a16.StackGraph, linear_stack);
  attention  causal sliding-window attention over a packed batch;
  head       the affinity head: one hidden state per pair, then a small int4
             linear with a bias (w4a16.gather_rows, linear_fused);
  topk       the k best of a screening set's scores;
  weights    weight preparation: quantise fp32 masters, dequantise the result.

Sizes are those of the decoder that the benchmark measures (width 12288, MLP
4x, 96 heads of 128, group 128), and ragged ones around them.
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_2608_30877_gb300 import synthetic as S
from paper_2608_30877_gb300 import w4a16 as W

D = S.D_MODEL
FF = S.D_FF
ACTS = {"none": W.ACT_NONE, "swiglu": W.ACT_SWIGLU, "gelu": W.ACT_GELU}
EXACT_FLOPS = 8e12  # above this the 64-bit product takes longer than it is worth


def _linear(name, M, N, K, g=128, act="none", bias=False, residual=False):
    return {"name": name, "kind": "linear", "M": M, "N": N, "K": K, "g": g, "act": act,
            "bias": bias, "residual": residual}


def listed():
    return [
        # the affinity head of one scored batch: 64 pairs' states, two readouts;
        # the smallest call, all latency
        {"name": "head_64_pairs", "kind": "head", "tokens": 65536, "pairs": 64, "D": D, "N": 2},
        # sorting the predictions of a whole screening set for export
        {"name": "topk_200k", "kind": "topk", "n": 200000, "k": 1000, "bf16": False},
        # one token through the widest layer: the weights stream once
        _linear("up_m1", 1, FF, D),
        # decode of a small batch: one decoder layer's four linears, captured
        {"name": "layer_m8_graph", "kind": "stack", "M": 8, "d": D, "g": 128, "graph": True},
        # a short batch on weights with the finer scale groups
        _linear("qkv_m24_g64", 24, 3 * D, D, g=64),
        # a short ragged prefill through the down projection and its residual
        _linear("down_m100_residual", 100, D, FF, bias=True, residual=True),
        # one pair's tokens through the attention output projection
        _linear("o_m333_residual", 333, D, D, residual=True),
        # prefill of eight packed pairs, fused QKV
        _linear("qkv_m4096", 4096, 3 * D, D),
        # the largest call: gate and up projections with SwiGLU in the output stage
        _linear("swiglu_m8192", 8192, 2 * FF, D, act="swiglu"),
        # attention of a scored batch of 64 pairs of ragged lengths
        {"name": "attention_64_pairs", "kind": "attention", "nseq": 64, "shortest": 200,
         "longest": 1024, "H": 96, "window": 32768},
        # one long sequence under a sliding window
        {"name": "attention_long_window", "kind": "attention", "nseq": 1, "shortest": 10007,
         "longest": 10007, "H": 96, "window": 4096},
        # preparing one square projection: fp32 masters to int4 and back to bf16
        {"name": "weights_square", "kind": "weights", "N": D, "K": D, "g": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["linear"] * 6 + ["attention"] * 2 + ["stack", "head", "topk", "weights"])
    if kind == "linear":
        g = rng.choice([128, 128, 128, 128, 64, 256])
        M = _log_int(rng, 1, 8192)
        # widths of a decoder's projections, ragged ones among them
        N = rng.choice([D, 2 * D, 3 * D, FF, _log_int(rng, 512, FF)])
        K = rng.choice([D, D, FF, _log_int(rng, 512, FF)]) // g * g
        act = rng.choice(["none", "none", "swiglu", "gelu"])
        if act == "swiglu":
            N += N % 2
        if M > 2048:  # no more work than the largest listed case
            N = min(N, 3 * D)
            K = min(K, D)
        return {"kind": "linear", "M": M, "N": N, "K": K, "g": g, "act": act,
                "bias": rng.random() < 0.5, "residual": rng.random() < 0.4}
    if kind == "stack":
        return {"kind": "stack", "M": _log_int(rng, 1, 128), "d": rng.choice([2048, 4096, 8192, D]),
                "g": 128, "graph": rng.random() < 0.7}
    if kind == "attention":
        if rng.random() < 0.6:  # packed pairs
            longest = rng.randint(256, 2048)
            return {"kind": "attention", "nseq": _log_int(rng, 2, 64),
                    "shortest": rng.randint(32, longest // 2), "longest": longest,
                    "H": rng.choice([16, 32, 64, 96]), "window": 32768}
        n = _log_int(rng, 2048, 12000)
        return {"kind": "attention", "nseq": 1, "shortest": n, "longest": n,
                "H": rng.choice([16, 32, 64]), "window": rng.choice([1000, 4096, 32768])}
    if kind == "head":
        return {"kind": "head", "tokens": _log_int(rng, 4096, 65536), "pairs": _log_int(rng, 8, 512),
                "D": rng.choice([2048, 4096, D]), "N": rng.choice([1, 2, 3, 8])}
    if kind == "topk":
        n = _log_int(rng, 2000, 2000000)
        return {"kind": "topk", "n": n, "k": min(n, _log_int(rng, 10, 1024)),
                "bf16": rng.random() < 0.3}
    g = rng.choice([64, 128, 256])
    return {"kind": "weights", "N": _log_int(rng, 500, 2 * D), "K": _log_int(rng, 1024, D) // g * g,
            "g": g}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16)


def _weights(gen, N, K, g):
    """N(0, 0.02) masters in the library's int4 format, as a stored model has them."""
    packed = torch.empty((N, K // 2), dtype=torch.uint8, device="cuda")
    scales = torch.empty((N, K // g), dtype=torch.bfloat16, device="cuda")
    step = max(1, (1 << 26) // K)
    for r in range(0, N, step):
        rows = min(step, N - r)
        w = torch.randn((rows, K // g, g), generator=gen, device="cuda").mul_(0.02)
        s = (w.abs().amax(-1) / 7.0).to(torch.bfloat16)
        q = (w / s.float().unsqueeze(-1)).round_().clamp_(-8, 7).add_(8).to(torch.uint8)
        q = q.view(rows, K)
        packed[r:r + rows] = q[:, 0::2] | (q[:, 1::2] << 4)
        scales[r:r + rows] = s
    return packed, scales


def _lengths(case):
    """The batch's sequence lengths: ragged over the range, the same for every seed, so
    that a case has one token count."""
    span = case["longest"] - case["shortest"] + 1
    return [case["shortest"] + (i * 0x9E3779B1 >> 8) % span for i in range(1, case["nseq"] + 1)]


def _stack_shapes(d):
    return [(3 * d, d), (d, d), (4 * d, d), (d, 4 * d)]  # (N, K): qkv, o, up, down


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        n_out = N // 2 if case["act"] == "swiglu" else N
        s["x"] = _normal(gen, M, K)
        s["w"], s["scales"] = _weights(gen, N, K, case["g"])
        s["bias"] = _normal(gen, N) if case["bias"] else None
        s["residual"] = _normal(gen, M, n_out) if case["residual"] else None
    elif kind == "stack":
        s["layers"] = []
        for N, K in _stack_shapes(case["d"]):
            w, sc = _weights(gen, N, K, case["g"])
            out = torch.empty((case["M"], N), dtype=torch.bfloat16, device="cuda")
            s["layers"].append((_normal(gen, case["M"], K), w, sc, out))
        if case["graph"]:
            s["graph"] = W.StackGraph(s["layers"], case["M"], case["g"])
    elif kind == "attention":
        starts = list(itertools.accumulate(_lengths(case), initial=0))
        s["seq_start"] = torch.tensor(starts, dtype=torch.int32, device="cuda")
        s["qkv"] = _normal(gen, starts[-1], 3 * case["H"] * 128)
    elif kind == "head":
        s["hidden"] = _normal(gen, case["tokens"], case["D"])
        last = torch.randperm(case["tokens"], generator=gen, device="cuda")[:case["pairs"]]
        s["last"] = last.sort().values.to(torch.int32)
        s["w"], s["scales"] = _weights(gen, case["N"], case["D"], 128)
        s["bias"] = _normal(gen, case["N"])
    elif kind == "topk":
        v = torch.randn(case["n"], generator=gen, device="cuda") * 3 - 8  # kcal/mol
        s["scores"] = v.to(torch.bfloat16) if case["bf16"] else v
    else:
        s["master"] = torch.randn((case["N"], case["K"]), generator=gen, device="cuda").mul_(0.02)
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "linear":
        if case["act"] == "none" and not case["bias"] and not case["residual"]:
            return W.linear(s["x"], s["w"], s["scales"], case["g"])
        return W.linear_fused(s["x"], s["w"], s["scales"], case["g"], act=ACTS[case["act"]],
                              bias=s["bias"], residual=s["residual"])
    if kind == "stack":
        if case["graph"]:
            s["graph"].launch()
        else:
            W.linear_stack(s["layers"], case["M"], case["g"])
        return [layer[3] for layer in s["layers"]]
    if kind == "attention":
        return W.attention_prefill(s["qkv"], s["seq_start"], case["H"], window=case["window"])
    if kind == "head":
        states = W.gather_rows(s["hidden"], s["last"])
        return [states, W.linear_fused(states, s["w"], s["scales"], 128, bias=s["bias"])]
    if kind == "topk":
        return W.topk_smallest(s["scores"], case["k"])
    packed, scales = W.quantize(s["master"], case["g"])
    return [packed, scales, W.dequant(packed, scales, case["g"])]


# ---------------------------------------------------------------- what a pass needs

def _linear_work(M, N, K, g, n_out, bias=False, residual=False):
    return {"bytes": N * K / 2 + 2 * N * (K // g) + 2 * M * K + 2 * M * n_out * (2 if residual else 1)
            + (2 * N if bias else 0), "flops": 2.0 * M * N * K}


def work(case):
    kind = case["kind"]
    if kind == "linear":
        n_out = case["N"] // 2 if case["act"] == "swiglu" else case["N"]
        return _linear_work(case["M"], case["N"], case["K"], case["g"], n_out, case["bias"],
                            case["residual"])
    if kind == "stack":
        parts = [_linear_work(case["M"], N, K, case["g"], N) for N, K in _stack_shapes(case["d"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "attention":
        lengths = _lengths(case)
        # keys visible over all queries: causal, at most `window` each
        full = [min(n, case["window"]) for n in lengths]
        visible = sum(f * (f + 1) / 2 + (n - f) * f for n, f in zip(lengths, full))
        return {"bytes": sum(lengths) * case["H"] * 128 * 2 * 4 + 4 * (case["nseq"] + 1),
                "flops": 4.0 * 128 * case["H"] * visible}
    if kind == "head":
        lin = _linear_work(case["pairs"], case["N"], case["D"], 128, case["N"], bias=True)
        return {"bytes": lin["bytes"] + 4 * case["pairs"] + 2 * case["pairs"] * case["D"],
                "flops": lin["flops"]}
    if kind == "topk":
        return {"bytes": case["n"] * (2 if case["bf16"] else 4) + 8 * case["k"], "flops": 0}
    NK = case["N"] * case["K"]
    # masters read, int4 and scales written; int4 and scales read, bf16 written
    return {"bytes": 4.0 * NK + 2 * (NK / 2 + 2.0 * NK / case["g"]) + 2.0 * NK, "flops": 0}


def tolerance(case):
    if case["kind"] in ("topk", "weights"):
        return "exact"
    # One bf16 rounding of the output is 1.7e-3 in the 2-norm; applying a group's scale
    # to the fp32 partial sum instead of rounding every weight adds 1.2e-3, and
    # P rounded to bf16 about 2e-3 in attention.
    return {"rel": 8e-3, "max": 6e-2}


# ---------------------------------------------------------------- 64-bit results

def _exact_product(x, packed, scales, g):
    """x times the dequantised weights (bf16 by definition of the format), in 64 bits."""
    N, K = packed.shape[0], packed.shape[1] * 2
    out = torch.empty((x.shape[0], N), dtype=torch.float64, device="cuda")
    xd = x.double()
    step = max(1, (1 << 26) // K)
    for r in range(0, N, step):
        b = packed[r:r + step]
        q = torch.stack([b & 15, b >> 4], dim=-1).view(b.shape[0], K // g, g).float() - 8
        wd = (q * scales[r:r + step].float().unsqueeze(-1)).to(torch.bfloat16)
        out[:, r:r + step] = xd @ wd.view(b.shape[0], K).double().t()
    return out


def _exact_fused(y, act, bias, residual):
    z = y if bias is None else y + bias.double()
    if act == "swiglu":
        z = torch.nn.functional.silu(z[:, 0::2]) * z[:, 1::2]
    elif act == "gelu":
        z = torch.nn.functional.gelu(z)
    return z if residual is None else z + residual.double()


def _exact_attention(qkv, starts, H, window):
    out = torch.empty((qkv.shape[0], H, 128), dtype=torch.float64, device="cuda")
    for a, b in zip(starts[:-1], starts[1:]):
        t = qkv[a:b].view(b - a, 3, H, 128).permute(1, 2, 0, 3)  # q, k, v: [H, n, 128]
        for i in range(0, b - a, 512):
            j = min(i + 512, b - a)
            lo = max(0, i - window + 1)
            rows = torch.arange(i, j, device="cuda").unsqueeze(1)
            keys = torch.arange(lo, j, device="cuda").unsqueeze(0)
            hidden = (keys > rows) | (keys <= rows - window)
            for h in range(0, H, 16):  # a few heads at a time
                q, k, v = (t[0, h:h + 16, i:j].double(), t[1, h:h + 16, lo:j].double(),
                           t[2, h:h + 16, lo:j].double())
                p = (q @ k.transpose(1, 2) / math.sqrt(128.0)).masked_fill_(hidden, -math.inf)
                out[a + i:a + j, h:h + 16] = (p.softmax(-1) @ v).transpose(0, 1)
    return out.view(qkv.shape[0], H * 128)


def exact(case, seed):
    if case["kind"] in ("topk", "weights") or work(case)["flops"] > EXACT_FLOPS:
        return None
    s = prepare({**case, "graph": False} if case["kind"] == "stack" else case, seed)
    kind = case["kind"]
    if kind == "linear":
        y = _exact_product(s["x"], s["w"], s["scales"], case["g"])
        return _exact_fused(y, case["act"], s["bias"], s["residual"])
    if kind == "stack":
        return [_exact_product(x, w, sc, case["g"]) for x, w, sc, _ in s["layers"]]
    if kind == "attention":
        return _exact_attention(s["qkv"], s["seq_start"].tolist(), case["H"], case["window"])
    states = s["hidden"][s["last"].long()]
    return [states.double(), _exact_product(states, s["w"], s["scales"], 128) + s["bias"].double()]
