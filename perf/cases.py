"""The work that programs built on this library have it do, as timed cases through its public calls.

A case is a dict of plain values; ``kind`` names the path:

* ``layer``    -- MXInt linear layers (``mx_linear``; ``mx_linear_q`` when the result is MXInt): activations in
                  floating point, weights stored quantized.  One or several layers per pass.
* ``stack``    -- decode: all weight matrices of a stack of decoder layers in one ``mx_linear_grouped`` call.
* ``quantize`` -- ``mx_quantize`` of a tensor (weights at load time, activations, a value cache along the tokens)
                  and ``mx_dequantize`` of the codes.
* ``block``    -- one pre-LayerNorm decoder block, ``decoder_block.run``.

Inputs are drawn on the GPU from the case's seed with the structure of the workloads in
``paper_2307_15517_b200/synth.py``: Gaussian weights of small variance, activations with a few large channels or
heavy tails.
"""
from __future__ import annotations

import math

import torch

from paper_2307_15517_b200 import binding as mxb
from paper_2307_15517_b200 import decoder_block as dblk
from paper_2307_15517_b200 import synth

DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16}


def _layer(name, tokens, layers, block, w_act, w_wgt, **more):
    """``layers``: "KxN" pairs separated by blanks; ``w_act`` / ``w_wgt`` / ``block``: one value, or one per layer."""
    case = dict(kind="layer", tokens=tokens, layers=layers, block=str(block), w_act=str(w_act), w_wgt=str(w_wgt),
                dtype="fp32", acts="outlier", bias=False, rows2=False, w_out=0)
    case.update(more)
    if name:
        case["name"] = name
    return case


def _stack(name, tokens, hidden, ffn, depth, **more):
    case = dict(kind="stack", tokens=tokens, hidden=hidden, ffn=ffn, depth=depth, w_act=8, w_wgt=4, dtype="fp32")
    case.update(more)
    if name:
        case["name"] = name
    return case


def _quantize(name, rows, K, block, width, dtype, along_rows=False, back=False):
    case = dict(kind="quantize", rows=rows, K=K, block=block, width=width, dtype=dtype, along_rows=along_rows, back=back)
    if name:
        case["name"] = name
    return case


def _block(name, seq, heads, head_dim, ffn, block=16, w_act=8, w_wgt=4):
    case = dict(kind="block", seq=seq, heads=heads, head_dim=head_dim, ffn=ffn, block=block, w_act=w_act, w_wgt=w_wgt)
    if name:
        case["name"] = name
    return case


def _mixed_pass():
    specs = synth.llama7b_mixed_layers(0)
    return dict(layers=" ".join("%dx%d" % (s.K, s.N) for s in specs), block=" ".join(str(s.block) for s in specs),
                w_act=" ".join(str(s.w_act) for s in specs), w_wgt=" ".join(str(s.w_wgt) for s in specs))


def listed():
    return [
        # one token through one projection of a 7B-parameter model: the smallest call a decode loop makes
        _layer("decode_layer_1", 1, "4096x4096", 32, 8, 4, acts="gauss"),
        # one small layer on its own (768 wide, a short prompt): launches and host work
        _layer("single_layer", 128, "768x768", 16, 4, 4),
        # the four linears of an OPT-1.3B-shaped block over a 2048-token prompt, MXInt4: the benchmark's step
        _layer("prefill_2048", 2048, "2048x6144 2048x2048 2048x8192 8192x2048", 16, 4, 4),
        # the seven linears of a LLaMA-7B-shaped block over 4096 tokens, a width and a block size searched per layer
        _layer("prefill_mixed", synth.LLAMA7B_TOKENS, acts="heavy", **_mixed_pass()),
        # a prompt and layer sizes that fit no tile, MXInt6, bias, bf16 activations
        _layer("layer_ragged", 1237, "2080x3002", 16, 6, 6, dtype="bf16", bias=True),
        # a gate projection whose result is the next operator's MXInt8 operand, bf16 activations
        _layer("layer_requant", 512, "4096x11008", 16, 8, 4, dtype="bf16", acts="heavy", w_out=8),
        # decode with 1 token: every weight matrix of 32 layers (2.7 GB packed) read once
        _stack("decode_stack_1", 1, 4096, 11008, 32),
        # decode with 16 sequences at a time, a quarter of the stack
        _stack("decode_stack_16", 16, 4096, 11008, 8),
        # a large fp32 tensor (a layer's weights at load time, a long prompt's activations) to MXInt4
        _quantize("quantize_large", 16384, 8192, 16, 4, "fp32"),
        # a short prompt's bf16 values to MXInt8 along the tokens (the operand of P V), and back
        _quantize("quantize_tokens", 352, 2048, 32, 8, "bf16", along_rows=True, back=True),
        # one OPT-6.7B-shaped decoder block over a 2048-token prompt
        _block("block_2048", 2048, 32, 128, 16384),
        # one OPT-1.3B-shaped decoder block over a short prompt whose length fills no tile
        _block("block_352", 352, 32, 64, 8192),
    ]


def _log(rng, lo, hi, step):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(max(int(v / step + 0.5) * step, -(-lo // step) * step), hi // step * step))


def draw(rng):
    kind = rng.choice(("layer", "layer", "layer", "stack", "quantize", "block"))
    if kind == "layer":
        block = rng.choice((16, 32))
        tokens = rng.choice((1, 2, 5, 16, _log(rng, 17, 512, 1), _log(rng, 128, 4096, 1), _log(rng, 128, 4096, 64)))
        K = _log(rng, 512, 16384, rng.choice((block, 128, 512)))
        while True:                      # at most the work of the largest listed layer, weights included
            N = _log(rng, 256, 16384, rng.choice((2, 32, 256)))
            if tokens * N * K <= 4096 * 11008 * 4096:
                break
            K = max(512, K // 2 // 512 * 512)
        w_act, w_wgt = rng.choice(synth.WIDTH_CHOICES), rng.choice(synth.WIDTH_CHOICES)
        if rng.random() < 0.4:
            w_act, w_wgt = rng.choice(((4, 4), (8, 4), (8, 8), (6, 6)))
        w_out = rng.choice((0, 0, 0, 4, 8)) if tokens > 16 and N % 32 == 0 else 0
        rows2 = rng.random() < 0.15 and tokens > 16 and tokens % 2 == 0 and w_out == 0
        return _layer(None, tokens, "%dx%d" % (K, N), block, w_act, w_wgt, dtype=rng.choice(("fp32", "bf16")),
                      acts=rng.choice(("gauss", "outlier", "heavy")), bias=rng.random() < 0.5, rows2=rows2, w_out=w_out)
    if kind == "stack":
        hidden, ffn = rng.choice(((768, 3072), (2048, 8192), (4096, 11008), (4096, 16384)))
        return _stack(None, rng.randint(1, 16), hidden, ffn, rng.randint(1, 8), w_act=rng.choice((4, 6, 8)),
                      w_wgt=rng.choice((2, 3, 4)), dtype=rng.choice(("fp32", "bf16")))
    if kind == "quantize":
        block = rng.choice((16, 32))
        along = rng.random() < 0.3
        rows, K = _log(rng, 16, 16384, 32 if along else 1), _log(rng, 256, 8192, 32)
        return _quantize(None, rows, K, block, rng.choice(synth.WIDTH_CHOICES), rng.choice(("fp32", "bf16")),
                         along, rng.random() < 0.5)
    heads, head_dim, ffn = rng.choice(((12, 64, 3072), (32, 64, 8192), (32, 128, 11008), (32, 128, 16384)))
    return _block(None, _log(rng, 64, 2048, 32), heads, head_dim, ffn, block=rng.choice((16, 32)),
                  w_act=rng.choice((4, 6, 8)), w_wgt=rng.choice((4, 4, 6, 8)))


# ---------------------------------------------------------------------------------------------------------

def _per_layer(case):
    shapes = [tuple(int(v) for v in s.split("x")) for s in case["layers"].split()]
    cols = [[int(v) for v in case[f].split()] for f in ("block", "w_act", "w_wgt")]
    return [(K, N) + tuple(c[i] if len(c) > 1 else c[0] for c in cols) for i, (K, N) in enumerate(shapes)]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _activations(g, rows, K, acts, dtype):
    x = torch.randn(rows, K, generator=g, device="cuda")
    if acts == "outlier":                # 0.5 % of the channels 40 times as large
        idx = torch.randperm(K, generator=g, device="cuda")[:max(1, K // 200)]
        x[:, idx] *= 40.0
    elif acts == "heavy":                # Student-t with 3 degrees of freedom
        chi2 = torch.zeros_like(x)
        for _ in range(3):
            chi2 += torch.randn(rows, K, generator=g, device="cuda") ** 2
        x /= torch.sqrt(chi2 / 3)
    return x.to(dtype)


def _weights(g, N, K, fmt):
    return mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fmt)


def prepare(case, seed):
    return {"layer": _prepare_layer, "stack": _prepare_stack, "quantize": _prepare_quantize,
            "block": _prepare_block}[case["kind"]](case, _generator(seed))


def run(state):
    return state["run"](state)


def _prepare_layer(case, g):
    layers, M = [], case["tokens"]
    rows2 = 2 if case["rows2"] else 1
    for K, N, block, w_act, w_wgt in _per_layer(case):
        fa, fw = mxb.MxFormat(block, w_act, block_rows=rows2), mxb.MxFormat(block, w_wgt, block_rows=rows2)
        wm, we = _weights(g, N, K, fw)
        L = dict(x=_activations(g, M, K, case["acts"], DTYPES[case["dtype"]]), fa=fa, fw=fw, N=N, wm=wm, we=we,
                 bias=torch.randn(N, generator=g, device="cuda") if case["bias"] else None,
                 ws=mxb.alloc_workspace(mxb.mx_workspace_bytes(M, N, K, fa, fw)))
        if case["w_out"]:
            fy = mxb.MxFormat(block, case["w_out"])
            L["fy"] = fy
            L["y_mant"] = torch.empty(M, N // 2 if fy.elem_bits <= 4 else N, dtype=torch.uint8, device="cuda")
            L["y_exp"] = torch.empty(M, N // block, dtype=torch.uint8, device="cuda")
        else:
            L["y"] = torch.empty(M, N, dtype=torch.float32, device="cuda")
        layers.append(L)
    return dict(run=_run_layer_q if case["w_out"] else _run_layer, layers=layers)


def _run_layer(state):
    return [mxb.mx_linear(L["x"], L["fa"], L["wm"], L["we"], L["fw"], L["N"], bias=L["bias"], y=L["y"], workspace=L["ws"])
            for L in state["layers"]]


def _run_layer_q(state):
    return [mxb.mx_linear_q(L["x"], L["fa"], L["wm"], L["we"], L["fw"], L["N"], L["fy"], bias=L["bias"],
                            y_mant=L["y_mant"], y_exp=L["y_exp"], workspace=L["ws"]) for L in state["layers"]]


def _stack_shapes(case):
    h, f = case["hidden"], case["ffn"]
    return [(h, h)] * 4 + [(h, f)] * 2


def _prepare_stack(case, g):
    fa, fw = mxb.MxFormat(32, case["w_act"]), mxb.MxFormat(32, case["w_wgt"])
    layers, T = [], case["tokens"]
    # the results of all matrices lie in one buffer, one decoder layer after the other
    ys = torch.empty(case["depth"], T * sum(N for _, N in _stack_shapes(case)), dtype=torch.float32, device="cuda")
    for d in range(case["depth"]):
        x, at = _activations(g, T, case["hidden"], "gauss", DTYPES[case["dtype"]]), 0
        for K, N in _stack_shapes(case):
            wm, we = _weights(g, N, K, fw)
            layers.append(dict(x=x, fa=fa, w_mant=wm, w_exp=we, fw=fw, N=N, y=ys[d, at:at + T * N].view(T, N)))
            at += T * N
    args = mxb.make_linear_args(layers)
    return dict(run=_run_stack, layers=layers, args=args, ys=ys,
                ws=mxb.alloc_workspace(mxb.mx_linear_grouped_workspace_bytes(args)))


def _run_stack(state):
    mxb.mx_linear_grouped(state["args"], workspace=state["ws"])
    return state["ys"]


def _prepare_quantize(case, g):
    x = _activations(g, case["rows"], case["K"], "outlier", DTYPES[case["dtype"]])
    return dict(run=_run_quantize, x=x.t() if case["along_rows"] else x, back=case["back"], dtype=x.dtype,
                f=mxb.MxFormat(case["block"], case["width"]))


def _run_quantize(state):
    mant, exps = mxb.mx_quantize(state["x"], state["f"])
    if not state["back"]:
        return mant, exps
    return mant, exps, mxb.mx_dequantize(mant, exps, state["x"].shape[1], state["f"], dtype=state["dtype"])


def _prepare_block(case, g):
    cfg = dblk.BlockConfig(hidden=case["heads"] * case["head_dim"], heads=case["heads"], head_dim=case["head_dim"],
                           ffn=case["ffn"], block=case["block"], w_act=case["w_act"], w_wgt=case["w_wgt"])
    h, f = cfg.hidden, cfg.ffn
    rnd = lambda *shape: torch.randn(*shape, generator=g, device="cuda")      # noqa: E731
    qweights = dblk.quantize_weights(cfg, {k: rnd(n, m) * 0.02 for k, n, m in (
        ("wq", h, h), ("wk", h, h), ("wv", h, h), ("wo", h, h), ("w1", f, h), ("w2", h, f))})
    params = {"ln1_g": 1 + 0.1 * rnd(h), "ln1_b": 0.1 * rnd(h), "ln2_g": 1 + 0.1 * rnd(h), "ln2_b": 0.1 * rnd(h)}
    params.update({b: 0.02 * rnd(f if b == "b1" else h) for b in ("bq", "bk", "bv", "bo", "b1", "b2")})
    return dict(run=_run_block, cfg=cfg, x=_activations(g, case["seq"], h, "outlier", torch.float32), qweights=qweights,
                params=dblk.prepare_params(params))


def _run_block(state):
    return dblk.run(state["cfg"], state["x"], state["qweights"], state["params"])


# ---------------------------------------------------------------------------------------------------------

def _packed(rows, K, block, width, block_rows=1):
    """Bytes of an MXInt tensor in its container."""
    return rows * K * (0.5 if width <= 4 else 1.0) + rows // block_rows * K / block


def work(case):
    size = {"fp32": 4, "bf16": 2}.get(case.get("dtype"), 4)
    if case["kind"] == "layer":
        M, nbytes, flops = case["tokens"], 0.0, 0.0
        rows2 = 2 if case["rows2"] else 1
        for K, N, block, _, w_wgt in _per_layer(case):
            nbytes += M * K * size + _packed(N, K, block, w_wgt, rows2) + (4 * N if case["bias"] else 0)
            nbytes += _packed(M, N, block, case["w_out"]) if case["w_out"] else 4 * M * N
            flops += 2.0 * M * N * K
        return {"bytes": nbytes, "flops": flops}
    if case["kind"] == "stack":
        T, nbytes, flops = case["tokens"], 0.0, 0.0
        for K, N in _stack_shapes(case):
            nbytes += _packed(N, K, 32, case["w_wgt"]) + 4 * T * N
            flops += 2.0 * T * N * K
        return {"bytes": case["depth"] * (nbytes + T * case["hidden"] * size), "flops": case["depth"] * flops}
    if case["kind"] == "quantize":
        n, codes = case["rows"] * case["K"], _packed(case["rows"], case["K"], case["block"], case["width"])
        return {"bytes": n * size + codes + (codes + n * size if case["back"] else 0), "flops": 0.0}
    h, f, S = case["heads"] * case["head_dim"], case["ffn"], case["seq"]
    weights = sum(_packed(n, m, case["block"], case["w_wgt"]) for n, m in ((4 * h, h), (f, h), (h, f)))
    flops = 2.0 * S * (4 * h * h + 2 * h * f) + 2 * 2.0 * case["heads"] * case["head_dim"] * S * (S + 1) / 2
    return {"bytes": 2 * 4.0 * S * h + weights, "flops": flops}


def tolerance(case):
    if case["kind"] == "quantize":
        return "exact"                   # codes, exponent bytes and decoded values are defined bit by bit
    if case["kind"] == "block":
        # The attention probabilities and the feed-forward activation are quantized inside: an fp32 value next to a
        # rounding boundary may take either code.  The fused sequence against the one that stores every intermediate
        # differs by 1.0e-3 of the norm (largest difference 0.022 of the rms) at 6- and 8-bit activations and by
        # 3.4e-3 (0.27) at 4-bit ones.
        return {"rel": 4e-3, "max": 0.1} if case["w_act"] >= 6 else {"rel": 1.4e-2, "max": 0.9}
    if case["kind"] == "layer" and case["w_out"]:
        return {"rel": 0.0, "differ": 1e-5}      # no code differed from the 64-bit product's
    # fp32 sums of exact products against the 64-bit product over 80 layers of these ranges: 0 without a bias, 2.7e-8 of
    # the norm (6.0e-8 of a value) with one
    return {"rel": 2e-7, "max": 1e-6}
