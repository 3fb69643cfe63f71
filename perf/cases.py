"""Performance cases of the sparse linear attention library: what a program that uses it has it do, through the public
entry points of ``paper_2605_11354_b200.binding``.

Four kinds of case:

``attention``  the attention forward of one layer (``SlaForward.run`` or its graph replay ``run_graph``): quantise
               Q, K, V, classify the block pairs, forward.
``layer``      a whole attention layer in its deployed FP8 form: activations quantised per token, qkv projection
               with the block quantiser in its epilogue, plan, forward, output re-quantised, out-projection.
``train``      one distillation step of a module: forward, linear branch alone, MSE term with its gradient, gradient
               of the linear branch's projection.
``linear``     one FP8 linear layer: per-token quantiser and GEMM (weights are quantised once, offline).

Queries and keys follow the clustered recipe of ``workloads.py`` (token positions tied to cluster centres that all
frames share, plus noise); values, weights and biases are Gaussian.
"""
import math

import torch

from paper_2605_11354_b200 import binding as lt
from paper_2605_11354_b200 import workloads as wk

FRAME = wk.TOKENS_PER_FRAME
D = 64
FLOAT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}
# Bounds of a drawn case: the token rows and the critical (query, key) pairs of the largest listed one.
MOST_ROWS = 16 * 100 * FRAME
MOST_PAIRS = 0.10 * 16 * (100.0 * FRAME) ** 2
MOST_LAYER_ROWS = 32 * FRAME


def attention(name, batch, heads, tokens, block, crit, neg, src="bf16", out="f32", phi="softmax", layout="heads",
              call="run", plan_inside=False):
    """layout "heads": contiguous [B, H, N, 64] tensors; "tokens": Q, K, V are views of one packed [B, N, 3, H, 64]
    projection output and the result is written token-major, as a transformer layer holds them."""
    return {"name": name, "kind": "attention", "batch": batch, "heads": heads, "tokens": tokens, "block": block,
            "crit": crit, "neg": neg, "src": src, "out": out, "phi": phi, "layout": layout, "call": call,
            "plan_inside": plan_inside}


def listed():
    return [
        # the smallest configuration: two heads of 512 fp32 tokens, called eagerly; launches and host work decide
        attention("tiny", 1, 2, 512, 64, 0.25, 0.50, src="f32"),
        # one frame through one eager layer, the latency of single-image inference, token-major bf16 tensors
        attention("frame1", 1, 16, FRAME, 64, 0.25, 0.50, out="bf16", layout="tokens"),
        # odd sizes and the other options: block 128, ELU+1 feature map, fp32 in, fp16 out, block plan made inside the
        # forward's workspace
        attention("odd_elu", 3, 5, 3001, 128, 0.15, 0.55, src="f32", out="f16", phi="elu1", plan_inside=True),
        # global attention over eight frames replayed as a graph: the benchmark's default
        attention("vggt8", 1, 16, 8 * FRAME, 64, 0.10, 0.60, call="graph"),
        # frame attention: 32 short sequences
        attention("frame32", 32, 16, FRAME, 64, 0.25, 0.50, out="bf16", layout="tokens"),
        # global attention over 32 frames
        attention("vggt32", 1, 16, 32 * FRAME, 64, 0.05, 0.75, call="graph"),
        # four scenes of 16 views in blocks of 128 tokens
        attention("da3l", 4, 16, 16 * FRAME, 128, 0.08, 0.70, out="bf16"),
        # the longest sequence: a hundred frames
        attention("stress100", 1, 16, 100 * FRAME, 64, 0.10, 0.60),
        # a whole attention layer of ViT-L width on one frame (small, many launches) and on eight
        {"name": "layer1", "kind": "layer", "batch": 1, "heads": 16, "tokens": FRAME, "block": 64, "crit": 0.25, "neg": 0.50},
        {"name": "layer8", "kind": "layer", "batch": 1, "heads": 16, "tokens": 8 * FRAME, "block": 64, "crit": 0.10, "neg": 0.60},
        # a distillation step of one module on eight frames (forward and backward of the linear branch's projection)
        {"name": "train8", "kind": "train", "batch": 1, "heads": 16, "tokens": 8 * FRAME, "block": 64, "crit": 0.10,
         "neg": 0.60, "src": "bf16"},
        # the out-projection of 32 frames
        {"name": "linear32", "kind": "linear", "rows": 32 * FRAME, "d_in": 1024, "d_out": 1024, "src": "bf16", "out": "bf16"},
    ]


def _spread(rng, low, high):
    """A whole number between low and high, spread over their logarithm."""
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _tokens(rng, low, high):
    n = _spread(rng, low, high)
    return max(1, n // FRAME) * FRAME if n > FRAME and rng.random() < 0.4 else n


def draw(rng):
    kind = rng.choice(["attention"] * 8 + ["layer", "layer", "train", "linear"])
    if kind == "linear":
        return {"kind": "linear", "rows": _spread(rng, 300, 32 * FRAME), "d_in": 128 * rng.randint(4, 16),
                "d_out": 64 * rng.randint(8, 48), "src": rng.choice(["bf16", "bf16", "f32"]),
                "out": rng.choice(["bf16", "bf16", "f16", "f32"])}
    block = rng.choice([64, 64, 128])
    crit, neg = rng.choice([(0.25, 0.50), (0.10, 0.60), (0.05, 0.75), (0.08, 0.70), (0.05, 0.60), (0.15, 0.55)])
    if kind != "attention":
        case = {"kind": kind, "batch": rng.choice([1, 1, 2]), "heads": rng.choice([4, 8, 12, 16]),
                "tokens": _tokens(rng, 500, 16 * FRAME), "block": block, "crit": crit, "neg": neg}
        if kind == "train":
            case["src"] = rng.choice(["bf16", "bf16", "f32"])
        while case["batch"] * case["tokens"] > MOST_LAYER_ROWS:
            case["tokens"] = case["tokens"] // 2
        return case
    while True:
        batch, heads = rng.choice([1, 1, 1, 2, 4, 8, 32]), rng.choice([2, 5, 8, 12, 16, 16, 16])
        tokens = _tokens(rng, 300, 100 * FRAME)
        if batch * heads * tokens <= MOST_ROWS and crit * batch * heads * float(tokens) ** 2 <= MOST_PAIRS:
            break
    case = attention("", batch, heads, tokens, block, crit, neg, src=rng.choice(["bf16", "bf16", "bf16", "f32"]),
                     out=rng.choice(["f32", "bf16", "bf16", "f16"]), phi=rng.choice(["softmax", "softmax", "elu1"]),
                     layout=rng.choice(["heads", "tokens"]), call=rng.choice(["run", "graph"]),
                     plan_inside=rng.random() < 0.25)
    if case["plan_inside"]:
        case["call"] = "run"
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------------ preparation
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, shape, dtype=torch.float32):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _positions(tokens, centres):
    return torch.from_numpy(wk.centre_of_token(tokens, centres)).cuda()


def _sources(g, case):
    """Q, K, V as views [B, H, N, 64] in the case's type and layout."""
    B, H, N = case["batch"], case["heads"], case["tokens"]
    dtype = FLOAT[case["src"]]
    at = _positions(N, 64)
    centres = _normal(g, (H, 64, D), dtype)
    if case.get("layout", "heads") == "tokens":
        packed = _normal(g, (B, N, 3, H, D), dtype)
        parts = [packed[:, :, i].permute(0, 2, 1, 3) for i in range(3)]
    else:
        parts = [_normal(g, (B, H, N, D), dtype) for _ in range(3)]
    for x in parts[:2]:
        x.mul_(0.3).add_(centres[:, at][None])
    return parts


def _weight(g, d_out, d_in):
    return lt.lite3r_quantize_rows_fp8(_normal(g, (d_out, d_in)) / math.sqrt(d_in))


def _engine(case, out="bf16"):
    return lt.SlaForward(case["batch"], case["heads"], case["tokens"], case["block"], case["crit"], case["neg"],
                         phi=case.get("phi", "softmax"), out_dtype=FLOAT[out],
                         plan_inside=case.get("plan_inside", False))


def _projection(g, heads):
    return _normal(g, (heads, D, D)) / 8.0


def _token_major(case, out):
    """Output buffer [B, N, H * 64] and its [B, H, N, 64] view."""
    buf = torch.empty((case["batch"], case["tokens"], case["heads"], D), dtype=FLOAT[out], device="cuda")
    return buf, buf.permute(0, 2, 1, 3)


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "linear":
        scale = torch.exp(0.5 * _normal(g, (case["rows"], 1)))  # tokens differ in magnitude
        s["x"] = (_normal(g, (case["rows"], case["d_in"])) * scale).to(FLOAT[case["src"]])
        s["w"] = _weight(g, case["d_out"], case["d_in"])
        s["bias"] = 0.1 * _normal(g, (case["d_out"],))
        s["y"] = torch.empty((case["rows"], case["d_out"]), dtype=FLOAT[case["out"]], device="cuda")
        s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s
    B, H, N = case["batch"], case["heads"], case["tokens"]
    s["proj"] = _projection(g, H)
    if kind == "attention":
        s["qkv"] = _sources(g, case)
        s["engine"] = _engine(case, case["out"])
        s["graph"] = case["call"] == "graph"
        s["out"] = _token_major(case, case["out"])[1] if case["layout"] == "tokens" else None
    elif kind == "layer":
        d = H * D
        x = _normal(g, (B, N, d)) * 0.3 + _normal(g, (64, d))[_positions(N, 64)]
        s["x"] = x.to(torch.bfloat16).view(B * N, d)
        s["w_qkv"], s["w_out"] = _weight(g, 3 * d, d), _weight(g, d, d)
        s["b_qkv"], s["b_out"] = 0.1 * _normal(g, (3 * d,)), 0.1 * _normal(g, (d,))
        s["engine"] = _engine(case)
        buf, s["out"] = _token_major(case, "bf16")
        s["rows"] = buf.view(B * N, d)
        s["y"] = torch.empty((B * N, d), dtype=torch.bfloat16, device="cuda")
    else:
        s["qkv"] = _sources(g, case)
        s["engine"] = _engine(case, "f32")
        s["teacher"] = 0.2 * _normal(g, (B, H, N, D))  # the size of an attention output
        shape = s["engine"].shape
        nbytes = lt.lite3r_train_workspace(shape, case["crit"], case["neg"])
        raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        s["workspace"] = raw[(-raw.data_ptr()) % 256:][:nbytes]
        s["o_lin"] = torch.empty((B, H, N, D), dtype=torch.bfloat16, device="cuda")
        s["grad"] = torch.empty((B, H, N, D), dtype=torch.bfloat16, device="cuda")
        s["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["d_proj"] = torch.empty((H, D, D), device="cuda")
    return s


# ------------------------------------------------------------------------------------------------------ one pass
def run(s):
    kind = s["kind"]
    if kind == "linear":
        codes, scales = lt.lite3r_quantize_rows_fp8(s["x"])
        lt.lite3r_linear_fp8(codes, scales, *s["w"], s["bias"], s["y"], s["status"])
        return {"codes": codes, "scales": scales, "y": s["y"]}
    eng = s["engine"]
    if kind == "attention":
        step = eng.run_graph if s["graph"] else eng.run
        out = step(*s["qkv"], s["proj"], out=s["out"])
        return {"out": out} if eng.plan_inside else {"out": out, "classes": eng.plan.cls}
    if kind == "layer":
        codes, scales = lt.lite3r_quantize_rows_fp8(s["x"])
        lt.lite3r_qkv_project_fp8(codes, scales, *s["w_qkv"], s["b_qkv"], eng.shape, eng.q8, eng.k8, eng.v8, eng.status)
        eng.make_plan()
        eng.forward(s["proj"], out=s["out"])
        codes, scales = lt.lite3r_quantize_rows_fp8(s["rows"])
        lt.lite3r_linear_fp8(codes, scales, *s["w_out"], s["b_out"], s["y"], eng.status)
        return {"attention": s["rows"], "y": s["y"]}
    out = eng.run(*s["qkv"], s["proj"])
    lt.lite3r_sla_linear_branch(eng.q8, eng.k8, eng.v8, eng.shape, eng.phi, eng.plan, s["o_lin"], s["workspace"], eng.status)
    lt.lite3r_mse_distill(out, s["teacher"], s["grad"], s["loss"], s["workspace"])
    lt.lite3r_proj_lin_backward(s["o_lin"], s["grad"], eng.shape, s["d_proj"], s["workspace"], eng.status)
    return {"out": out, "o_lin": s["o_lin"], "grad": s["grad"], "loss": s["loss"], "d_proj": s["d_proj"]}


# ------------------------------------------------------------------------------------------------------ what it takes
def _counts(case):
    nb = -(-case["tokens"] // case["block"])
    crit = min(nb, max(1, math.floor(case["crit"] * nb + 0.5)))
    return nb, crit, nb - crit - min(nb - crit, math.floor(case["neg"] * nb + 0.5))


def _attention_flops(case):
    """Pooled scores, critical pairs (Q K^T and P V), key-block summaries, their sums over the marginal blocks, linear
    output."""
    nb, crit, marg = _counts(case)
    bs, tiles = case["block"], case["batch"] * case["heads"] * nb
    return tiles * (2.0 * nb * D + crit * 4.0 * bs * bs * D + 2.0 * (bs + D) * D * D + marg * (D * D + D) + 2.0 * bs * D * D)


def work(case):
    kind = case["kind"]
    if kind == "linear":
        r, i, o = case["rows"], case["d_in"], case["d_out"]
        return {"bytes": r * i * (BYTES[case["src"]] + 1) + 4 * r + o * i + 8 * o + r * o * BYTES[case["out"]], "flops": 2.0 * r * i * o}
    B, H, N = case["batch"], case["heads"], case["tokens"]
    values, nb = B * H * N * D, _counts(case)[0]
    flops, proj = _attention_flops(case), 4 * H * D * D
    if kind == "attention":
        classes = 0 if case["plan_inside"] else B * H * nb * nb
        return {"bytes": values * (3 * BYTES[case["src"]] + BYTES[case["out"]]) + proj + classes, "flops": flops}
    if kind == "layer":
        d = H * D
        return {"bytes": 3 * 2 * values + 4 * d * d + 32 * d + proj, "flops": flops + 8.0 * B * N * d * d}
    return {"bytes": values * (3 * BYTES[case["src"]] + 4 + 4 + 2 + 2) + 2 * proj + 8,
            "flops": flops + 4.0 * B * H * N * D * D + 3.0 * values}


def tolerance(case):
    """The attention's intermediates are 16-bit (probabilities fp16, summaries bf16): 2e-3 relative is the library's
    stated bound; bf16 results add their own rounding.  Integer results are exact."""
    kind = case["kind"]
    if kind == "linear":
        # exact products; only the order of the fp32 sums differs, and with it now and then the rounding of the result
        return {"rel": {"f32": 1e-5, "f16": 2e-4, "bf16": 1e-3}[case["out"]], "max": 1e-4 if case["out"] == "f32" else 1e-2}
    if kind == "attention":
        return {"rel": {"f32": 2e-3, "f16": 2e-3, "bf16": 4e-3}[case["out"]]}
    # a layer re-quantises its attention output to e4m3 (a value at a rounding boundary moves by 2^-4); a training step
    # rounds the gradient and the linear branch to bf16
    return {"rel": 1e-2 if kind == "layer" else 4e-3}
