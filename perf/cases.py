"""The work this library is used for, as timed cases: linear layers of a diffusion transformer's blocks, called
through the Python binding on activations that change from call to call while weights stay.

A case is a dict of plain values:
  op    "layer"   one whole layer on device tensors                         Lynx.act_sparse_linear
        "shared"  one pruning shared by several products (separate Q, K, V) Lynx.prune_compress + Lynx.sparse_linear
        "lora"    the layer with its low-rank branch                        Lynx.act_sparse_linear_lora
        "fp8"     the layer on E4M3 operands, weights quantised beforehand  Lynx.act_sparse_linear_fp8
        "host"    activations and result in pinned host memory              Lynx.act_sparse_linear_host
  M, K, N         tokens, input and output width (of each product)
  mode            norm compensation: "none", "row" (what a program uses unless it has a reason), "tensor", "group"
  dist            the activations: "outlier" (a few large channels, what attention and MLP-up inputs look like) or
                  "gelu" (GELU output with per-channel gains, what MLP-down inputs look like)
  products        number of products of "shared";  rank: of "lora";  residual: with the M x N addend or without
"""
import math

import torch

from paper_2605_26632_b200 import binding, inputs

MODES = {"none": binding.COMP_NONE, "row": binding.COMP_ROW, "tensor": binding.COMP_TENSOR, "group": binding.COMP_GROUP}


def _case(op, M, K, N, mode="row", dist="outlier", **more):
    return dict({"op": op, "M": M, "K": K, "N": N, "mode": mode, "dist": dist}, **more)


def listed():
    w = inputs.WORKLOADS
    tiny, down, qkv, out, up = (w[n] for n in ("tiny", "mlp_down", "attn_qkv", "attn_out", "mlp_up"))
    cases = {
        # the smallest call: launches and host work are all there is
        "tiny": _case("layer", tiny.M, tiny.K, tiny.N, dist="gelu"),
        # the text tokens' own projection in a double-stream block: 256 rows, one row tile
        "text_tokens_out": _case("layer", 256, out.K, out.N),
        # output projection of a small image (512 x 512 pixels), added to a residual stream
        "small_image_out_residual": _case("layer", 1024, out.K, out.N, residual=True),
        # Q, K and V kept as separate weights: one pruning, three products
        "qkv_shared_pruning": _case("shared", qkv.M, qkv.K, 3072, products=3),
        # fused QKV of a 1024 x 1024 image with its text tokens
        "attn_qkv": _case("layer", qkv.M, qkv.K, qkv.N),
        # MLP up projection without compensation (the plain activation-sparse layer)
        "mlp_up": _case("layer", up.M, up.K, up.N, mode="none"),
        # MLP down projection: the headline shape
        "mlp_down": _case("layer", down.M, down.K, down.N, dist="gelu"),
        # another model's widths and a ragged number of tokens: no size is a multiple of a tile
        "ragged_tokens_up": _case("layer", 1337, 3840, 10240),
        # a 2048 x 2048 image: the largest layer
        "large_image_down": _case("layer", 16384, down.K, down.N, dist="gelu"),
        # output projection with a rank-64 low-rank branch
        "attn_out_lora": _case("lora", out.M, out.K, out.N, rank=64),
        # MLP down projection on FP8 operands
        "mlp_down_fp8": _case("fp8", down.M, down.K, down.N, dist="gelu"),
        # the same layer called with host buffers, end to end
        "mlp_down_host": _case("host", down.M, down.K, down.N, dist="gelu"),
    }
    return [dict(c, name=n) for n, c in cases.items()]


# a drawn case costs no more than the largest listed one
_MOST_MNK = 16384 * 12288 * 3072
_MOST_HOST_ELEMS = 4096 * (12288 + 3072)
_WIDTHS = inputs.SWEEP_KN + inputs.OTHER_FAMILY_KN


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["layer"] * 5 + ["lora"] * 2 + ["fp8"] * 2 + ["shared", "host"])
    M = _spread(rng, 64, 16384)
    if rng.random() < 0.5:  # widths of the models the repository names, or any that the layer takes
        K, N = rng.choice(_WIDTHS)
    else:
        K, N = 256 * _spread(rng, 2, 64), 8 * _spread(rng, 32, 2688)
    products = rng.choice([2, 3]) if op == "shared" else 1
    M = min(M, _MOST_MNK // (K * N * products))
    more = {}
    if op == "host":
        M = min(M, _MOST_HOST_ELEMS // (K + N))
    elif op == "shared":
        more["products"] = products
    elif op == "lora":
        more["rank"] = rng.choice([64, 64, 128])
    modes = ["row"] * 6 + ["none"] * 3
    if op in ("layer", "shared"):
        modes += ["group", "tensor"]
    if op in ("layer", "fp8") and rng.random() < 0.3:
        more["residual"] = True
    return _case(op, M, K, N, rng.choice(modes), rng.choice(["outlier", "gelu"]), **more)


# ------------------------------------------------------------------------------------ state ----

_contexts = {}


def _context():
    """One library context for the process, as a program with one stream keeps it."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = binding.Lynx(dev)
    return _contexts[dev]


def _activations(c, g):
    x = torch.randn(c["M"], c["K"], device="cuda", generator=g)
    if c["dist"] == "gelu":
        x = torch.nn.functional.gelu(x) * torch.exp(0.5 * torch.randn(c["K"], device="cuda", generator=g))
    else:
        x[:, torch.randperm(c["K"], device="cuda", generator=g)[: c["K"] // 100]] *= 20.0
    return x.to(torch.bfloat16)


def _normal(shape, std, g):
    return (torch.randn(*shape, device="cuda", generator=g) * std).to(torch.bfloat16)


def prepare(case, seed):
    c = case
    M, K, N, op = c["M"], c["K"], c["N"], c["op"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    lx = _context()
    lx.reserve(M, N, K)
    s = {"op": op, "lx": lx, "mode": MODES[c["mode"]], "X": _activations(c, g), "residual": None}
    n = c.get("products", 1)
    s["W"] = [_normal((N, K), K ** -0.5, g) for _ in range(n)]
    s["bias"] = [_normal((N,), 0.01, g) for _ in range(n)]
    if c.get("residual"):
        s["residual"] = _normal((M, N), 0.05, g)
    if op == "lora":
        lx.reserve_lora(M, K, c["rank"])
        s["LB"], s["LA"] = _normal((c["rank"], K), K ** -0.5, g), _normal((N, c["rank"]), 0.3 * c["rank"] ** -0.5, g)
    elif op == "fp8":
        s["Wq"], s["wscale"] = lx.quantize_weights_fp8(s.pop("W")[0], per_channel=True)
    elif op == "host":
        s["X"] = s["X"].cpu().pin_memory()
        s["Y"] = torch.empty(M, N, dtype=torch.bfloat16, pin_memory=True)
    return s


def run(state):
    s, lx = state, state["lx"]
    if s["op"] == "layer":
        return lx.act_sparse_linear(s["X"], s["W"][0], s["bias"][0], s["mode"], s["residual"])
    if s["op"] == "shared":
        values, meta, scale = lx.prune_compress(s["X"], s["mode"])
        return [values, meta, scale] + [lx.sparse_linear(values, meta, W, b, scale) for W, b in zip(s["W"], s["bias"])]
    if s["op"] == "lora":
        return lx.act_sparse_linear_lora(s["X"], s["W"][0], s["LA"], s["LB"], s["bias"][0], s["mode"])
    if s["op"] == "fp8":
        return lx.act_sparse_linear_fp8(s["X"], s["Wq"], s["wscale"], s["bias"][0], s["mode"], s["residual"])
    return lx.act_sparse_linear_host(s["X"], s["W"][0], s["bias"][0], s["mode"], s["Y"])


def work(case):
    """Multiply-adds of the kept half of X only (2 flops each), and each input and output once."""
    c = case
    M, K, N, n, R = c["M"], c["K"], c["N"], c.get("products", 1), c.get("rank", 0)
    weight = 1 if c["op"] == "fp8" else 2
    b = 2 * M * K + n * (weight * N * K + 2 * N + 2 * M * N)
    if c.get("residual"):
        b += 2 * M * N
    if c["op"] == "shared":
        b += M * K + M * K // 8 + 4 * M  # values, metadata and scale are results too
    return {"bytes": b + 2 * R * (K + N), "flops": n * M * N * K + 2 * M * R * (K + N)}


def tolerance(case):
    """bf16 results of fp32 sums: another order of additions moves a result by one bf16 step (2^-8 of itself) now and
    then.  Measured against the same products summed in 64 bits and rounded to bf16: rel 2e-4, max 7.8e-3; with a
    low-rank branch, whose intermediate is rounded to bf16, rel 1.3e-3, max 7.8e-3.  On FP8 operands the accumulation
    inside the tensor core is coarser than fp32: rel 2.2e-3, max 8.4e-2 at K = 12288.  About four times that."""
    if case["op"] == "fp8":
        return {"rel": 9e-3, "max": 0.3, "differ": 0.0}
    if case["op"] == "lora":
        return {"rel": 5e-3, "max": 3e-2, "differ": 0.0}
    return {"rel": 8e-4, "max": 3e-2, "differ": 0.0}
