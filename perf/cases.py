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


def _inputs(c, seed):
    """The tensors of a case, from the seed alone: activations, weights, biases and whatever else its call takes."""
    M, K, N = c["M"], c["K"], c["N"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n = c.get("products", 1)
    t = {"X": _activations(c, g), "residual": None}
    t["W"] = [_normal((N, K), K ** -0.5, g) for _ in range(n)]
    t["bias"] = [_normal((N,), 0.01, g) for _ in range(n)]
    if c.get("residual"):
        t["residual"] = _normal((M, N), 0.05, g)
    if c["op"] == "lora":
        t["LB"], t["LA"] = _normal((c["rank"], K), K ** -0.5, g), _normal((N, c["rank"]), 0.3 * c["rank"] ** -0.5, g)
    return t


def prepare(case, seed):
    c, op = case, case["op"]
    lx = _context()
    lx.reserve(c["M"], c["N"], c["K"])
    s = dict(_inputs(c, seed), op=op, lx=lx, mode=MODES[c["mode"]])
    if op == "lora":
        lx.reserve_lora(c["M"], c["K"], c["rank"])
    elif op == "fp8":
        s["Wq"], s["wscale"] = lx.quantize_weights_fp8(s.pop("W")[0], per_channel=True)
    elif op == "host":
        s["X"] = s["X"].cpu().pin_memory()
        s["Y"] = torch.empty(c["M"], c["N"], dtype=torch.bfloat16, pin_memory=True)
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


def _keep_mask(X):
    """The two of each four elements of largest magnitude, of equal ones the first (a stable sort keeps their order)."""
    order = X.abs().reshape(-1, 4).sort(dim=1, descending=True, stable=True).indices
    return torch.zeros_like(order, dtype=torch.bool).scatter_(1, order[:, :2], True)


def _e4m3(x):
    return x.clamp(-448.0, 448.0).to(torch.float8_e4m3fn).double()


def exact(case, seed):
    """What run() returns, in 64 bits.  The FP8 codes are part of the layer's definition (fp32 rule, E4M3 result) and are
    made as it says; everything behind them, and every other case throughout, is in 64 bits and never rounded."""
    c = case
    t = _inputs(c, seed)
    X, M = t["X"].float(), c["M"]
    mask = _keep_mask(X)
    groups = X.double().reshape(-1, 4)
    kept = groups * mask
    scale = None
    if c["mode"] == "row":
        num, den = groups.square().reshape(M, -1).sum(1), kept.square().reshape(M, -1).sum(1)
        scale = (num / (den + 1e-8)).sqrt()
    elif c["mode"] == "tensor":
        scale = (groups.square().sum() / (kept.square().sum() + 1e-8)).sqrt().expand(M)
    elif c["mode"] == "group":
        kept = kept * (groups.square().sum(1, keepdim=True) / (kept.square().sum(1, keepdim=True) + 1e-8)).sqrt()
    values = kept[mask].reshape(M, -1) if c["op"] == "shared" else None
    kept, weights = kept.reshape(M, -1), [w.double() for w in t["W"]]
    if c["op"] == "fp8":
        amax = X.abs().amax(1, keepdim=True)
        kept = _e4m3(kept.float() * torch.where(amax > 0, 448.0 / amax, 0.0)) * (amax.double() / 448.0)
        W = t["W"][0].float()
        wmax = W.abs().amax(1, keepdim=True)
        weights = [_e4m3(W * torch.where(wmax > 0, 448.0 / wmax, 0.0)) * (wmax.double() / 448.0)]
    results = []
    for W, b in zip(weights, t["bias"]):
        Y = kept @ W.T
        if scale is not None:
            Y *= scale[:, None]
        Y += b.double()
        if c["op"] == "lora":
            Y += (X.double() @ t["LB"].double().T) @ t["LA"].double().T
        if t["residual"] is not None:
            Y += t["residual"].double()
        results.append(Y)
    if c["op"] == "shared":
        return [values, None, scale] + results  # (the metadata is whole numbers)
    return results[0].cpu() if c["op"] == "host" else results[0]


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
