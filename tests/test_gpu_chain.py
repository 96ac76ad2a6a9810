"""Layers queued one behind the other without a synchronisation: a launch's CTAs may be placed while the launch that writes their X,
W, residual or bias still runs.  Every result is compared bit for bit with that of a context whose launches never overlap."""
import pytest
import torch

from paper_2605_26632_b200 import binding, inputs

pytestmark = pytest.mark.gpu

ROUNDS = 3
# name: M, K, call, overrides.  The split kernel lets the next launch begin at once where a quarter of the SMs stay free:
# tiles of 256 x 128 in two splits are 4 * ceil(K / 128) CTAs per 256 rows.
KINDS = {
    "split, next begins early": (200, 2048, "plain", {"LYNX_SPLIT": "12"}),
    "split, most SMs held": (300, 2560, "plain", {"LYNX_SPLIT": "12"}),
    "one tile": (300, 2048, "plain", {"LYNX_SPLIT": "0", "LYNX_RT2": "0"}),
    "two row tiles": (1100, 1024, "plain", {"LYNX_SPLIT": "0", "LYNX_RT2": "1"}),
    "none": (200, 2048, "none", {}),
    "tensor": (200, 2048, "tensor", {}),
    "tensor, one tile": (1100, 1024, "tensor", {"LYNX_SPLIT": "0", "LYNX_RT2": "0"}),
    "own calls": (200, 2048, "calls", {"LYNX_SPLIT": "12"}),
    "lora": (300, 2048, "lora", {"LYNX_SPLIT": "0", "LYNX_RT2": "0"}),
    "lora, split": (200, 2048, "lora", {"LYNX_SPLIT": "13"}),
    "fp8, rows in blocks of 16": (300, 1536, "fp8", {"LYNX_SPLIT": "0", "LYNX_RT2": "0"}),
    "fp8, a row at a time": (300, 2304, "fp8", {"LYNX_SPLIT": "0", "LYNX_RT2": "0"}),
    "fp8, split": (200, 2304, "fp8", {"LYNX_SPLIT": "12"}),
    "fp8, two row tiles": (1100, 1536, "fp8", {"LYNX_SPLIT": "0", "LYNX_RT2": "1"}),
}


def _layer(c, call, t, X, W, bias=None, residual=None, out=None):
    if call == "lora":
        return c.act_sparse_linear_lora(X, W, t["LA"], t["LB"], bias, binding.COMP_ROW, residual, out)
    if call == "fp8":
        codes = c.quantize_weights_fp8(W) if torch.is_tensor(W) else W  # (codes made here: that launch overlaps with nothing)
        return c.act_sparse_linear_fp8(X, *codes, bias, binding.COMP_ROW, residual, out)
    if call == "calls":
        values, meta, scale = c.prune_compress(X, binding.COMP_ROW)
        return c.sparse_linear(values, meta, W, bias, scale, residual, out)
    mode = {"plain": binding.COMP_ROW, "none": binding.COMP_NONE, "tensor": binding.COMP_TENSOR}[call]
    return c.act_sparse_linear(X, W, bias, mode, residual, out)


def _chain(c, call, t, streams):
    """`streams`: a buffer per round, which a layer adds to in place."""
    kept, h = [], t["X"]
    W = [c.quantize_weights_fp8(w) for w in t["W"]] if call == "fp8" else t["W"]
    for i, stream in enumerate(streams):
        a = _layer(c, call, t, h, W[i % 2], t["bias"])                            # the last round's result is X
        b = _layer(c, call, t, t["other"], W[1 - i % 2])                          # another X and another number of rows
        _layer(c, call, t, a, W[0], residual=stream, out=stream)                  # in place, as a residual stream is kept
        w = _layer(c, call, t, t["tall"], W[1])                                   # K rows: the next layer's W
        d = _layer(c, call, t, stream, w, b[0])                                   # X, W and bias are all results
        h = _layer(c, call, t, d, W[i % 2], residual=a)
        kept += [a, b, stream, w, d, h]
    return kept


@pytest.mark.parametrize("kind", KINDS)
def test_chain(kind, monkeypatch):
    m, k, call, env = KINDS[kind]
    t = {"X": inputs.make_x(m, k, "outlier", 31), "other": inputs.make_x(m // 3, k, "gelu", 32), "tall": inputs.make_x(k, k, "gelu", 33),
         "bias": inputs.make_bias(k, 34)}
    t = {n: v.cuda() for n, v in t.items()}
    t["tall"] *= k ** -0.5  # (its product is a W)
    t["W"] = [inputs.make_w(k, k, 35 + i).cuda() for i in range(2)]
    t["LA"], t["LB"] = (v.cuda() for v in inputs.make_lora(k, k, 64, 37))
    start = inputs.make_residual(m, k, 38).cuda()
    for name, value in env.items():
        monkeypatch.setenv(name, value)
    got = []
    for overlap in ("0", "1"):
        monkeypatch.setenv("LYNX_PDL", overlap)
        c = binding.Lynx(0)
        c.reserve(k, k, k)
        c.reserve_lora(k, k, 64)
        torch.cuda.synchronize()
        for _ in range(1 if overlap == "0" else 3):  # (the first pass loads the kernels one by one)
            streams = [start.clone() for _ in range(ROUNDS)]
            torch.cuda.synchronize()
            got.append(_chain(c, call, t, streams))
            torch.cuda.synchronize()
        assert c.last_error() == 0
        c.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert bool(x.isfinite().all()) and torch.equal(x, y)
