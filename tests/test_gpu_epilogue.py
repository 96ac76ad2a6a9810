"""GPU tests of the GEMM epilogue where tiles follow one another on a CTA pair: staging boxes that are used again (16- and
32-row ones), the last tile staged in the ring, ragged rows and columns, with and without bias and residual."""
import pytest
import torch

from paper_2605_26632_b200 import inputs

pytestmark = pytest.mark.gpu


def _reference(X, W, bias, residual):
    """The layer without compensation in fp64, and the bound of a correct bf16 result around it: half a bf16 step of the
    result (2^-9 relative) and of what a carry into the next binade adds (another 2^-9), plus fp32 sums of K terms
    (K 2^-24 of the sum of magnitudes)."""
    g = X.double().reshape(-1, 4)
    order = g.abs().sort(dim=1, descending=True, stable=True).indices
    kept = (g * torch.zeros_like(g).scatter_(1, order[:, :2], 1.0)).reshape(X.shape)
    ref, mag = kept @ W.double().T, kept.abs() @ W.double().abs().T
    for addend in (bias, residual):
        if addend is not None:
            ref, mag = ref + addend.double(), mag + addend.double().abs()
    return ref, ref.abs() * 2.0 ** -8 + mag * (X.shape[1] * 2.0 ** -24)


# M and N ragged, over two tiles per CTA pair (one-CTA tiles: per CTA) in every configuration; the last column tile is
# narrower than one epilogue chunk for 48- and 64-column chunks
M, K, N = 2570, 256, 6160


@pytest.fixture(scope="module")
def data():
    d = inputs.make_workload(inputs.Workload("t", M, K, N, "outlier", 91), with_bias=True, with_residual=True)
    return {k: d[k].cuda() for k in ("X", "W", "bias", "residual")}


@pytest.mark.parametrize("cfg", [1, 2, 3, 4, 5, 6, 7, 8, "doubles", "mixed"])
@pytest.mark.parametrize("bias,residual", [(True, True), (False, True), (True, False)])
def test_tiles_in_a_row(cfg, bias, residual, data, monkeypatch):
    from paper_2605_26632_b200 import binding

    if isinstance(cfg, int):
        monkeypatch.setenv("LYNX_GEMM_CFG", str(cfg))
    else:  # two-row-tile kernel: 5 x 26 double slots, all of them or 100 and the rest as singles
        monkeypatch.setenv("LYNX_RT2", "1")
        monkeypatch.setenv("LYNX_RT2_D", "100000" if cfg == "doubles" else "100")
    b, r = data["bias"] if bias else None, data["residual"] if residual else None
    ref, bound = _reference(data["X"], data["W"], b, r)
    ctx = binding.Lynx(0)
    try:
        out = torch.full((M, N + 8), float("nan"), dtype=torch.bfloat16, device="cuda")  # pitch wider than N
        for _ in range(2):
            Y = ctx.act_sparse_linear(data["X"], data["W"], b, binding.COMP_NONE, r, out=out[:, :N])
            assert bool(((Y.double() - ref).abs() <= bound).all())
        assert bool(out[:, N:].isnan().all()), "columns past N were written"
        torch.cuda.synchronize()
        assert ctx.last_error() == 0
    finally:
        ctx.close()
