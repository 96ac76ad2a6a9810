"""GPU tests of the GEMM epilogue where tiles follow one another on a CTA pair: staging boxes that are used again (16- and
32-row ones), the last tile staged in the ring, ragged rows and columns, with and without bias and residual."""
import pytest
import torch

from paper_2605_26632_b200 import inputs

pytestmark = pytest.mark.gpu


def _reference(X, W, bias, residual, row_scale=False):
    """The layer in fp64, and the bound of a correct bf16 result around it: half a bf16 step of the
    result (2^-9 relative) and of what a carry into the next binade adds (another 2^-9), plus fp32 sums of K terms
    (K 2^-24 of the sum of magnitudes).  With the rows' scales sqrt(num / den), num and den fp32 sums of K non-negative
    terms: K 2^-24 of each, halved by the root and added, and four roundings (+, /, root, the product with it)."""
    g = X.double().reshape(-1, 4)
    order = g.abs().sort(dim=1, descending=True, stable=True).indices
    kept = (g * torch.zeros_like(g).scatter_(1, order[:, :2], 1.0)).reshape(X.shape)
    ref, mag, terms = kept @ W.double().T, kept.abs() @ W.double().abs().T, X.shape[1]
    if row_scale:
        s = (g.square().reshape(X.shape).sum(1) / (kept.square().sum(1) + 1e-8)).sqrt()[:, None]
        ref, mag, terms = ref * s, mag * s, 2 * terms + 4
    for addend in (bias, residual):
        if addend is not None:
            ref, mag = ref + addend.double(), mag + addend.double().abs()
    return ref, ref.abs() * 2.0 ** -8 + mag * (terms * 2.0 ** -24)


# M and N ragged, over two tiles per CTA pair (one-CTA tiles: per CTA) in every configuration.  The last column tile holds 16
# columns, less than one epilogue chunk, of the 128-, 192- and 256-wide tiles (a 240-wide one 160); with N = 6256 also of these.
M, K, N, N_240 = 2570, 256, 6160, 6256


def _data(n):
    d = inputs.make_workload(inputs.Workload("t", M, K, n, "outlier", 91), with_bias=True, with_residual=True)
    return {k: d[k].cuda() for k in ("X", "W", "bias", "residual")}


@pytest.fixture(scope="module")
def data():
    return _data(N)


@pytest.fixture(scope="module")
def data_240():
    return _data(N_240)


def _select(cfg, monkeypatch):
    if isinstance(cfg, int):
        monkeypatch.setenv("LYNX_GEMM_CFG", str(cfg))
    else:  # two-row-tile kernel: 5 x 26 (27) double slots, all of them or 100 and the rest as singles
        monkeypatch.setenv("LYNX_RT2", "1")
        monkeypatch.setenv("LYNX_RT2_D", "100000" if cfg == "doubles" else "100")


def _check_twice(data, bias, residual, row_scale):
    from paper_2605_26632_b200 import binding

    X, W = data["X"], data["W"]
    N = W.shape[0]
    b, r = data["bias"] if bias else None, data["residual"] if residual else None
    ref, bound = _reference(X, W, b, r, row_scale)
    ctx = binding.Lynx(0)
    try:
        out = torch.full((M, N + 8), float("nan"), dtype=torch.bfloat16, device="cuda")  # pitch wider than N
        for _ in range(2):
            Y = ctx.act_sparse_linear(X, W, b, binding.COMP_ROW if row_scale else binding.COMP_NONE, r, out=out[:, :N])
            assert bool(((Y.double() - ref).abs() <= bound).all())
        assert bool(out[:, N:].isnan().all()), "columns past N were written"
        torch.cuda.synchronize()
        assert ctx.last_error() == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("cfg", [1, 2, 3, 4, 5, 6, 7, 8, "doubles", "mixed"])
@pytest.mark.parametrize("bias,residual", [(True, True), (False, True), (True, False)])
def test_tiles_in_a_row(cfg, bias, residual, data, monkeypatch):
    _select(cfg, monkeypatch)
    _check_twice(data, bias, residual, False)


@pytest.mark.parametrize("cfg", [7, "doubles", "mixed"])
@pytest.mark.parametrize("residual", [True, False])
def test_last_column_tile_under_one_chunk(cfg, residual, data_240, monkeypatch):
    """240-wide tiles: the second warp of each lane quarter stores nothing of the last column tile."""
    _select(cfg, monkeypatch)
    _check_twice(data_240, True, residual, False)


@pytest.mark.parametrize("cfg", [1, 2, 3, 4, 5, 6, 7, 8, "doubles", "mixed"])
def test_row_scales_of_tiles_in_a_row(cfg, data, monkeypatch):
    """Every row has a scale of its own: one that reached another row, or stayed from the tile before, shows."""
    _select(cfg, monkeypatch)
    _check_twice(data, True, True, True)


@pytest.mark.parametrize("cfg", [4, 5, 7])
def test_stream_k_pieces_with_residual(cfg, monkeypatch):
    """The residual is fetched into the registers of the results: the pieces of a split tile must not add it twice."""
    from paper_2605_26632_b200 import binding

    # 9 x 15, 11 or 12 tiles: 61, 25 or 34 of them left after one round of 74 CTA pairs, 16 K blocks each (4 per pair at least)
    m, k, n = 2300, 2048, 2760
    monkeypatch.setenv("LYNX_GEMM_CFG", str(cfg))
    monkeypatch.setenv("LYNX_STREAMK", "1")
    d = inputs.make_workload(inputs.Workload("t", m, k, n, "outlier", 92), with_bias=True, with_residual=True)
    X, W, b, r = (d[name].cuda() for name in ("X", "W", "bias", "residual"))
    ref, bound = _reference(X, W, b, r, True)
    ctx = binding.Lynx(0)
    try:
        ys = [ctx.act_sparse_linear(X, W, b, binding.COMP_ROW, r) for _ in range(2)]
        assert bool(((ys[0].double() - ref).abs() <= bound).all()) and torch.equal(*ys)
        torch.cuda.synchronize()
        assert ctx.last_error() == 0
    finally:
        ctx.close()
