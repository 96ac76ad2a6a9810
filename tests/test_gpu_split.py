"""GPU tests of the GEMM that splits K over the members of a cluster: every tile and number of splits, with K blocks that do not
divide evenly, ragged rows and columns and a row tile that holds no row."""
import pytest
import torch

import oracle
from paper_2605_26632_b200 import inputs
from test_gpu_epilogue import _reference
from test_gpu_fp8 import check_y, u16

pytestmark = pytest.mark.gpu

# 300 rows: the second 256-row tile holds 44, its second 128-row block none.  The last column tile holds 104 columns of 128-wide
# tiles (less than a quarter's two chunks), 40 of 192-wide ones.  13 K blocks (9 of the FP8 kernel's)
M, N, K, K_FP8 = 300, 1000, 1664, 2304
FORMS = [(tile, s) for tile, most in ((1, 4), (2, 4), (5, 8)) for s in range(2, most + 1)]


@pytest.fixture
def ctx(request, monkeypatch):
    from paper_2605_26632_b200 import binding

    monkeypatch.setenv("LYNX_SPLIT", str(10 * request.param[0] + request.param[1]))
    c = binding.Lynx(0)
    yield c
    torch.cuda.synchronize()
    assert c.last_error() == 0
    c.close()


@pytest.mark.parametrize("ctx", FORMS, indirect=True, ids=str)
@pytest.mark.parametrize("m,n,bias,residual,mode", [(M, N, True, True, 1), (M, N, False, False, 0), (1, 8, True, True, 1), (256, 384, True, False, 1)])
def test_layer(ctx, m, n, bias, residual, mode):
    d = inputs.make_workload(inputs.Workload("t", m, K, n, "outlier", 95), with_bias=True, with_residual=True)
    X, W, b, r = (d[name].cuda() for name in ("X", "W", "bias", "residual"))
    b, r = b if bias else None, r if residual else None
    ref, bound = _reference(X, W, b, r, mode == 1)
    out = torch.full((2, m, n + 8), float("nan"), dtype=torch.bfloat16, device="cuda")  # pitch wider than N
    for i in range(2):
        Y = ctx.act_sparse_linear(X, W, b, mode, r, out=out[i, :, :n])
        assert bool(((Y.double() - ref).abs() <= bound).all())
    assert torch.equal(out[0, :, :n], out[1, :, :n]) and bool(out[:, :, n:].isnan().all())


@pytest.mark.parametrize("ctx", FORMS, indirect=True, ids=str)
@pytest.mark.parametrize("R", [64, 128])
def test_layer_with_low_rank_branch(ctx, R):
    X = inputs.make_x(M, K, "outlier", 96)
    W, b, res = inputs.make_w(N, K, 96), inputs.make_bias(N, 96), inputs.make_residual(M, N, 96)
    LA, LB = inputs.make_lora(N, K, R, 96)
    ref = oracle.act_sparse_linear_lora(u16(X), u16(W), u16(LA), u16(LB), bias=u16(b), comp_mode=1, Yr=u16(res))
    check_y(ctx.act_sparse_linear_lora(X.cuda(), W.cuda(), LA.cuda(), LB.cuda(), b.cuda(), 1, res.cuda()), ref["Y"])


@pytest.mark.parametrize("ctx", FORMS, indirect=True, ids=str)
def test_fp8_layer(ctx):
    X = inputs.make_x(M, K_FP8, "outlier", 97)
    W, b, res = inputs.make_w(N, K_FP8, 97), inputs.make_bias(N, 97), inputs.make_residual(M, N, 97)
    oq, ows = oracle.quantize_weights_fp8(u16(W), True)
    ref = oracle.act_sparse_linear_fp8(u16(X), oq, ows, bias=u16(b), comp_mode=1, Yr=u16(res))
    Wq, ws = ctx.quantize_weights_fp8(W.cuda(), True)
    check_y(ctx.act_sparse_linear_fp8(X.cuda(), Wq, ws, b.cuda(), 1, res.cuda()), ref["Y"])


@pytest.mark.parametrize("ctx", FORMS, indirect=True, ids=str)
def test_whole_tensor_and_group_scales(ctx):
    X, W, b, res = inputs.make_x(M, K, "outlier", 98), inputs.make_w(N, K, 98), inputs.make_bias(N, 98), inputs.make_residual(M, N, 98)
    for mode in (2, 3):
        ref = oracle.act_sparse_linear(u16(X), u16(W), bias=u16(b), comp_mode=mode, Yr=u16(res))
        check_y(ctx.act_sparse_linear(X.cuda(), W.cuda(), b.cuda(), mode, res.cuda()), ref["Y"])


def test_the_forced_form_is_what_runs(monkeypatch):
    """Every split adds its own K blocks: some last bits differ from the unsplit product's and from another split's.  A form that
    does not exist is refused."""
    from paper_2605_26632_b200 import binding

    X, W = inputs.make_x(M, K, "outlier", 99).cuda(), inputs.make_w(N, K, 99).cuda()
    got = []
    for form in ("0", "12", "13", "14"):
        monkeypatch.setenv("LYNX_SPLIT", form)
        c = binding.Lynx(0)
        got.append(c.act_sparse_linear(X, W))
        torch.cuda.synchronize()
        assert c.last_error() == 0
        c.close()
    for i in range(len(got)):
        for j in range(i):
            assert not torch.equal(got[i], got[j]), (i, j)
    for form in ("11", "15", "31", "59"):  # one split, ten CTAs in a cluster, no such tile, nine splits
        monkeypatch.setenv("LYNX_SPLIT", form)
        c = binding.Lynx(0)
        with pytest.raises(binding.LynxError):
            c.act_sparse_linear(X, W)
        c.close()
