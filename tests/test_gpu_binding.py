"""The binding's compiled calls against its general path: what they take gives the same results, what they do not take (and
what the library refuses) still ends where it did."""
import pytest
import torch

from paper_2605_26632_b200 import binding, inputs

pytestmark = pytest.mark.gpu

M, K, N, R = 200, 512, 264, 64


@pytest.fixture(scope="module")
def pair():
    fast, general = binding.Lynx(0), binding.Lynx(0)
    assert fast._calls is binding.load_calls()
    general._calls = binding._GeneralPathOnly
    yield fast, general
    torch.cuda.synchronize()
    fast.close()
    general.close()


@pytest.fixture(scope="module")
def t():
    d = inputs.make_workload(inputs.Workload("t", M, K, N, "outlier", 7), with_bias=True, with_residual=True)
    t = {k: v.cuda() for k, v in d.items() if torch.is_tensor(v)}
    LA, LB = inputs.make_lora(N, K, R, 7)
    t["LA"], t["LB"] = LA.cuda(), LB.cuda()
    t["wide"] = torch.zeros(M, K + 32, dtype=torch.bfloat16, device="cuda")  # a leading dimension of its own
    t["wide"][:, :K] = t["X"]
    return t


def _calls(t):
    X, W, b, r = t["X"], t["W"], t["bias"], t["residual"]
    P = torch.nn.Parameter(W, requires_grad=False)
    yield "layer", lambda c: c.act_sparse_linear(X, W, b, 1)
    yield "positional out", lambda c: c.act_sparse_linear(X, P, None, 0, r, torch.zeros(M, N, dtype=torch.bfloat16, device="cuda"), 0)
    yield "strided", lambda c: c.act_sparse_linear(t["wide"][:, :K], W, b, 1, r, out=torch.zeros(M, N + 8, dtype=torch.bfloat16, device="cuda")[:, :N])
    yield "gradients on", lambda c: c.act_sparse_linear(X, torch.nn.Parameter(W), b, 1)
    for mode in (0, 1, 2, 3):
        yield f"mode {mode}", lambda c, mode=mode: c.act_sparse_linear(X, W, b, mode, r)
        yield f"prune {mode}", lambda c, mode=mode: c.prune_compress(X, mode)
    yield "prune into", lambda c: c.prune_compress(X, 1, torch.zeros(M, K // 2, dtype=torch.bfloat16, device="cuda"),
                                                   torch.zeros(binding.meta_bytes(M, K), dtype=torch.uint8, device="cuda"))
    yield "two calls", lambda c: c.sparse_linear(*c.prune_compress(X, 1)[:2], W, b, c.prune_compress(X, 1)[2], r)
    yield "deferred", lambda c: c.sparse_linear(*c.prune_compress(X, 1, row_scale=binding.ROW_SCALE_DEFERRED)[:2], W, b, binding.ROW_SCALE_DEFERRED)
    yield "lora", lambda c: c.act_sparse_linear_lora(X, W, t["LA"], t["LB"], b, 1, r)
    yield "fp8", lambda c: c.act_sparse_linear_fp8(X, *c.quantize_weights_fp8(W), b, 1, r)
    yield "fp8 maxima", lambda c: c.act_sparse_linear_fp8(X, *c.quantize_weights_fp8(W), row_amax=X.float().abs().amax(1))


def test_same_results(pair, t):
    for name, call in _calls(t):
        a, b = (call(c) for c in pair)
        for x, y in zip(a if type(a) is tuple else (a,), b if type(b) is tuple else (b,)):
            assert (x is None) == (y is None), name
            if torch.is_tensor(x):
                assert type(x) is type(y) and x.shape == y.shape and x.dtype == y.dtype and x.requires_grad == y.requires_grad, name
                assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), name


def test_out_is_returned_as_it_came(pair, t):
    out = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    for c in pair:
        assert c.act_sparse_linear(t["X"], t["W"], out=out) is out


def test_other_streams_and_modes(pair, t):
    want = pair[1].act_sparse_linear(t["X"], t["W"], t["bias"], 1)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        got = pair[0].act_sparse_linear(t["X"], t["W"], t["bias"], 1)
    side.synchronize()
    assert torch.equal(got, want)
    with torch.inference_mode():
        got = pair[0].act_sparse_linear(t["X"], t["W"], t["bias"], 1)
    assert got.is_inference() and torch.equal(got, want)
    seen = []

    class Mode(torch.overrides.TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))

    with Mode():  # sees what it saw of the general path
        assert torch.equal(pair[0].act_sparse_linear(t["X"], t["W"], t["bias"], 1), want) and seen


def test_what_was_refused_is_refused(pair, t):
    X, W, b = t["X"], t["W"], t["bias"]
    odd = torch.zeros(M, N + 4, dtype=torch.bfloat16, device="cuda")
    bad = [(lambda c: c.act_sparse_linear(X.float(), W, b), TypeError), (lambda c: c.act_sparse_linear(X, W.t(), b), TypeError),
           (lambda c: c.act_sparse_linear(X[0], W, b), TypeError), (lambda c: c.act_sparse_linear(X, W, b, 7), binding.LynxError),
           (lambda c: c.act_sparse_linear(X, W[:, :256].contiguous(), b), binding.LynxError),
           (lambda c: c.act_sparse_linear(X, W, b, out=odd[:, :N]), binding.LynxError),
           (lambda c: c.act_sparse_linear(X[:0], W, b), binding.LynxError),
           (lambda c: c.act_sparse_linear_fp8(X, torch.zeros(N, 300, dtype=torch.uint8, device="cuda")), binding.LynxError),
           (lambda c: c.prune_compress(X[:, :200].contiguous(), 1), binding.LynxError),
           (lambda c: c.act_sparse_linear(X, W, b, mode=2, fuse=2), binding.LynxError)]
    for call, error in bad:
        caught = []
        for c in pair:
            with pytest.raises(error) as e:
                call(c)
            caught.append(str(e.value))
        assert caught[0] == caught[1]


def test_wrapped_tensors_take_the_general_path(pair, t):
    calls = pair[0]._calls

    class Sub(torch.Tensor):
        pass

    def layer(X, W=t["W"]):
        return calls.layer(pair[0]._address, X, W, None, 1, None, None, 0)

    assert layer(t["X"]) is not None
    assert layer(t["X"].as_subclass(Sub)) is None and layer(t["X"].cpu()) is None and layer(t["X"], None) is None
    answers = []
    torch.vmap(lambda x: answers.append(layer(x)) or x)(t["X"][None])
    assert answers == [None]
