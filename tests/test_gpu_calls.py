"""The native marshalling of the frequent calls (no stream named) against the ctypes route (a stream named): same results, same
errors, results in the caller's tensors."""
import pytest
import torch

from paper_2307_15517_b200 import binding as mxb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", (torch.float32, torch.bfloat16))
def test_native_and_ctypes_routes_agree(dtype):
    st = torch.cuda.current_stream()
    M, K, N = 48, 256, 96
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    fa, fw, fy = mxb.MxFormat(16, 8), mxb.MxFormat(16, 4), mxb.MxFormat(32, 4)
    x = torch.randn(M, K, generator=g, device="cuda").to(dtype)
    bias, res = torch.randn(N, generator=g, device="cuda"), torch.randn(M, N, generator=g, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda"), fw)
    for f, t in ((fa, x), (fy, x.t()[:64, :32]), (mxb.MxFormat(16, 8, block_rows=2), x)):
        a, b = mxb.mx_quantize(t, f), mxb.mx_quantize(t, f, stream=st)
        assert all(torch.equal(u, v) for u, v in zip(a, b))
        out = tuple(torch.empty_like(u) for u in a)
        got = mxb.mx_quantize(t, f, out[0], out[1])
        assert got[0] is out[0] and got[1] is out[1] and torch.equal(out[0], a[0])
    am, ae = mxb.mx_quantize(x, fa)
    d = torch.empty(M, K, dtype=dtype, device="cuda")
    assert mxb.mx_dequantize(am, ae, K, fa, dtype=dtype, out=d) is d
    assert torch.equal(d, mxb.mx_dequantize(am, ae, K, fa, dtype=dtype, stream=st)) and d.dtype == dtype
    y = torch.empty(M, N, device="cuda")
    assert mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y) is y
    assert torch.equal(y, mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, stream=st))
    ln = (torch.rand(K, generator=g, device="cuda"), torch.rand(K, generator=g, device="cuda"), 1e-5)
    for more in (dict(relu=True), dict(residual=res), dict(fy=fy, relu=True)) + ((dict(layernorm=ln),) if dtype == torch.float32 else ()):
        a, b = (mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, stream=s, **more) for s in (None, st))
        assert all(torch.equal(u, v) for u, v in zip(a, b))
        if "layernorm" not in more:
            a, b = (mxb.mx_gemm_fused(am, ae, fa, wm, we, fw, M, N, K, bias=bias, stream=s, **more) for s in (None, st))
            assert all(torch.equal(u, v) for u, v in zip(a, b))
    q = torch.randn(64, 3 * 128, generator=g, device="cuda").to(dtype)
    a, b = (mxb.mx_attention_fp(q[:, :128], q[:, 128:256], q[:, 256:], fa, fa, 2, 64, 0.125, fa, stream=s) for s in (None, st))
    assert torch.equal(a, b)
    assert mxb.mx_poll_status() == 0


def test_errors_are_those_of_the_ctypes_route():
    f = mxb.MxFormat(16, 4)
    x = torch.zeros(4, 64, device="cuda")
    wm, we = mxb.mx_quantize(torch.zeros(8, 64, device="cuda"), f)
    for bad, err in ((lambda **k: mxb.mx_quantize(torch.zeros(4, 64), f, **k), ValueError),
                     (lambda **k: mxb.mx_quantize(x.half(), f, **k), TypeError),
                     (lambda **k: mxb.mx_quantize(x[:, :40], f, **k), mxb.MxError),
                     (lambda **k: mxb.mx_linear(x, f, wm, we, mxb.MxFormat(32, 4), 8, **k), mxb.MxError),
                     (lambda **k: mxb.mx_linear(x, f, wm, we, f, 8, workspace=torch.empty(8, dtype=torch.uint8, device="cuda"), **k), mxb.MxError),
                     (lambda **k: mxb.mx_linear(x.t(), f, wm, we, f, 8, **k), AssertionError),
                     (lambda **k: mxb.mx_dequantize(wm, we, 64, mxb.MxFormat(16, 9), **k), mxb.MxError)):
        texts = []
        for more in ({}, dict(stream=torch.cuda.current_stream())):
            with pytest.raises(err) as e:
                bad(**more)
            texts.append(str(e.value))
        assert texts[0] == texts[1]


@pytest.mark.parametrize("transform", ("vmap", "grad", "functionalize"))
def test_tensors_without_storage_are_refused_as_by_the_ctypes_route(transform):
    """The wrappers that vmap, grad and functionalize pass in have the Python type torch.Tensor and no storage: their pointer
    cannot be taken, in no argument of no call."""
    f, fy = mxb.MxFormat(16, 8), mxb.MxFormat(32, 4)
    x, q = torch.randn(32, 64, device="cuda"), torch.randn(32, 3 * 64, device="cuda")
    (wm, we), (am, ae) = mxb.mx_quantize(torch.randn(32, 64, device="cuda"), f), mxb.mx_quantize(x, f)
    y, ctx = torch.empty(32, 32, device="cuda"), torch.empty(32, 64, device="cuda")
    ws = mxb.alloc_workspace(1 << 20)

    def under(call, t):                                                   # `call` with a wrapper of t
        if transform == "vmap":
            return torch.func.vmap(call, randomness="different")(t[None])
        if transform == "grad":
            return torch.func.grad(lambda v: call(v).sum())(t)
        return torch.func.functionalize(call)(t)

    calls = [(x, lambda t, **m: mxb.mx_quantize(t, f, **m)[0]),
             (wm, lambda t, **m: mxb.mx_dequantize(t, we, 64, f, **m)),
             (x, lambda t, **m: mxb.mx_linear(t, f, wm, we, f, 32, workspace=ws, **m)),
             (y, lambda t, **m: mxb.mx_linear(x, f, wm, we, f, 32, y=t, workspace=ws, **m)),
             (x, lambda t, **m: mxb.mx_linear_fused(t, f, wm, we, f, 32, fy=fy, workspace=ws, **m)[0]),
             (y, lambda t, **m: mxb.mx_linear_fused(x, f, wm, we, f, 32, residual=t, workspace=ws, **m)),
             (am, lambda t, **m: mxb.mx_gemm_fused(t, ae, f, wm, we, f, 32, 32, 64, workspace=ws, **m)),
             (q, lambda t, **m: mxb.mx_attention_fp(t[:, :64], t[:, 64:128], t[:, 128:], f, f, 1, 64, 0.125, f, workspace=ws, **m)),
             (ctx, lambda t, **m: mxb.mx_attention_fp(q[:, :64], q[:, 64:128], q[:, 128:], f, f, 1, 64, 0.125, f, ctx=t, workspace=ws, **m))]
    for t, call in calls:
        if transform == "grad" and not t.is_floating_point():
            continue
        texts = []
        for more in ({}, dict(stream=torch.cuda.current_stream())):
            with pytest.raises(RuntimeError) as e:
                under(lambda v: call(v, **more), t)
            texts.append(str(e.value).splitlines()[0])
        assert texts[0] == texts[1]
    # the interpreter goes on, with its lock
    assert torch.equal(mxb.mx_quantize(x, f)[0], am)
    assert mxb.mx_poll_status() == 0
