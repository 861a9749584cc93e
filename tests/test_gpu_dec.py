"""Up to 384 rows with the packed weights decoded inside the product: gemm_dec_kernel (1) at the edges of its panels (128 rows), tiles
(128 columns), pieces of K (pairs of 64) and stages, for every storage form of the weights, and sizes that gemm_tmw_kernel (2) takes:
against the same product behind a pass over the weights.  Both add exact products up in fp32, in orders of their own: at most K/16
rounded additions of partial sums on either side, each within 2^-24 of the absolute sum S, for K <= 16384 2^-13 S at the very most;
1e-5 S as elsewhere.  The fused tail and the MXInt result come from the same sums."""
import pytest
import torch

from paper_2307_15517_b200 import binding as mxb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,block,wa,ww,rows2,kernel", [
    (17, 4096, 4112, 16, 8, 4, 1, 0),      # one panel, K in four pieces (the query starts at 33 rows)
    (33, 784, 3002, 16, 8, 8, 1, 1),       # K % 64 == 16, exponent rows of 49 bytes, a ragged last tile; bytes
    (128, 8224, 2050, 32, 7, 4, 2, 1),     # odd K steps in eight pieces, weights in two-row blocks
    (64, 96, 32000, 32, 6, 3, 1, 2),       # two K steps
    (100, 2080, 2001, 16, 8, 2, 1, 1),     # odd row length: stores of single values
    (40, 4096, 2000, 16, 4, 4, 1, 1),      # operands that could be records
    (129, 3104, 4100, 16, 8, 4, 1, 1),     # two panels
    (256, 4096, 4096, 32, 8, 8, 1, 1),
    (256, 1040, 16200, 16, 8, 6, 1, 2),
    (257, 4112, 4090, 16, 8, 8, 2, 0),     # (near the line between them)
    (384, 8192, 4096, 16, 8, 4, 1, 2),
    (384, 4192, 4200, 32, 4, 4, 1, 1),     # three panels
    (64, 160, 14400, 32, 6, 3, 1, 2),      # three K steps
    (100, 1344, 28416, 16, 8, 4, 1, 2),
    (96, 720, 130, 16, 8, 8, 1, 1),        # few weights: twelve K steps in three pieces
    (33, 960, 300, 32, 8, 4, 1, 1),        # ... fifteen
    (256, 3088, 16200, 16, 8, 6, 1, 2),
    (71, 288, 7760, 16, 8, 8, 1, 1),       # K not cut
    (151, 5280, 2862, 32, 8, 4, 1, 1),     # two panels, K in five pieces
    (264, 4512, 13286, 16, 8, 3, 1, 1),    # three panels, K not cut
    (272, 4160, 29707, 32, 8, 8, 1, 1),    # two waves
    (309, 9568, 1831, 16, 8, 6, 1, 1),     # three panels in eight pieces
])
def test_weights_decoded_in_the_product(M, K, N, block, wa, ww, rows2, kernel):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + N)
    fa, fw = mxb.MxFormat(block, wa), mxb.MxFormat(block, ww, block_rows=rows2)
    assert not kernel or mxb.mx_selftest_route(M, N, K, fa, fw)[0] == kernel
    ld = -(-K // 8) * 8
    x = torch.randn(M, ld, generator=g, device="cuda")[:, :K]
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02 * torch.exp2(torch.randint(-9, 9, (N, 1), generator=g, device="cuda").float())
    wm, we = mxb.mx_quantize(w, fw)
    bias = torch.randn(N, generator=g, device="cuda")

    def absolute(m, e, f):
        return mxb.mx_dequantize(m, e, K, f).abs()

    am, ae = mxb.mx_quantize(x, fa)
    S = absolute(am, ae, fa).double() @ absolute(wm, we, fw).double().t() + bias.abs().double()
    y = torch.full((M, N + 4), -7.0, device="cuda")
    mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y[:, :N])
    want = mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, algo=mxb.MX_ALGO_TCGEN05)
    assert mxb.mx_poll_status() == 0
    assert (y[:, N:] == -7.0).all()
    y = y[:, :N].contiguous()
    assert ((y - want).abs().double() <= 1e-5 * S).all(), float(((y - want).abs().double() / S).max())
    assert torch.equal(mxb.mx_gemm(am, ae, fa, wm, we, fw, M, N, K, bias=bias), y)
    res = torch.randn(M, N, generator=g, device="cuda")
    z = torch.relu(y) + res
    assert torch.equal(mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res), z)
    assert torch.equal(mxb.mx_gemm_fused(am, ae, fa, wm, we, fw, M, N, K, bias=bias, relu=True, residual=res), z)
    for fy in (mxb.MxFormat(16, 8), mxb.MxFormat(32, 4)):
        if N % fy.block == 0:
            for r, call in ((y, lambda: mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias)),
                            (z, lambda: mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res, fy=fy))):
                ym, ye = call()
                qm, qe = mxb.mx_quantize(r, fy)
                assert torch.equal(ym, qm) and torch.equal(ye, qe)
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("block,ww", [(32, 4), (16, 8)])
def test_exponent_rows_at_any_address_and_a_normalised_input(block, ww):
    M, K, N = 70, 4096, 2048
    g = torch.Generator(device="cuda")
    g.manual_seed(ww)
    fa, fw = mxb.MxFormat(block, 8), mxb.MxFormat(block, ww)
    x = torch.randn(M, K, generator=g, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    y = mxb.mx_linear(x, fa, wm, we, fw, N)
    buf = torch.empty(we.numel() + 1, dtype=torch.uint8, device="cuda")
    buf[1:] = we.flatten()
    shifted = buf[1:].view(we.shape)
    assert shifted.data_ptr() % 4 == 1
    assert torch.equal(mxb.mx_linear(x, fa, wm, shifted, fw, N), y)
    gamma, beta = torch.randn(K, generator=g, device="cuda"), torch.randn(K, generator=g, device="cuda")
    a = mxb.mx_linear_fused(x, fa, wm, we, fw, N, layernorm=(gamma, beta, 1e-5))
    n = torch.nn.functional.layer_norm(x.double(), (K,), gamma.double(), beta.double(), 1e-5).float()
    # a normalised value that lands on the other side of a rounding step moves by a step of its block, at most
    # 2^-6 of the block's largest value: the outputs' error is that of quantizing, the same for both
    b = mxb.mx_linear(n, fa, wm, we, fw, N, algo=mxb.MX_ALGO_TCGEN05)
    assert (a - b).norm() <= 2e-3 * b.norm()
    assert mxb.mx_poll_status() == 0


def _launches(call):
    mxb.mx_profile_begin()
    call()
    return {kind: n for kind, (_, n) in mxb.mx_profile_end().items()}


@pytest.mark.parametrize("M,K,N,block,wa,ww,kernel", [
    (64, 704, 512, 16, 8, 4, 5), (64, 768, 512, 16, 8, 4, 1), (33, 960, 256, 16, 8, 4, 1), (33, 992, 256, 16, 8, 4, 4),
    (128, 768, 256, 16, 8, 4, 5), (128, 768, 768, 16, 4, 4, 1), (128, 896, 768, 16, 8, 4, 5),
    (128, 1024, 9600, 16, 8, 4, 2), (64, 1024, 9600, 16, 8, 4, 2), (128, 256, 9600, 16, 8, 4, 2), (128, 4096, 9600, 16, 8, 4, 2),
    (128, 1024, 18944, 16, 8, 4, 2), (128, 1024, 19072, 16, 8, 4, 2), (128, 1024, 28672, 16, 8, 4, 2),
    (128, 1344, 28672, 16, 8, 4, 2), (128, 4096, 19072, 16, 8, 4, 2), (128, 2048, 19072, 16, 8, 4, 2),
    (256, 1024, 16384, 16, 8, 4, 2), (256, 3072, 14336, 16, 8, 4, 2), (384, 4096, 6144, 16, 8, 4, 2),
    (384, 4096, 4096, 16, 8, 4, 2), (100, 2080, 3002, 16, 8, 4, 1), (1237, 2080, 3002, 16, 6, 6, 7), (352, 2048, 1024, 16, 8, 4, 4),
    (256, 4096, 4096, 32, 8, 8, 1), (1536, 4096, 11008, 16, 8, 4, 2), (1537, 4096, 11008, 16, 8, 4, 6), (1400, 768, 31, 16, 8, 4, 5),
])
def test_sizes_at_which_the_weights_are_decoded_in_the_product(M, K, N, block, wa, ww, kernel):
    """Sizes of every route, by the query and by the launches: with kernels 1 and 2 a pass over the activations alone."""
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("sizes for 148 SMs")
    fa, fw = mxb.MxFormat(block, wa), mxb.MxFormat(block, ww)
    assert mxb.mx_selftest_route(M, N, K, fa, fw)[0] == kernel
    x = torch.randn(M, K, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, device="cuda"), fw)
    n = _launches(lambda: mxb.mx_linear(x, fa, wm, we, fw, N))
    assert (n["quantize"] == 1 and n["prep"] == n["dequantize"] == 0) == (kernel in (1, 2)), n
    assert n["gemm_tc"] == 1


def check_ends_of_the_range(M, K, N, block, ww):
    """Weight blocks with the exponent bytes 0, 225, 226, 254 and 255, a NaN and an infinity among the activations, against the
    CUDA-core kernel: the same NaN, the other sums within the tolerance (1e-37: sums below the normal range)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + ww)
    fa, fw = mxb.MxFormat(block, 8), mxb.MxFormat(block, ww)
    x = torch.randn(M, K, generator=g, device="cuda")
    x[:12] *= 2.0 ** -20
    x[2, 100], x[7, K - 1] = float("nan"), float("inf")
    x[-1] *= 2.0 ** -110
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    per = block // 2 if ww <= 4 else block                # bytes of a block
    for row, blk, e in ((3, 1, 0), (4, 2, 225), (5, 3, 226), (6, 0, 254), (N - 1, K // block - 1, 255), (130, 4, 255)):
        we[row, blk] = e
        if e not in (0, 255):                             # one small mantissa: the row's sums stay below the largest float
            wm[row, blk * per:(blk + 1) * per] = 0
            wm[row, blk * per] = 1
            x[:, blk * block] *= 2.0 ** -30
    y = mxb.mx_linear(x, fa, wm, we, fw, N)
    want = mxb.mx_linear(x, fa, wm, we, fw, N, algo=mxb.MX_ALGO_SIMT)
    assert mxb.mx_poll_status() == 0
    nan = torch.isnan(want)
    assert nan[2].all() and nan[7].all() and nan[:, N - 1].all() and nan[:, 130].all() and not nan[0, :130].any()
    assert torch.equal(torch.isnan(y), nan)
    a, w = (mxb.mx_dequantize(*mxb.mx_quantize(x, fa), K, fa), mxb.mx_dequantize(wm, we, K, fw))
    S = a.nan_to_num(0.0).abs().double() @ w.nan_to_num(0.0).abs().double().t()
    ok = ~nan
    assert torch.isfinite(want[ok]).all()
    assert ((y - want).abs().double()[ok] <= 1e-5 * S[ok] + 1e-37).all()


@pytest.mark.parametrize("M,K,N,block,ww", [(40, 4096, 2048, 16, 4), (128, 4128, 4096, 16, 8), (200, 4096, 4100, 32, 4), (300, 4112, 4224, 16, 8)])
def test_exponents_at_the_ends_of_the_range_decoded_in_the_product(M, K, N, block, ww):
    assert _launches(lambda: mxb.mx_linear(torch.zeros(M, K, device="cuda"), mxb.MxFormat(block, 8), *mxb.mx_quantize(
        torch.zeros(N, K, device="cuda"), mxb.MxFormat(block, ww)), mxb.MxFormat(block, ww), N))["prep"] == 0
    check_ends_of_the_range(M, K, N, block, ww)


@pytest.mark.parametrize("case", ("decoded", "decoded, exponents at odd addresses", "grouped", "one token"))
def test_weights_written_by_the_launch_in_front(case):
    """The kernels that fetch weights while the pass over the activations still runs: weights quantized into the same buffers
    right before each call, with nothing in between, are the ones that it uses."""
    M, K, N = {"grouped": (5, 2048, 8192), "one token": (1, 4096, 11008)}.get(case, (128, 4096 + 16 * ("odd" in case), 4096))
    block = 16 if "decoded" in case else 32
    g = torch.Generator(device="cuda")
    g.manual_seed(len(case))
    fa, fw = mxb.MxFormat(block, 8), mxb.MxFormat(block, 8 if "odd" in case else 4)
    x = torch.randn(M, K, generator=g, device="cuda")
    ws = [torch.randn(N, K, generator=g, device="cuda") for _ in range(6)]
    wm, we = mxb.mx_quantize(ws[0], fw)
    work = mxb.alloc_workspace(mxb.mx_workspace_bytes(M, N, K, fa, fw))

    def call(m, e, y):
        if case == "grouped":
            args = mxb.make_linear_args([dict(x=x, fa=fa, w_mant=m, w_exp=e, fw=fw, N=N, y=y)] * 2)
            mxb.mx_linear_grouped(args, workspace=grouped)
        else:
            mxb.mx_linear(x, fa, m, e, fw, N, y=y, workspace=work)

    if case == "grouped":
        grouped = mxb.alloc_workspace(mxb.mx_linear_grouped_workspace_bytes(
            mxb.make_linear_args([dict(x=x, fa=fa, w_mant=wm, w_exp=we, fw=fw, N=N, y=x)] * 2)))
    want = []
    for w in ws:
        m, e = mxb.mx_quantize(w, fw)
        want.append(torch.empty(M, N, device="cuda"))
        torch.cuda.synchronize()
        call(m, e, want[-1])
        torch.cuda.synchronize()
    got = [torch.empty(M, N, device="cuda") for _ in range(24)]
    for i, y in enumerate(got):
        mxb.mx_quantize(ws[i % 6], fw, wm, we)
        call(wm, we, y)
    for i, y in enumerate(got):
        assert torch.equal(y, want[i % 6]), i
    assert mxb.mx_poll_status() == 0
