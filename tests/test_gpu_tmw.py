"""Packed weights decoded into tensor memory (gemm_tmw_kernel) at the edges of its tiles (256 features, 64 .. 256 tokens), rounds
(one and two accumulators), K steps (odd numbers of 64, a rest of 16 k) and stages, for both containers, against the same product
behind a pass over the weights.  Both are one chain of K steps per output, whose 16 exact products the MMA adds with the
accumulator in whatever order the operands have: the same bits.  The element-wise tail and the MXInt result come from those."""
import pytest
import torch

from paper_2307_15517_b200 import binding as mxb

pytestmark = pytest.mark.gpu


def runs(M, K, N, fa, fw, tokens, pieces, quantized=False):
    """The kernel, and on 148 SMs its tile and its pieces of K, for the fp32 or the MXInt result."""
    route = mxb.mx_selftest_route(M, N, K, fa, fw, quantized)
    tile = torch.cuda.get_device_properties(0).multi_processor_count == 148
    assert route[0] == 2 and (not tile or route[1:] == (tokens, pieces)), route


@pytest.mark.parametrize("M,K,N,block,wa,ww,rows2,tokens", [
    (400, 784, 8200, 16, 8, 8, 1, 224),    # K % 64 == 16, exponent rows of 49 bytes; one accumulator
    (385, 4128, 16200, 32, 6, 4, 1, 224),  # two rounds, a ragged last tile of features
    (700, 592, 16001, 16, 7, 5, 1, 192),   # four rounds; rows of 37 exponent bytes; odd row length
    (640, 4096, 4100, 16, 8, 3, 1, 160),   # one round
    (900, 8192, 4102, 32, 8, 4, 2, 256),   # weights in two-row blocks
    (513, 1344, 12290, 16, 8, 6, 1, 192),  # a last token tile of 129, whole tiles of the second CTA outside
    (257, 2080, 12290, 16, 8, 2, 1, 96),   # 33 K steps
    (130, 1296, 16162, 16, 8, 8, 2, 160),  # 21 K steps; bytes in two-row blocks
    (500, 96, 16384, 32, 8, 4, 1, 192),    # two K steps (one and a half)
    (600, 160, 14000, 32, 6, 8, 1, 160),   # three K steps
    (1400, 512, 11582, 16, 8, 4, 1, 192),
    (1500, 64, 16384, 16, 8, 4, 1, 192),   # tiles of one step, each a stage of packed weights, of which a group has every third
    (1500, 32, 16384, 32, 4, 3, 1, 192),
    (1500, 48, 16384, 16, 8, 8, 1, 192),
    (1000, 96, 16000, 16, 8, 8, 1, 160),   # two steps, one stage
    (768, 4096, 11008, 32, 8, 8, 1, 256),  # bytes: a group has no step in every third stage; eight stages of decoded weights
    (500, 1104, 8192, 16, 8, 6, 1, 256),
    (33, 32, 136, 32, 8, 3, 1, 64),        # the smallest: half a step, a token beyond the first CTA's
    (170, 32, 9522, 16, 8, 3, 1, 64),      # two rounds
    (152, 80, 10562, 16, 8, 6, 1, 160),
    (245, 32, 10196, 16, 8, 8, 1, 256),
    (198, 32, 11144, 32, 8, 4, 1, 96),
    (524, 80, 6612, 16, 8, 6, 1, 128),
    (485, 32, 6322, 32, 8, 4, 1, 128),
    (275, 352, 13702, 32, 8, 3, 1, 160),
    (1505, 272, 4630, 16, 8, 5, 1, 224),   # bytes, one accumulator, several rounds
    (1098, 416, 6702, 16, 8, 4, 1, 224),
    (984, 416, 9006, 16, 8, 2, 2, 256),
])
def test_weights_decoded_into_tensor_memory(M, K, N, block, wa, ww, rows2, tokens):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + N)
    fa, fw = mxb.MxFormat(block, wa), mxb.MxFormat(block, ww, block_rows=rows2)
    runs(M, K, N, fa, fw, tokens, 1)
    ld = -(-K // 8) * 8
    x = torch.randn(M, ld, generator=g, device="cuda")[:, :K]
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02 * torch.exp2(torch.randint(-9, 9, (N, 1), generator=g, device="cuda").float())
    wm, we = mxb.mx_quantize(w, fw)
    bias = torch.randn(N, generator=g, device="cuda")
    y = torch.full((M, N + 4), -7.0, device="cuda")
    mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y[:, :N])
    want = mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, algo=mxb.MX_ALGO_TCGEN05)
    assert mxb.mx_poll_status() == 0
    assert (y[:, N:] == -7.0).all()
    y = y[:, :N].contiguous()
    assert torch.equal(y, want)
    am, ae = mxb.mx_quantize(x, fa)
    assert torch.equal(mxb.mx_gemm(am, ae, fa, wm, we, fw, M, N, K, bias=bias), y)
    res = torch.randn(M, N, generator=g, device="cuda")
    z = torch.relu(y) + res
    assert torch.equal(mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res), z)
    assert torch.equal(mxb.mx_gemm_fused(am, ae, fa, wm, we, fw, M, N, K, bias=bias, relu=True, residual=res), z)
    for fy in (mxb.MxFormat(16, 8), mxb.MxFormat(32, 4), mxb.MxFormat(16, 5, block_rows=2)):
        if N % fy.block == 0 and M % fy.block_rows == 0:
            for r, call in ((y, lambda: mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias)),
                            (z, lambda: mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res, fy=fy))):
                ym, ye = call()
                qm, qe = mxb.mx_quantize(r, fy)
                assert torch.equal(ym, qm) and torch.equal(ye, qe)
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("M,K,N,block,wa,ww,tokens,pieces", [
    (226, 3312, 6184, 16, 8, 6, 256, 2),   # the last K step of 48; a ragged last tile of features
    (640, 8192, 2048, 32, 6, 4, 160, 2),
    (352, 8192, 2048, 16, 8, 4, 192, 3),
    (400, 16400, 4096, 16, 8, 8, 224, 2),  # bytes
    (502, 4192, 2693, 32, 8, 4, 256, 3),   # pieces of unequal length, the last K step of 32; odd row length
    (38, 464, 137, 16, 8, 6, 64, 2),       # a second piece of two stages of packed weights, half of the features outside
    (36, 5920, 4273, 16, 8, 2, 64, 3),
    (194, 1104, 1668, 16, 8, 7, 96, 3),
    (207, 1232, 2919, 16, 8, 8, 128, 2),
    (126, 8224, 4788, 16, 8, 2, 128, 3),
    (104, 11104, 3807, 16, 8, 4, 128, 4),
    (139, 3552, 3196, 32, 8, 3, 160, 4),
    (188, 1584, 5964, 16, 8, 5, 192, 2),
    (171, 2352, 3573, 16, 8, 8, 192, 4),
    (395, 3296, 2524, 32, 8, 3, 224, 3),
    (239, 10528, 2543, 32, 8, 3, 256, 4),
])
def test_pieces_of_K_added_up_in_a_cluster(M, K, N, block, wa, ww, tokens, pieces):
    """The partial sums of two to four pieces are added in fp32: at most one rounding of a partial sum more than one chain per
    piece, 2^-22 of the absolute sum S; 1e-5 S as elsewhere.  The tail and the MXInt result come from the same sums."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + N)
    fa, fw = mxb.MxFormat(block, wa), mxb.MxFormat(block, ww)
    runs(M, K, N, fa, fw, tokens, pieces)
    x = torch.randn(M, K, generator=g, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    bias = torch.randn(N, generator=g, device="cuda")
    am, ae = mxb.mx_quantize(x, fa)
    S = mxb.mx_dequantize(am, ae, K, fa).abs().double() @ mxb.mx_dequantize(wm, we, K, fw).abs().double().t() + bias.abs().double()
    y = torch.full((M, N + 4), -7.0, device="cuda")
    mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y[:, :N])
    want = mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, algo=mxb.MX_ALGO_TCGEN05)
    assert (y[:, N:] == -7.0).all()
    y = y[:, :N].contiguous()
    assert ((y - want).abs().double() <= 1e-5 * S).all()
    assert torch.equal(mxb.mx_gemm(am, ae, fa, wm, we, fw, M, N, K, bias=bias), y)
    assert torch.equal(mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias), y)                # the same every time
    res = torch.randn(M, N, generator=g, device="cuda")
    z = torch.relu(y) + res
    assert torch.equal(mxb.mx_gemm_fused(am, ae, fa, wm, we, fw, M, N, K, bias=bias, relu=True, residual=res), z)
    for fy in (mxb.MxFormat(16, 8), mxb.MxFormat(32, 4)):
        if N % fy.block == 0:
            ym, ye = mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res, fy=fy)
            qm, qe = mxb.mx_quantize(z, fy)
            assert torch.equal(ym, qm) and torch.equal(ye, qe)
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("M,K,N,block,wa,ww,tokens,pieces", [
    (36, 32, 128, 16, 8, 5, 64, 1), (164, 32, 10304, 32, 8, 6, 64, 1), (130, 32, 9568, 32, 8, 2, 64, 1),
    (200, 32, 9664, 16, 8, 8, 96, 1), (200, 32, 9536, 16, 8, 2, 96, 1), (102, 32, 9536, 32, 8, 7, 128, 1), (296, 32, 9536, 32, 8, 7, 128, 1),
    (306, 32, 9632, 32, 8, 2, 128, 1), (130, 32, 9952, 32, 8, 8, 160, 1), (388, 32, 9568, 32, 8, 6, 160, 1), (386, 32, 9600, 32, 8, 3, 160, 1),
    (322, 32, 6240, 32, 8, 6, 192, 1), (484, 32, 9728, 32, 8, 8, 192, 1), (352, 160, 6208, 16, 8, 4, 192, 1), (516, 32, 9760, 32, 8, 4, 192, 1),
    (388, 32, 7712, 16, 8, 6, 224, 1), (642, 32, 9664, 32, 8, 7, 224, 1), (202, 32, 12768, 32, 8, 4, 224, 1), (670, 32, 11328, 32, 8, 2, 224, 1),
    (486, 144, 7264, 16, 8, 6, 256, 1), (730, 4960, 12256, 32, 8, 6, 256, 1), (240, 1056, 11424, 32, 8, 4, 256, 1), (766, 2208, 12480, 16, 8, 2, 256, 1),
    (40, 400, 192, 16, 8, 7, 64, 2), (40, 1104, 128, 16, 8, 7, 64, 3), (38, 1296, 960, 16, 8, 7, 64, 4), (136, 2304, 3552, 32, 8, 4, 96, 2),
    (148, 4544, 2592, 16, 8, 4, 96, 3), (224, 3328, 3744, 32, 8, 2, 128, 2), (158, 1200, 7104, 16, 8, 8, 160, 2), (140, 2080, 4416, 32, 8, 3, 160, 3),
    (132, 3376, 3360, 16, 8, 6, 160, 4), (164, 2448, 5984, 16, 8, 5, 192, 2), (162, 2176, 5216, 32, 8, 5, 192, 3), (172, 5248, 3552, 16, 8, 3, 192, 4),
    (212, 3248, 5952, 16, 8, 7, 224, 2), (202, 2208, 5504, 32, 8, 4, 224, 3), (222, 8224, 3648, 32, 8, 3, 224, 4), (238, 4432, 5920, 16, 8, 6, 256, 2),
    (478, 5024, 2720, 32, 8, 2, 256, 3),
])
def test_MXInt_results_of_every_tile_and_cut(M, K, N, block, wa, ww, tokens, pieces):
    """Uncut: the quantized sums of a product behind a pass.  Cut sums differ from those by 2^-22 of the absolute sum S at most (see
    above), some 1600 steps of a code: a code next to a rounding boundary may move by one step, 8e-4 of them at the very most."""
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + N)
    fa, fw = mxb.MxFormat(block, wa), mxb.MxFormat(block, ww)
    runs(M, K, N, fa, fw, tokens, pieces, True)
    x = torch.randn(M, K, generator=g, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    bias = torch.randn(N, generator=g, device="cuda")
    y = mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, algo=mxb.MX_ALGO_TCGEN05)
    for fy in (mxb.MxFormat(16, 8), mxb.MxFormat(32, 4), mxb.MxFormat(16, 5, block_rows=2)):
        ym, ye = mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias)
        qm, qe = mxb.mx_quantize(y, fy)
        if pieces == 1:
            assert torch.equal(ym, qm) and torch.equal(ye, qe)
        else:
            a, b = mxb.mx_dequantize(ym, ye, N, fy), mxb.mx_dequantize(qm, qe, N, fy)
            step = b.abs().view(M, N // fy.block, fy.block).amax(2, keepdim=True).expand(-1, -1, fy.block).reshape(M, N) * 2.0 ** (3 - fy.elem_bits)
            if fy.block_rows == 2:
                step = step.view(M // 2, 2, N).amax(1, keepdim=True).expand(-1, 2, -1).reshape(M, N)
            assert ((a - b).abs() <= step).all() and (a != b).float().mean() <= 1e-3
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("block,ww", [(16, 4), (32, 8)])
def test_any_exponents_any_address_and_a_normalised_input(block, ww):
    """Exponent bytes at the ends of the range, rows of them at odd addresses, activations from a LayerNorm: as behind a pass."""
    M, K, N = 448, 4096, 9216
    g = torch.Generator(device="cuda")
    g.manual_seed(ww)
    fa, fw = mxb.MxFormat(block, 8), mxb.MxFormat(block, ww)
    x = torch.randn(M, K, generator=g, device="cuda") * 2.0 ** -40
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    for row, blk, e in ((3, 1, 0), (4, 2, 1), (5, 3, 226), (6, 0, 227), (7, 5, 150), (N - 1, K // block - 1, 255), (130, 4, 255)):
        we[row, blk] = e
    runs(M, K, N, fa, fw, 224, 1)
    y = mxb.mx_linear(x, fa, wm, we, fw, N)
    want = mxb.mx_linear(x, fa, wm, we, fw, N, algo=mxb.MX_ALGO_TCGEN05)
    nan = torch.isnan(want)
    assert nan[:, N - 1].all() and nan[:, 130].all() and not nan[:, :130].any()
    assert torch.equal(torch.isnan(y), nan) and torch.equal(y[~nan], want[~nan])
    buf = torch.empty(we.numel() + 1, dtype=torch.uint8, device="cuda")
    buf[1:] = we.flatten()
    shifted = mxb.mx_linear(x, fa, wm, buf[1:].view(we.shape), fw, N)
    assert torch.equal(shifted[~nan], y[~nan])
    gamma, beta = torch.randn(K, generator=g, device="cuda"), torch.randn(K, generator=g, device="cuda")
    a = mxb.mx_linear_fused(x, fa, wm, we, fw, N, layernorm=(gamma, beta, 1e-5))
    b = mxb.mx_linear(mxb.mx_layernorm(x, gamma, beta, 1e-5), fa, wm, we, fw, N)       # the same values, normalised apart
    assert torch.equal(a[~nan], b[~nan])
    assert mxb.mx_poll_status() == 0


def test_weights_written_by_the_launch_in_front():
    """The weights are fetched while the pass over the activations still runs: those quantized into the same buffers right before
    each call, with nothing in between, are the ones that it uses."""
    M, K, N = 640, 4096, 4096
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    fa, fw = mxb.MxFormat(16, 8), mxb.MxFormat(16, 4)
    runs(M, K, N, fa, fw, 160, 1)
    x = torch.randn(M, K, generator=g, device="cuda")
    ws = [torch.randn(N, K, generator=g, device="cuda") for _ in range(5)]
    want = [mxb.mx_linear(x, fa, *mxb.mx_quantize(w, fw), fw, N, algo=mxb.MX_ALGO_TCGEN05) for w in ws]
    wm, we = mxb.mx_quantize(ws[0], fw)
    work = mxb.alloc_workspace(mxb.mx_workspace_bytes(M, N, K, fa, fw))
    got = [torch.empty(M, N, device="cuda") for _ in range(15)]
    torch.cuda.synchronize()
    for i, y in enumerate(got):
        mxb.mx_quantize(ws[i % 5], fw, wm, we)
        mxb.mx_linear(x, fa, wm, we, fw, N, y=y, workspace=work)
    for i, y in enumerate(got):
        assert torch.equal(y, want[i % 5]), i
    assert mxb.mx_poll_status() == 0
