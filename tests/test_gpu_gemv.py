"""Few tokens through one launch (gemv_single_kernel) and grouped calls of three to sixteen tokens (gemv_mma_kernel):
every storage form of the weights at the edges of the steps (256 bytes of a row), groups (64 bytes), 16-byte units, row
tiles and K slices, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import mx_oracle as orc
from paper_2307_15517_b200 import binding as mxb
from paper_2307_15517_b200 import synth

pytestmark = pytest.mark.gpu


def _case(T, K, N, block, wa, ww, rows2=1, dtype=torch.float32, bias=False, seed=0):
    x = synth.student_t_activations(T, K, seed).to(dtype)
    w = synth.gaussian_weights(N, K, seed + 1).numpy()
    b = synth.gaussian_weights(1, N, seed + 2, std=1.0)[0].numpy() if bias else None
    qa, ea, _ = orc.quantize(x.float().numpy(), block, wa)
    qw, ew, _ = orc.quantize_2d(w, block, rows2, ww)
    return x, qa, ea, qw, ew, b


def _run(x, qw, ew, b, T, K, N, block, wa, ww, rows2, **more):
    y = torch.full((T, N + 4), -7.0, device="cuda")                       # ldy > N: nothing outside the result
    mxb.mx_linear(x.cuda(), mxb.MxFormat(block, wa), torch.from_numpy(orc.pack(qw, ww)).cuda(), torch.from_numpy(ew).cuda(),
                  mxb.MxFormat(block, ww, block_rows=rows2), N, bias=None if b is None else torch.from_numpy(b).cuda(), y=y[:, :N], **more)
    assert mxb.mx_poll_status() == 0
    assert (y[:, N:] == -7.0).all()
    return y[:, :N].cpu().numpy()


@pytest.mark.parametrize("T,K,N,block,wa,ww,rows2,dtype", [
    (1, 4096, 130, 32, 8, 4, 1, torch.float32),        # whole words of exponent bytes, a ragged last row tile
    (16, 4096, 272, 32, 8, 4, 1, torch.bfloat16),
    (9, 544, 37, 32, 8, 3, 1, torch.float32),          # K of whole 16-byte units only, odd rows of exponent bytes
    (5, 768, 768, 16, 4, 4, 1, torch.float32),         # nibbles in blocks of 16
    (8, 1056, 64, 16, 8, 2, 2, torch.bfloat16),        # ... that two rows share
    (2, 2048, 40, 16, 6, 6, 1, torch.float32),         # bytes in blocks of 16
    (16, 528, 129, 16, 8, 8, 1, torch.float32),        # ... K % 32 == 16
    (1, 16, 16, 16, 8, 8, 1, torch.float32),           # one unit
    (3, 32, 2, 32, 3, 4, 2, torch.float32),
    (16, 1312, 200, 32, 5, 8, 1, torch.bfloat16),      # bytes in blocks of 32, slices of odd groups
    (4, 8192, 4096, 16, 8, 8, 1, torch.float32),
    (12, 16384, 1536, 16, 4, 4, 1, torch.bfloat16),    # a long slice per CTA, several row groups per cluster
    (7, 160, 37900, 32, 8, 4, 1, torch.float32),       # so many rows that K is not cut
    (10, 96, 38000, 16, 8, 8, 1, torch.float32),
])
def test_few_tokens_in_one_launch(T, K, N, block, wa, ww, rows2, dtype):
    x, qa, ea, qw, ew, b = _case(T, K, N, block, wa, ww, rows2, dtype, bias=N % 3 == 1)
    y = _run(x, qw, ew, b, T, K, N, block, wa, ww, rows2)
    y_ref, y_seq, S = orc.gemm(qa, ea, wa, qw, orc.expand_exponent_rows(ew, rows2), ww, block, bias=b)
    err = np.abs(y.astype(np.float64) - y_ref)
    assert (err <= 1e-5 * S + 1e-37).all(), float((err / np.maximum(S, 1e-300)).max())
    if N >= 37889:                                     # 296 groups of 128 rows and more: one chain of ascending blocks
        assert np.array_equal(y, y_seq)


@pytest.mark.parametrize("block,ww", [(32, 4), (16, 4), (32, 8), (16, 8)])
def test_exponents_at_the_ends_of_the_range(block, ww):
    """Weight blocks with the exponent bytes 0, 225, 226, 254 and 255 (the rescale of two steps) and a non-finite token, K cut
    over a cluster.  The inputs keep every sum finite, so both sides agree on what is NaN."""
    T, K, N, wa = 6, 1024, 150, 8
    x, qa, ea, qw, ew, _ = _case(T, K, N, block, wa, ww, seed=5)
    x[2, 100] = float("nan")
    x[5] *= 2.0 ** -110
    qa, ea, _ = orc.quantize(x.numpy(), block, wa)
    ew[3, 1], ew[4, 2], ew[5, 3], ew[6, 0], ew[7, 4] = 0, 225, 226, 254, 255
    qw[3, block:2 * block] = 1
    for r, c in ((4, 2), (5, 3), (6, 0)):              # small mantissas there: |y| stays below the largest float
        qw[r, c * block:(c + 1) * block] = 0
        qw[r, c * block] = 1
    x[:2, :], x[3:5, :] = x[:2, :] * 2.0 ** -20, x[3:5, :] * 2.0 ** -20
    qa, ea, _ = orc.quantize(x.numpy(), block, wa)
    y = _run(x, qw, ew, None, T, K, N, block, wa, ww, 1)
    y_ref, _, S = orc.gemm(qa, ea, wa, qw, ew, ww, block)
    assert np.array_equal(np.isnan(y), np.isnan(y_ref))
    ok = ~np.isnan(y_ref)
    # subnormal sums: one step of 2^-149 per block beside the relative bound
    assert (np.abs(y[ok].astype(np.float64) - y_ref[ok]) <= 1e-5 * S[ok] + K / block * 2.0 ** -149).all()


@pytest.mark.parametrize("T", (3, 8, 11, 16))
def test_grouped_layers_of_many_shapes_bit_exact(T):
    """More rows than the warps of the chip, K of half a step to several, activations that change inside a CTA's range, two-row
    weight blocks: ascending blocks, the oracle's sequential sum."""
    layers, want = [], []
    for i, (K, N, rows2) in enumerate(((512, 8192, 1), (128, 8200, 1), (512, 4096, 2), (1152, 8192, 1), (640, 9000, 1), (1152, 37, 1))):
        x, qa, ea, qw, ew, b = _case(T, K, N, 32, 8 - i % 2, 4, rows2, bias=i == 1, seed=20 + i)
        layers.append(dict(x=x.cuda(), fa=mxb.MxFormat(32, 8 - i % 2), fw=mxb.MxFormat(32, 4, block_rows=rows2), N=N,
                           w_mant=torch.from_numpy(orc.pack(qw, 4)).cuda(), w_exp=torch.from_numpy(ew).cuda(),
                           bias=None if b is None else torch.from_numpy(b).cuda(), y=torch.empty(T, N, device="cuda")))
        want.append(orc.gemm(qa, ea, 8 - i % 2, qw, orc.expand_exponent_rows(ew, rows2), 4, 32, bias=b)[1])
    mxb.mx_linear_grouped(mxb.make_linear_args(layers))
    assert mxb.mx_poll_status() == 0
    for L, y_seq in zip(layers, want):
        assert np.array_equal(L["y"].cpu().numpy(), y_seq)


@pytest.mark.parametrize("T,K,N,block,ww", [(17, 768, 768, 16, 4), (32, 1056, 200, 32, 4), (24, 4096, 1030, 16, 8), (31, 2048, 4096, 32, 8),
                                            (20, 11008, 272, 32, 4)])
def test_up_to_32_tokens(T, K, N, block, ww):
    x, qa, ea, qw, ew, b = _case(T, K, N, block, 8, ww, seed=9, bias=True)
    y = _run(x, qw, ew, b, T, K, N, block, 8, ww, 1)
    y_ref, _, S = orc.gemm(qa, ea, 8, qw, ew, ww, block, bias=b)
    assert (np.abs(y.astype(np.float64) - y_ref) <= 1e-5 * S + 1e-37).all()


def test_a_tokens_bits_do_not_depend_on_the_others():
    """The cut of K is a function of the layer: every batch of up to 16 tokens gives a token the same bits."""
    K, N, block = 4096, 1500, 16
    x, _, _, qw, ew, _ = _case(16, K, N, block, 8, 8, seed=31)
    whole = _run(x, qw, ew, None, 16, K, N, block, 8, 8, 1)
    for t0, t1 in ((0, 1), (3, 8), (7, 16)):
        assert np.array_equal(_run(x[t0:t1].contiguous(), qw, ew, None, t1 - t0, K, N, block, 8, 8, 1), whole[t0:t1])


@pytest.mark.parametrize("T,K,N,block,ww", [(1, 768, 768, 16, 4), (4, 4096, 4096, 32, 4), (16, 2048, 2048, 16, 8), (24, 768, 768, 16, 4)])
def test_the_result_may_take_the_activations_place(T, K, N, block, ww):
    """y = x, rows of x that y starts later in, and two column ranges of one tensor: the activations are read before any
    result is written."""
    x, _, _, qw, ew, _ = _case(T, K, N, block, 8, ww, seed=41)
    fa, fw = mxb.MxFormat(block, 8), mxb.MxFormat(block, ww)
    wm, we = torch.from_numpy(orc.pack(qw, ww)).cuda(), torch.from_numpy(ew).cuda()
    S = x.abs().cuda().double() @ mxb.mx_dequantize(wm, we, K, fw).abs().double().t()
    want = mxb.mx_linear(x.cuda(), fa, wm, we, fw, N)
    for pitch, xc, yc in ((K, 0, 0), (2 * K, 0, K // 2), (2 * K, K // 2, 0), (2 * K, 0, K), (2 * K, K, 0)):
        buf = torch.zeros(T, pitch, device="cuda")
        xv, yv = buf[:, xc:xc + K], buf[:, yc:yc + N]
        xv.copy_(x)
        mxb.mx_linear(xv, fa, wm, we, fw, N, y=yv)
        assert ((yv - want).abs().double() <= 1e-5 * S).all()
        if abs(xc - yc) == K:
            assert torch.equal(yv, want) and torch.equal(xv, x.cuda())
    assert mxb.mx_poll_status() == 0


def _spread(x, block):
    """Blocks up to 18 binades apart: their terms round when they are added, so that another order gives other bits."""
    g = torch.Generator().manual_seed(7)
    return x * torch.exp2(torch.randint(-9, 10, (x.shape[0], x.shape[1] // block), generator=g).float()).repeat_interleave(block, dim=1)


@pytest.mark.parametrize("T", (1, 2, 4, 16))
def test_named_stream_and_grouped_calls_keep_their_chain(T):
    """K = 1152 has no whole pieces: one chain of ascending blocks, the CUDA-core kernel's bits, whatever AUTO does with the layer.
    K = 4096 is cut over the warps of a CTA, the same way whether the tokens come packed or not."""
    N = 4096
    for K in (1152, 4096):
        x, _, _, qw, ew, _ = _case(T, K, N, 32, 8, 4, seed=51)
        x = _spread(x, 32)
        fa, fw, xd = mxb.MxFormat(32, 8), mxb.MxFormat(32, 4), x.cuda()
        wm, we = torch.from_numpy(orc.pack(qw, 4)).cuda(), torch.from_numpy(ew).cuda()
        y = mxb.mx_linear(xd, fa, wm, we, fw, N, algo=mxb.MX_ALGO_STREAM)
        if K == 1152:
            assert torch.equal(y, mxb.mx_linear(xd, fa, wm, we, fw, N, algo=mxb.MX_ALGO_SIMT))
        am, ae = mxb.mx_quantize(xd, fa)
        assert torch.equal(y, mxb.mx_gemm(am, ae, fa, wm, we, fw, T, N, K, algo=mxb.MX_ALGO_STREAM))
        g = torch.empty(T, N, device="cuda")
        mxb.mx_linear_grouped(mxb.make_linear_args([dict(x=xd, fa=fa, w_mant=wm, w_exp=we, fw=fw, N=N, y=g)]))
        assert torch.equal(y, g)
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("K,N,least", [(4096, 1500, 1), (8192, 4100, 2)])        # 4100 * 8192 > 2^25: one token goes its own way
def test_bits_of_a_token_among_others_in_4_bits(K, N, least):
    x, _, _, qw, ew, _ = _case(16, K, N, 32, 8, 4, seed=33)
    x = _spread(x, 32)
    whole = _run(x, qw, ew, None, 16, K, N, 32, 8, 4, 1)
    for t0, t1 in ((0, 1), (2, 4), (3, 8), (7, 16)):
        if t1 - t0 >= least:
            assert np.array_equal(_run(x[t0:t1].contiguous(), qw, ew, None, t1 - t0, K, N, 32, 8, 4, 1), whole[t0:t1])
