"""GPU parity of the block-scaled product on records (mantissa widths up to 5 on both sides, blocks of 16 and 32): the
route of mx_linear / mx_gemm and their fused and MXInt-result forms where there are too many 128 x 128 tiles to cut K (more
than 74), from K = 2048 or 4 M operand elements on.  Calls of fewer tiles take the product whose K is cut, here as well."""
import numpy as np
import pytest
import torch

from oracle import mx_oracle as orc
from paper_2307_15517_b200 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def mxb():
    from paper_2307_15517_b200 import binding
    return binding


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _framed(M, N):
    big = torch.full((M + 3, N + 8), -77.0, device="cuda")
    return big[:M, :N], lambda: bool((big[M:] == -77.0).all()) and bool((big[:, N:] == -77.0).all())


def _poison_free(mxb):
    assert mxb.mx_poll_status() == 0


# records: one row panel / one and a bit / two CTAs' worth; one record step of K, a remainder of 32, of 64; odd and even
# numbers of panels of W; N odd in every unit of the stores; a wide result behind a short reduction
SHAPES = [(17, 8450, 2080, 32, 4, 4, 1, "fp32"), (128, 9602, 2080, 16, 5, 5, 1, "bf16"), (129, 5002, 2176, 16, 4, 3, 1, "fp32"),
          (300, 3201, 2336, 16, 2, 4, 1, "fp32"), (256, 4864, 2080, 32, 5, 2, 2, "fp32"), (386, 2562, 2080, 16, 3, 5, 2, "bf16"),
          (100, 8195, 544, 16, 4, 4, 1, "fp32"), (2100, 2330, 2048, 32, 5, 5, 1, "fp32")]
# narrow mantissas in few tiles: K is cut
SHAPES += [(17, 130, 2048, 32, 4, 4, 1, "fp32"), (128, 256, 2080, 16, 5, 5, 1, "bf16"), (129, 258, 2176, 16, 4, 3, 1, "fp32"),
           (300, 385, 2336, 16, 2, 4, 1, "fp32"), (256, 512, 2080, 32, 5, 2, 2, "fp32"), (386, 514, 2080, 16, 3, 5, 2, "bf16"),
           (100, 6147, 544, 16, 4, 4, 1, "fp32")]


@pytest.mark.parametrize("shape", SHAPES)
def test_layer_and_product_within_tolerance(mxb, shape):
    M, N, K, B, wa, ww, rows2, dt = shape
    x = synth.student_t_activations(M, K, M).to(torch.bfloat16 if dt == "bf16" else torch.float32)
    x[M // 2, :64] = 0.0
    w, bias = synth.gaussian_weights(N, K, N), synth.gaussian_weights(1, N, 5)[0]
    qa, ea, _ = orc.quantize_2d(x.float().numpy(), B, rows2, wa)
    qw, ew, _ = orc.quantize_2d(w.numpy(), B, rows2, ww)
    y_ref, _, S = orc.gemm(qa, orc.expand_exponent_rows(ea, rows2), wa, qw, orc.expand_exponent_rows(ew, rows2), ww, B,
                           bias=bias.numpy())
    fa, fw = mxb.MxFormat(B, wa, block_rows=rows2), mxb.MxFormat(B, ww, block_rows=rows2)
    wm, we = _dev(orc.pack(qw, ww)), _dev(ew)
    for form in ("linear", "gemm"):
        y, intact = _framed(M, N)
        if form == "linear":
            mxb.mx_linear(x.cuda(), fa, wm, we, fw, N, bias=bias.cuda(), y=y)
        else:
            mxb.mx_gemm(_dev(orc.pack(qa, wa)), _dev(ea), fa, wm, we, fw, M, N, K, bias=bias.cuda(), y=y)
        _poison_free(mxb)
        err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
        assert (err <= TOL * (S + np.abs(bias.numpy())) + 1e-37).all(), (form, float((err / S).max()))
        assert intact()


@pytest.mark.parametrize("N", (5000, 300))         # records; K cut
@pytest.mark.parametrize("B", (16, 32))
def test_any_exponents_are_exact(mxb, B, N):
    """Exponent bytes anywhere, -2^(w-1) and zero groups included, on operands whose sums are exact in any order: the
    blocks of a row that meet nonzero weights share one exponent, the others lie up to 60 binades away."""
    M, K, wa, ww = 200, 2080, 4, 5
    rng = np.random.default_rng(B)
    qa = rng.integers(-8, 8, (M, K)).astype(np.int8)
    qw = rng.integers(-16, 16, (N, K)).astype(np.int8)
    nb = K // B
    keep = rng.random(nb) < 0.5                  # blocks of K where the weights are not zero
    qw[:, ~np.repeat(keep, B)] = 0
    ea = rng.integers(100, 160, (M, nb)).astype(np.uint8)
    ea[:, keep] = rng.integers(100, 160, (M, 1))
    ew = rng.integers(100, 160, (N, nb)).astype(np.uint8)        # exponents of zero blocks do not matter
    ew[:, keep] = rng.integers(100, 160, (N, 1))
    y_ref, y_seq, _ = orc.gemm(qa, ea, wa, qw, ew, ww, B)
    assert np.array_equal(y_ref, y_seq)
    fa, fw = mxb.MxFormat(B, wa), mxb.MxFormat(B, ww)
    wm, we = _dev(orc.pack(qw, ww)), _dev(ew)
    y = mxb.mx_gemm(_dev(orc.pack(qa, wa)), _dev(ea), fa, wm, we, fw, M, N, K)
    _poison_free(mxb)
    assert np.array_equal(y.cpu().numpy(), y_ref)
    # the layer: the same values as floating-point activations (-8 is no quantizer output: the grid below it)
    qa2 = np.clip(qa, -7, 7)
    qa2[:, ::B] = 7                              # a block's exponent is that of its largest value
    y_ref, y_seq, _ = orc.gemm(qa2, ea, wa, qw, ew, ww, B)
    assert np.array_equal(y_ref, y_seq)
    x = orc.dequantize(qa2, ea, B, wa).astype(np.float32)
    y = mxb.mx_linear(_dev(x), fa, wm, we, fw, N)
    _poison_free(mxb)
    assert np.array_equal(y.cpu().numpy(), y_ref)
    # a block that held Inf/NaN poisons its row or column, and nothing else
    ea2, ew2 = ea.copy(), ew.copy()
    ea2[5, 3] = ew2[11, 1] = 255
    qz, qwz = qa2.copy(), qw.copy()
    qz[5, 3 * B:4 * B] = 0
    qwz[11, B:2 * B] = 0
    want = np.zeros((M, N), bool)
    want[5], want[:, 11] = True, True
    x[5, 3 * B + 2] = np.inf
    wm, we = _dev(orc.pack(qwz, ww)), _dev(ew2)
    for y in (mxb.mx_gemm(_dev(orc.pack(qz, wa)), _dev(ea2), fa, wm, we, fw, M, N, K), mxb.mx_linear(_dev(x), fa, wm, we, fw, N)):
        _poison_free(mxb)
        y = y.cpu().numpy()
        assert np.array_equal(np.isnan(y), want)
        assert np.array_equal(y[~want], y_ref[~want])


@pytest.mark.parametrize("N", (5000, 260))         # records; K cut
def test_general_operands_far_apart(mxb, N):
    """Every block with an exponent of its own, +-20 binades: each MMA step cuts its addends (16 products and the
    accumulator) at the ulp of the largest, so K/16 steps stay within K/16 * 17 * 2^-23 of S."""
    M, K, B = 150, 2144, 16
    x = synth.student_t_activations(M, K, 1).numpy() * np.ldexp(1.0, np.random.default_rng(1).integers(-20, 21, (M, K // B))).repeat(B, 1)
    w = synth.gaussian_weights(N, K, 2).numpy() * np.ldexp(1.0, np.random.default_rng(2).integers(-20, 21, (N, K // B))).repeat(B, 1)
    x, w = x.astype(np.float32), w.astype(np.float32)
    qa, ea, _ = orc.quantize(x, B, 5)
    qw, ew, _ = orc.quantize(w, B, 4)
    y_ref, _, S = orc.gemm(qa, ea, 5, qw, ew, 4, B)
    y = mxb.mx_linear(_dev(x), mxb.MxFormat(B, 5), _dev(orc.pack(qw, 4)), _dev(ew), mxb.MxFormat(B, 4), N)
    _poison_free(mxb)
    assert (np.abs(y.cpu().numpy().astype(np.float64) - y_ref) <= K / 16 * 17 * 2.0 ** -23 * S).all()


@pytest.mark.parametrize("shape", [(150, 5024, 2080, 16), (300, 4128, 2048, 32), (150, 288, 2080, 16), (300, 544, 2048, 32)])
def test_fused_tail_and_mxint_result_are_the_plain_result_passed_on(mxb, shape):
    M, N, K, B = shape
    fa, fw = mxb.MxFormat(B, 4), mxb.MxFormat(B, 4)
    x = synth.student_t_activations(M, K, 3).cuda()
    wm, we = mxb.mx_quantize(synth.gaussian_weights(N, K, 4).cuda(), fw)
    am, ae = mxb.mx_quantize(x, fa)
    bias, res = synth.gaussian_weights(1, N, 5)[0].cuda(), synth.gaussian_weights(M, N, 6).cuda()
    y = mxb.mx_linear(x, fa, wm, we, fw, N)
    tail = torch.relu(y + bias) + res
    assert torch.equal(mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res), tail)
    assert torch.equal(mxb.mx_gemm_fused(am, ae, fa, wm, we, fw, M, N, K, bias=bias, relu=True, residual=res), tail)
    for w_out in (4, 8):
        fy = mxb.MxFormat(B, w_out)
        for got, src in ((mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias), y + bias),
                         (mxb.mx_gemm_q(am, ae, fa, wm, we, fw, M, N, K, fy), y),
                         (mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res, fy=fy), tail)):
            want = mxb.mx_quantize(src, fy)
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    _poison_free(mxb)


@pytest.mark.parametrize("shape", [(64, 256, 8192), (200, 512, 4096), (1, 1024, 4096)])
def test_few_tiles_take_the_cut_reduction_whatever_the_width(mxb, shape):
    """The same values in 4-bit and in 6-bit containers (exponent byte + 2 for the two more fraction bits).  Few tiles and a
    long K: both calls must run the product whose K is cut, so their sums are rounded alike, bit for bit; the block exponents
    are spread so that another order of the sum shows."""
    M, N, K = shape
    B = 16
    rng = np.random.default_rng(K)
    qa, qw = rng.integers(-7, 8, (M, K)).astype(np.int8), rng.integers(-7, 8, (N, K)).astype(np.int8)
    ea = rng.integers(121, 134, (M, K // B)).astype(np.uint8)
    ew = rng.integers(121, 134, (N, K // B)).astype(np.uint8)
    y = [mxb.mx_gemm(_dev(orc.pack(qa, w)), _dev(ea + np.uint8(w - 4)), mxb.MxFormat(B, w), _dev(orc.pack(qw, w)),
                     _dev(ew + np.uint8(w - 4)), mxb.MxFormat(B, w), M, N, K) for w in (4, 6)]
    _poison_free(mxb)
    assert torch.equal(y[0], y[1])
    chain = mxb.mx_gemm(_dev(orc.pack(qa, 4)), _dev(ea), mxb.MxFormat(B, 4), _dev(orc.pack(qw, 4)), _dev(ew),
                        mxb.MxFormat(B, 4), M, N, K, algo=mxb.MX_ALGO_TCGEN05)
    assert not torch.equal(y[0], chain)


@pytest.mark.parametrize("form", ("gemm", "linear"))
def test_wide_steps_between_narrow_ones(mxb, form):
    """Single K steps with scales per half block between steps with one scale per row: right before and after each other, at
    and around a step that reloads the scales of four (multiples of 4), at both sides of the 32 steps that one look at the
    flags covers, at the end of a tile; in some panels of A and of W only, with up to three tiles per CTA pair.  Codes of at
    most 3 with exponents 0 to 3 binades above one unit: every sum is exact in any order (9 * 4480 * 2^6 < 2^24)."""
    M, N, K, B, w = 1280, 7936, 4480, 16, 4                # 155 tiles of 256 x 256, 35 steps
    steps = K // 128
    g = torch.Generator().manual_seed(11)
    sides = []
    for rows, zero, wild, where in ((M, 1, 0, {130: (1, 5, 31, 32), 600: (2,), 1000: (5, 7, 8, 33, 34)}),
                                    (N, 0, 1, {77: (2, 31, 34), 5000: (2, 3, 4, 28, 31, 32), 7900: (33,)})):
        q = torch.randint(-3, 4, (rows, steps, 8, B), generator=g, dtype=torch.int8)
        e = torch.randint(0, 4, (rows, steps, 8), generator=g) + 125
        q[:, :, zero] = 0                                 # what the other side has there does not count
        for row, kbs in where.items():
            for kb in kbs:
                q[row, kb, wild] = 3
                e[row, kb, wild] = 125 - 40
        q, e = q.view(rows, K), e.view(rows, K // B)
        value = q.double() * torch.exp2((e - 127 - (w - 2)).double()).repeat_interleave(B, 1)
        sides.append((_dev(orc.pack(q.numpy(), w)), e.to(torch.uint8).cuda(), value.cuda()))
    (am, ae, a), (wm, we, b) = sides
    f = mxb.MxFormat(B, w)
    want = (a @ b.t()).float()
    if form == "gemm":
        y = mxb.mx_gemm(am, ae, f, wm, we, f, M, N, K)
    else:
        y = mxb.mx_linear(a.float(), f, wm, we, f, N)     # every value is on the grid of its block's own exponent
    _poison_free(mxb)
    assert torch.equal(y, want)


def test_narrow_steps_of_blocks_twelve_binades_apart(mxb):
    """Block exponents anywhere within the 12 binades that one scale per row and 128 k can span: no step is wide.  The pipe
    aligns the 32 products of a step and the accumulator to the largest and truncates: bounded here by one unit in the last
    place of S per step, 8.0e-6; measured 1.9e-6 (2.1e-6 for the bf16 chain)."""
    M, N, K, B, wa, ww = 150, 5000, 2144, 16, 5, 4
    rng = np.random.default_rng(3)
    qa, qw = rng.integers(-15, 16, (M, K)).astype(np.int8), rng.integers(-7, 8, (N, K)).astype(np.int8)
    ea, ew = (rng.integers(121, 134, (rows, K // B)).astype(np.uint8) for rows in (M, N))
    fa, fw = mxb.MxFormat(B, wa), mxb.MxFormat(B, ww)
    args = (_dev(orc.pack(qa, wa)), _dev(ea), fa, _dev(orc.pack(qw, ww)), _dev(ew), fw, M, N, K)
    y = mxb.mx_gemm(*args)
    _poison_free(mxb)
    y_ref, _, S = orc.gemm(qa, ea, wa, qw, ew, ww, B)
    err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref) / S
    assert err.max() <= K / 32 * 2.0 ** -23
