"""GPU parity of the product whose reduction is cut over the CTAs of a cluster (few 128 x 128 tiles, K from 1024 on, a
mantissa of more than 5 bits): two, three and four pieces, ragged tiles, every kind of result."""
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


# tiles 1, 4 (four pieces, K steps that do not divide), 18 (four), 42 (three or two), 60 (two; not cut), a K remainder of 32
SHAPES = [(17, 100, 1024, 16, 8, 4), (200, 131, 1120, 32, 6, 6), (130, 1056, 1552, 16, 8, 4), (300, 1790, 2064, 16, 8, 8),
          (250, 3840, 2080, 32, 8, 6), (250, 3840, 1568, 32, 8, 6)]


@pytest.mark.parametrize("shape", SHAPES)
def test_split_product_within_tolerance(mxb, shape):
    M, N, K, B, wa, ww = shape
    x, w, bias = synth.student_t_activations(M, K, M), synth.gaussian_weights(N, K, N), synth.gaussian_weights(1, N, 5)[0]
    qa, ea, _ = orc.quantize(x.numpy(), B, wa)
    qw, ew, _ = orc.quantize(w.numpy(), B, ww)
    y_ref, _, S = orc.gemm(qa, ea, wa, qw, ew, ww, B, bias=bias.numpy())
    fa, fw = mxb.MxFormat(B, wa), mxb.MxFormat(B, ww)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()             # noqa: E731
    wm, we = dev(orc.pack(qw, ww)), dev(ew)
    big = torch.full((M + 3, N + 8), -77.0, device="cuda")
    y = big[:M, :N]
    mxb.mx_linear(x.cuda(), fa, wm, we, fw, N, bias=bias.cuda(), y=y)
    assert mxb.mx_poll_status() == 0
    err = np.abs(y.cpu().numpy().astype(np.float64) - y_ref)
    assert (err <= TOL * (S + np.abs(bias.numpy()))).all(), float((err / S).max())
    assert bool((big[M:] == -77.0).all()) and bool((big[:, N:] == -77.0).all())


@pytest.mark.parametrize("shape", [(200, 160, 1120, 32), (130, 1056, 1552, 16), (130, 1056, 1040, 16), (300, 1792, 2064, 16),
                                   (250, 3840, 2080, 32)])
def test_fused_tail_and_mxint_result_of_a_split_product(mxb, shape):
    """Operands whose sums are exact in any order (4-bit mantissas, one exponent per operand; 6-bit containers keep the
    call on this route): every form must equal the oracle's value carried on in fp32."""
    M, N, K, B = shape
    rng = np.random.default_rng(N)
    qa, qw = rng.integers(-7, 8, (M, K)).astype(np.int8), rng.integers(-7, 8, (N, K)).astype(np.int8)
    ea, ew = np.full((M, K // B), 127, np.uint8), np.full((N, K // B), 125, np.uint8)
    y_ref, y_seq, _ = orc.gemm(qa, ea, 6, qw, ew, 6, B)
    assert np.array_equal(y_ref, y_seq)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()             # noqa: E731
    f = mxb.MxFormat(B, 6)
    args = (dev(orc.pack(qa, 6)), dev(ea), f, dev(orc.pack(qw, 6)), dev(ew), f, M, N, K)
    y = dev(y_ref)
    assert torch.equal(mxb.mx_gemm(*args), y)
    bias, res = synth.gaussian_weights(1, N, 5)[0].cuda(), synth.gaussian_weights(M, N, 6).cuda()
    tail = torch.relu(y + bias) + res
    assert torch.equal(mxb.mx_gemm_fused(*args, bias=bias, relu=True, residual=res), tail)
    fy = mxb.MxFormat(B, 8)
    for got, src in ((mxb.mx_gemm_q(*args, fy, bias=bias), y + bias),
                     (mxb.mx_gemm_fused(*args, bias=bias, relu=True, residual=res, fy=fy), tail)):
        want = mxb.mx_quantize(src, fy)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert mxb.mx_poll_status() == 0


def test_an_item_does_not_depend_on_the_number_of_items(mxb):
    """mx_gemm_batched of the first item alone and of both: the same bits, and those of the product that never cuts K, on
    operands (block exponents 24 binades apart) whose sums show their order."""
    M, N, K, B = 200, 131, 1120, 16
    rng = np.random.default_rng(7)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()             # noqa: E731
    f = mxb.MxFormat(B, 8)
    qa, qw = rng.integers(-127, 128, (M, 2 * K)).astype(np.int8), rng.integers(-127, 128, (N, 2 * K)).astype(np.int8)
    ea, ew = (rng.integers(115, 140, (rows, 2 * K // B)).astype(np.uint8) for rows in (M, N))
    am, wm = dev(orc.pack(qa, 8)), dev(orc.pack(qw, 8))
    y = [torch.zeros(n * M, N, device="cuda") for n in (1, 2)]
    for n in (1, 2):
        mxb.mx_gemm_batched(am, dev(ea), f, 2 * K, K, wm, dev(ew), f, 2 * K, K, M, N, K, n, y[n - 1], N, M * N)
    assert mxb.mx_poll_status() == 0
    assert torch.equal(y[0], y[1][:M])
    first = [dev(a[:, :a.shape[1] // 2]) for a in (orc.pack(qa, 8), ea, orc.pack(qw, 8), ew)]
    chain = mxb.mx_gemm(first[0], first[1], f, first[2], first[3], f, M, N, K, algo=mxb.MX_ALGO_TCGEN05)
    assert torch.equal(y[0], chain)
