"""The product on wide CTA-pair tiles: the bits of narrow calls (one-CTA kernel) over slices of the weights, for shapes whose
tiles are cut by the last row, the last column and the last K step; the fused tail and the MXInt result from the same sums."""
import pytest
import torch

from paper_2307_15517_b200 import binding as mxb

pytestmark = pytest.mark.gpu


def _operands(M, N, K, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    fa, fw = mxb.MxFormat(16, 8), mxb.MxFormat(16, 4)
    x = torch.randn(M, K, generator=g, device="cuda")
    wm, we = mxb.mx_quantize(torch.randn(N, K, generator=g, device="cuda") * 0.02, fw)
    return g, x, fa, wm, we, fw


# 8-bit activations: bf16 operands.  256 x 256 tiles would take two rounds of 74 pairs, 256 x {320, 352, 448} ones take one
@pytest.mark.parametrize("M,N,K", [(500, 11008, 4096), (512, 10976, 1056), (700, 8160, 2064), (300, 16352, 8192), (512, 10001, 2048)])
def test_wide_tiles_have_the_bits_of_narrow_calls(M, N, K):
    g, x, fa, wm, we, fw = _operands(M, N, K, M + N)
    bias = torch.randn(N, generator=g, device="cuda")
    y = torch.full((M, N + 5), -3.0, device="cuda")                       # (odd row length: stores of single values)
    mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y[:, :N])
    want = torch.empty(M, N, device="cuda")
    for n in range(0, N, 1024):
        cols = min(1024, N - n)
        want[:, n:n + cols] = mxb.mx_linear(x, fa, wm[n:n + cols], we[n:n + cols], fw, cols, bias=bias[n:n + cols].clone(),
                                            algo=mxb.MX_ALGO_TCGEN05)
    assert mxb.mx_poll_status() == 0
    assert torch.equal(y[:, :N], want) and (y[:, N:] == -3.0).all()
    res = torch.randn(M, N, generator=g, device="cuda")
    z = mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res)
    assert torch.equal(z, torch.relu(want) + res)
    if N % 16 == 0:
        for fy in (mxb.MxFormat(16, 8), mxb.MxFormat(32 if N % 32 == 0 else 16, 4)):
            ym, ye = mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias)
            qm, qe = mxb.mx_quantize(want, fy)
            assert torch.equal(ym, qm) and torch.equal(ye, qe)
            zm, ze = mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res, fy=fy)
            qm, qe = mxb.mx_quantize(z, fy)
            assert torch.equal(zm, qm) and torch.equal(ze, qe)
    assert mxb.mx_poll_status() == 0
