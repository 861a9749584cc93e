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


def _width(M, N, K, pairs=74):
    """The host's rule for the width of the pair tiles (0: 256), restated: it decides what the shapes below run."""
    rows = (M + 255) // 256
    rounds = lambda w: (rows * ((N + w - 1) // w) + pairs - 1) // pairs      # noqa: E731
    tile, width = K * 29 // 5, 0
    best = (6000 + rounds(256) * tile) * 93 // 100
    for w in range(288, 513, 32):
        ns = 2000 + rounds(w) * (tile * max(w, 384) * 9 // 2560 + w * 75 // 4)
        if ns < best:
            best, width = ns, w
    return width


# more than 384 rows, so that no other kernel takes them; every width that the rule picks, ragged in M, N and K
@pytest.mark.parametrize("M,N,K,width", [(414, 9686, 1040, 288), (521, 7662, 1040, 320), (528, 7936, 1040, 352), (516, 8680, 2064, 384),
                                         (524, 9240, 2064, 416), (516, 10184, 4112, 448), (2040, 4080, 16400, 480)])
def test_every_width_has_the_bits_of_narrow_calls(M, N, K, width):
    assert torch.cuda.get_device_properties(0).multi_processor_count != 148 or _width(M, N, K) == width
    g, x, fa, wm, we, fw = _operands(M, N, K, M + N)
    bias = torch.randn(N, generator=g, device="cuda")
    y = mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, algo=mxb.MX_ALGO_TCGEN05)
    for n in range(0, N, 1024):
        cols = min(1024, N - n)
        assert torch.equal(y[:, n:n + cols], mxb.mx_linear(x, fa, wm[n:n + cols], we[n:n + cols], fw, cols, bias=bias[n:n + cols].clone(),
                                                           algo=mxb.MX_ALGO_TCGEN05))
    res = torch.randn(M, N, generator=g, device="cuda")
    assert torch.equal(mxb.mx_linear_fused(x, fa, wm, we, fw, N, bias=bias, relu=True, residual=res), torch.relu(y) + res)
    if N % 16 == 0:
        fy = mxb.MxFormat(16, 8)
        ym, ye = mxb.mx_linear_q(x, fa, wm, we, fw, N, fy, bias=bias)
        qm, qe = mxb.mx_quantize(y, fy)
        assert torch.equal(ym, qm) and torch.equal(ye, qe)
    assert mxb.mx_poll_status() == 0


def test_exponents_at_the_ends_of_the_range_on_wide_tiles():
    from tests.test_gpu_dec import check_ends_of_the_range
    check_ends_of_the_range(414, 1040, 9686, 16, 4)


# one round of tiles narrower than 256 columns: 224, 192 and 160 on 148 SMs, ragged in M, N and K
@pytest.mark.parametrize("M,N,K", [(1237, 3002, 2080), (760, 4600, 1040), (1530, 1900, 528), (250, 11008, 1040)])
def test_one_round_of_narrow_pair_tiles_has_the_bits_of_narrow_calls(M, N, K):
    g, x, fa, wm, we, fw = _operands(M, N, K, M + N)
    bias = torch.randn(N, generator=g, device="cuda")
    y = torch.full((M, N + 5), -3.0, device="cuda")
    mxb.mx_linear(x, fa, wm, we, fw, N, bias=bias, y=y[:, :N], algo=mxb.MX_ALGO_TCGEN05)
    for n in range(0, N, 512):
        cols = min(512, N - n)
        assert torch.equal(y[:, n:n + cols], mxb.mx_linear(x, fa, wm[n:n + cols], we[n:n + cols], fw, cols, bias=bias[n:n + cols].clone(),
                                                           algo=mxb.MX_ALGO_TCGEN05))
    assert (y[:, N:] == -3.0).all()
    assert mxb.mx_poll_status() == 0


@pytest.mark.parametrize("M,N,K,kernel,width", [
    (384, 6144, 2048, 5, 128), (384, 6144, 4096, 5, 128), (384, 5120, 5120, 5, 128),       # 144 and 120 tiles of 128 x 128
    (385, 6144, 2048, 7, 192), (250, 11008, 1040, 7, 160), (256, 9472, 2048, 5, 128), (256, 9600, 2048, 7, 160),
    (640, 4096, 256, 5, 256), (640, 4096, 320, 7, 192), (300, 6464, 96, 5, 256),                # few K steps
    (2048, 1408, 256, 7, 160), (2048, 1408, 240, 5, 256)])
def test_narrow_pair_tiles_only_where_they_are_faster(M, N, K, kernel, width):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("sizes for 148 SMs")
    assert mxb.mx_selftest_route(M, N, K, mxb.MxFormat(16, 8), mxb.MxFormat(16, 4), algo=mxb.MX_ALGO_TCGEN05)[:2] == (kernel, width)
