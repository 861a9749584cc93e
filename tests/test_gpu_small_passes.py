"""The quantizer along the slow axis at the edges of its items (32 rows x 32 k) and the launches of few items, which take one item
per warp and a dense tensor of short rows as one long row, against the CPU oracle: bit for bit."""
import numpy as np
import pytest
import torch

from oracle import mx_oracle as orc
from paper_2307_15517_b200 import binding as mxb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,K,B,w,dtype", [
    (2, 32, 32, 8, torch.float32), (31, 32, 16, 4, torch.bfloat16), (33, 96, 32, 5, torch.float32), (64, 4096, 16, 3, torch.bfloat16),
    (2049, 352, 32, 8, torch.bfloat16), (1000, 1056, 16, 4, torch.float32),
])
def test_blocks_along_the_slow_axis(rows, K, B, w, dtype):
    g = torch.Generator().manual_seed(rows + K)
    v = (torch.randn(K, rows, generator=g) * torch.exp2(torch.randint(-20, 20, (1, rows), generator=g).float())).to(dtype)
    v[0, 0], v[K - 1, rows - 1] = float("nan"), float("-inf")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    mant, exps = mxb.mx_quantize(v.cuda().t(), mxb.MxFormat(B, w), nonfinite_count=cnt)
    q, e, bad = orc.quantize(np.ascontiguousarray(v.float().numpy().T), B, w)
    assert np.array_equal(mant.cpu().numpy(), orc.pack(q, w)) and np.array_equal(exps.cpu().numpy(), e) and int(cnt) == bad


@pytest.mark.parametrize("rows,K", [(1, 32), (2, 992), (33, 352), (352, 1056), (147, 2048), (148, 4096), (149, 4128), (4097, 96),
                                    (7104, 64), (7105, 64), (13024, 32), (13025, 32)])
@pytest.mark.parametrize("B,w,dtype", [(16, 4, torch.float32), (32, 8, torch.bfloat16)])
def test_few_items(rows, K, B, w, dtype):
    """Both sides of the lines: 148 x 512 chunks of 8, or of 148 x 48 rows and 148 x 352 chunks (quantizer) and 148 x 256 items of 32 (decoder) on 148 SMs."""
    g = torch.Generator().manual_seed(rows + K)
    x = (torch.randn(rows, K, generator=g) * torch.exp2(torch.randint(-20, 20, (rows, 1), generator=g).float())).to(dtype)
    f = mxb.MxFormat(B, w)
    mant, exps = mxb.mx_quantize(x.cuda(), f)
    q, e, _ = orc.quantize(x.float().numpy(), B, w)
    assert np.array_equal(mant.cpu().numpy(), orc.pack(q, w)) and np.array_equal(exps.cpu().numpy(), e)
    out = torch.full((rows + 2, K), -7.0, dtype=torch.bfloat16, device="cuda")
    got = mxb.mx_dequantize(mant, exps, K, f, dtype=torch.bfloat16)
    want = torch.from_numpy(orc.dequantize(q, e, B, w)).to(torch.bfloat16)
    assert torch.equal(got.cpu(), want)
    mxb._check(mxb.lib.mx_dequantize(mant.data_ptr(), exps.data_ptr(), rows, K, f, out[1:-1].data_ptr(), mxb.MX_BF16, K,
                                     torch.cuda.current_stream().cuda_stream), "mx_dequantize")
    assert torch.equal(out[1:-1].cpu(), want) and (out[0] == -7).all() and (out[-1] == -7).all()
