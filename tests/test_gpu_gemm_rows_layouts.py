"""The weight-streaming kernel over its layouts: 8 to 112 weight rows per CTA (16-row blocks with and without their second half,
a last CTA with few rows), one to eight K ranges, one to four token tiles, every group size, blocks of 32 tokens.

The reference is the fp64 product of the decoded operands; products are exact, so what is left is the fp32 accumulation, below
K 2^-24 of the sum of magnitudes - taken as 1e-5 of the result's norm, as for this kernel elsewhere."""
import pytest
import torch

from paper_2411_09909_b200 import amx

pytestmark = pytest.mark.gpu

SHAPES = [(1, 14331, 1024), (8, 4096, 2048), (1, 520, 4096), (16, 9597, 1152), (16, 5120, 640), (24, 14336, 512), (24, 11003, 1024),
          (24, 6144, 1024), (20, 1500, 4096), (32, 14330, 640), (32, 12281, 512), (32, 2500, 2304), (12, 700, 3072), (31, 1024, 8192),
          (128, 1024, 1024), (200, 800, 512),
          # K ranges, and rows of a CTA in between
          (15, 65, 8192), (15, 1063, 5248), (8, 121, 8320), (10, 2647, 11776), (24, 1217, 7424), (12, 568, 8192), (13, 1327, 7296),
          (13, 5993, 512), (31, 4755, 7424), (17, 1061, 14720), (18, 13039, 512), (24, 15413, 512)]


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_layouts(M, N, K, gs):
    g = torch.Generator(device="cuda").manual_seed(M + N + K + gs)
    x = (torch.randn(M, K, device="cuda", generator=g) + 0.2).to(torch.bfloat16)
    w = (0.02 * torch.randn(N, K, device="cuda", generator=g)).to(torch.bfloat16)
    (ac, as_), (wc, ws) = amx.quantize(x, gs), amx.quantize(w, gs)
    assert amx.lib().amx_gemm_kernel_for(M, N, K, gs, amx.GEMM_AUTO) == amx.GEMM_ROWS
    wide = torch.full((M, N + 3), 5.0, dtype=torch.float32, device="cuda")
    got = amx.quant_gemm(x, wc, ws, gs, out=wide[:, :N])
    assert torch.all(wide[:, N:] == 5.0)
    ref = amx.dequantize(ac, as_, gs, torch.float32).double() @ amx.dequantize(wc, ws, gs, torch.float32).double().T
    assert float((got.double() - ref).norm() / ref.norm()) <= 1e-5
    assert torch.equal(amx.gemm(ac, as_, wc, ws, gs), got.contiguous())
