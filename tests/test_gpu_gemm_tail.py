"""GPU parity of the FP4 GEMM where the last wave's tiles are cut into halves or quarters of their columns: one CTA and pairs
of CTAs per tile, with and without whole waves before, one and two planes, fp32 and bf16 results, ragged edges.

The reference is the fp64 product of the decoded operands.  Decoded values are exact and so are the products; what is left is
the fp32 accumulation: K terms, relative to the sum of their magnitudes below K 2^-24 - taken here as 2^-12 of the result's norm
(inputs without cancellation of whole rows), and 2^-8 for a result rounded to bf16."""
import pytest
import torch

from paper_2411_09909_b200 import amx

pytestmark = pytest.mark.gpu

# (M, N): 128 x 256 tiles on 148 SMs, pairs of 256 x 256 on 74 from 149 tiles on
SHAPES = [
    (128, 256),        # one tile: quarters
    (130, 4700),       # 2 x 19 tiles: 38 -> quarters, the last one 36 columns wide
    (500, 4096),       # 4 x 16 = 64 tiles: halves
    (1000, 4096),      # 8 x 16 = 128 tiles: whole
    (1000, 4900),      # 8 x 20 = 160 tiles, 80 in pairs: a wave and 6 tiles in quarters
    (1920, 2816),      # 15 x 11 = 165 tiles, 88 in pairs (the last row block alone): a wave and 14 tiles in quarters
    (1100, 5400),      # 9 x 22 = 198 tiles (no pairs): a wave and 50 tiles in halves
    (2048, 3328),      # 16 x 13 = 208 tiles, 104 in pairs: a wave and 30 tiles in halves
    (2048, 4352),      # 16 x 17 = 272 tiles, 136 in pairs: a wave and 62 whole tiles
]


@pytest.mark.parametrize("fmt,out", [(amx.FMT_AMXFP4, torch.float32), (amx.FMT_AMXFP4, torch.bfloat16), (amx.FMT_MXFP4, torch.float32),
                                     (amx.FMT_MXFP4, torch.bfloat16)])
@pytest.mark.parametrize("M,N", SHAPES)
def test_parts_of_tiles(M, N, fmt, out):
    K = 416
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N)
    x = (torch.randn(M, K, device="cuda", generator=g) + 0.3).to(torch.bfloat16)
    w = (0.02 * torch.randn(N, K, device="cuda", generator=g)).to(torch.bfloat16)
    ac, as_, a = amx.quantize_prepared(x, False, fmt=fmt)
    wc, ws, b = amx.quantize_prepared(w, True, fmt=fmt)
    ref = amx.dequantize(ac, as_, 32, torch.float32).double() @ amx.dequantize(wc, ws, 32, torch.float32).double().T
    wide = torch.full((M, N + 16), -3.0, dtype=out, device="cuda")
    got = amx.gemm_prepared(a, b, M, N, K, out=wide[:, :N], sym=fmt != amx.FMT_AMXFP4, out_dtype=out)
    assert torch.all(wide[:, N:] == -3.0)
    assert float((got.double() - ref).norm() / ref.norm()) <= (2.0 ** -12 if out is torch.float32 else 2.0 ** -8)


@pytest.mark.parametrize("M,N,K,ranges", [(128, 512, 14336, True), (100, 1000, 28672, True), (64, 304, 8192, True), (300, 520, 11008, True),
                                          # (ragged: whole tiles of results stored one by one, ranges 23 us, parts 16 at 92 x 412 x 8192)
                                          (64, 300, 8192, False), (92, 412, 8192, False),
                                          (128, 8192, 14336, False), (500, 4096, 4096, False), (128, 512, 4096, False)])
def test_ranges_of_one_plane(M, N, K, ranges):
    """Products promised to be of one plane: long and narrow ones are cut into K ranges on the general kernel, where the promise changes
    nothing; the others, and all of them without scratch for ranges, check it."""
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    x = (torch.randn(M, K, device="cuda", generator=g) + 0.3).to(torch.bfloat16)
    w = (0.02 * torch.randn(N, K, device="cuda", generator=g)).to(torch.bfloat16)
    for fmt in (amx.FMT_MXFP4, amx.FMT_AMXFP4):
        ac, as_, a = amx.quantize_prepared(x, False, fmt=fmt)
        wc, ws, b = amx.quantize_prepared(w, True, fmt=fmt)
        ref = amx.dequantize(ac, as_, 32, torch.float32).double() @ amx.dequantize(wc, ws, 32, torch.float32).double().T
        for nbytes in (amx.lib().amx_gemm_prepared_workspace_bytes(M, N, K, 32), 256):
            work = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
            got = amx.gemm_prepared(a, b, M, N, K, workspace=work, sym=True)
            if fmt == amx.FMT_MXFP4 or (ranges and nbytes > 256):
                assert amx.gemm_status(work) == 0
                assert float((got.double() - ref).norm() / ref.norm()) <= 2.0 ** -12
            else:
                assert amx.gemm_status(work) == -5
