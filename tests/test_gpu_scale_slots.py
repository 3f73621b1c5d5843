"""Scale factors in tensor memory: a K block's copies overwrite those of the block two before while its MMAs may still be queued, and rely on
the order of issue.  Here every row's scales change by up to twelve binades from one stretch of 64 elements to the next, so that
factors taken from another K block would show as gross errors; repeated calls must agree bit for bit.

The reference is the fp64 product of the decoded operands; the fp32 accumulation is below K 2^-24 of the sum of magnitudes, taken
as 2^-12 of the norm."""
import pytest
import torch

from paper_2411_09909_b200 import amx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", [amx.FMT_AMXFP4, amx.FMT_MXFP4])
@pytest.mark.parametrize("M,N,K", [(128, 128, 4096), (128, 256, 8192), (130, 2500, 4096), (500, 4096, 2048), (1000, 4096, 1056), (2048, 3328, 1024),
                                   (4096, 5120, 512)])
def test_scales_that_change_from_block_to_block(M, N, K, fmt):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)

    def operand(rows):
        steps = torch.randint(-12, 1, (rows, (K + 63) // 64), device="cuda", generator=g).repeat_interleave(64, 1)[:, :K]
        x = torch.randn(rows, K, device="cuda", generator=g) + 0.3
        return torch.ldexp(x, steps).to(torch.bfloat16)
    ac, as_, a = amx.quantize_prepared(operand(M), False, fmt=fmt)
    wc, ws, b = amx.quantize_prepared(operand(N), True, fmt=fmt)
    assert amx.prepared_flushed_scales(a, M, K, is_weight=False) + amx.prepared_flushed_scales(b, N, K, is_weight=True) <= (M + N) * K // 32 // 50
    # what the kernel multiplies: scales of 15 and more binades below their row's largest are flushed
    dec = [amx.dequantize(c, s, 32, torch.float32).double() for c, s in ((ac, as_), (wc, ws))]
    ref = dec[0] @ dec[1].T
    work = torch.empty(256, dtype=torch.uint8, device="cuda")
    got = amx.gemm_prepared(a, b, M, N, K, workspace=work, sym=fmt != amx.FMT_AMXFP4)
    assert float((got.double() - ref).norm() / ref.norm()) <= 2.0 ** -12
    for _ in range(10):
        assert torch.equal(amx.gemm_prepared(a, b, M, N, K, workspace=work, sym=fmt != amx.FMT_AMXFP4), got)
