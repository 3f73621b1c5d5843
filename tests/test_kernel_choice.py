"""What AMX_GEMM_AUTO picks between 65 and 256 rows, where both the weight-streaming kernel and the FP4 kernel take the call:
the one that measured faster, at shapes where the two differ by more than a twentieth (us, weights from HBM, one call)."""
import pytest

from paper_2411_09909_b200 import amx

MEASURED = [  # M, N, K, streaming kernel (its best layout), FP4 route
    (72, 28672, 4096, 105.9, 81.8), (128, 28672, 4096, 129.0, 90.2), (256, 28672, 4096, 223.6, 97.4),
    (128, 12288, 4096, 58.0, 54.3), (256, 12288, 4096, 98.2, 63.5), (256, 6144, 4096, 57.6, 46.0), (160, 8192, 4096, 59.1, 48.2),
    (72, 6144, 4096, 26.2, 40.0), (128, 8192, 4096, 35.8, 47.7), (192, 6144, 4096, 36.1, 45.3), (256, 4096, 4096, 36.2, 43.4),
    (128, 4096, 4096, 23.5, 41.4), (128, 4096, 11008, 50.0, 85.1), (72, 4096, 14336, 62.2, 103.2), (128, 4096, 14336, 62.3, 107.8),
    (256, 1024, 4096, 15.4, 38.0), (256, 2048, 2048, 15.6, 27.9), (192, 256, 4096, 11.0, 40.7), (72, 12288, 640, 11.9, 21.3),
    (256, 12288, 640, 27.8, 22.8), (200, 14336, 512, 28.2, 20.0), (128, 8192, 640, 10.7, 20.6), (256, 28672, 1024, 78.2, 42.0),
    (96, 5120, 2560, 18.5, 31.1), (256, 4096, 512, 9.9, 17.5),
    (128, 1024, 1024, 6.3, 22.7)]


@pytest.mark.parametrize("M,N,K,rows_us,fp4_us", MEASURED)
def test_auto_takes_the_faster_kernel(M, N, K, rows_us, fp4_us):
    want = amx.GEMM_ROWS if rows_us < fp4_us else amx.GEMM_FP4
    assert amx.lib().amx_gemm_kernel_for(M, N, K, 32, amx.GEMM_AUTO) == want


def test_narrow_weights_keep_the_route_that_counts_flushed_scales():
    assert amx.lib().amx_gemm_kernel_for(128, 256, 8192, 32, amx.GEMM_AUTO) == amx.GEMM_FP4
    assert amx.lib().amx_gemm_kernel_for(64, 256, 8192, 32, amx.GEMM_AUTO) == amx.GEMM_ROWS


@pytest.mark.parametrize("M", [1, 33, 48, 64])
def test_up_to_64_rows_stream_the_weight(M):
    for N, K in ((28672, 4096), (4096, 14336), (12288, 4096), (128, 512)):
        assert amx.lib().amx_gemm_kernel_for(M, N, K, 32, amx.GEMM_AUTO) == amx.GEMM_ROWS


@pytest.mark.parametrize("gs", [16, 32, 128])
@pytest.mark.parametrize("N,K", [(512, 512), (1024, 4096), (4096, 4096), (12288, 4096), (28672, 1024), (28672, 512), (4096, 14336), (768, 8192),
                                 (16384, 2048), (5120, 2560)])
def test_the_choice_changes_once_as_rows_are_added(N, K, gs):
    """And within the streaming kernel's range no call needs more scratch than one of more rows."""
    L = amx.lib()
    kernels = [L.amx_gemm_kernel_for(M, N, K, gs, 0) for M in range(1, 257)]
    assert kernels == sorted(kernels, reverse=True)                     # GEMM_ROWS (0x100), then GEMM_FP4 (0x40)
    need = [L.amx_quant_gemm_workspace_bytes(M + 1, N, K, gs, 0) for M, k in enumerate(kernels) if k == amx.GEMM_ROWS]
    assert need == sorted(need)
