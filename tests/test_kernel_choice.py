"""What AMX_GEMM_AUTO picks between 65 and 256 rows, where both the weight-streaming kernel and the FP4 kernel take the call:
the one that measured faster, at shapes where the two differ by more than a twentieth (us, weights from HBM, one call).  And that the
shapes at which the streaming kernel is tested take the layouts they are there for."""
import ctypes

import pytest
import test_gpu_gemm_rows_layouts

from paper_2411_09909_b200 import amx

MEASURED = [  # M, N, K, streaming kernel (its best layout), FP4 route
    (72, 28672, 4096, 106.0, 70.3), (128, 28672, 4096, 129.2, 72.1), (256, 28672, 4096, 224.3, 88.2),
    (128, 12288, 4096, 58.1, 41.3), (256, 12288, 4096, 98.7, 49.1), (256, 6144, 4096, 57.7, 32.9),
    (160, 8192, 4096, 56.9, 35.8), (72, 6144, 4096, 27.2, 29.3), (128, 8192, 4096, 36.2, 33.0), (192, 6144, 4096, 36.3, 32.7),
    (256, 4096, 4096, 36.3, 29.8), (128, 4096, 4096, 23.7, 29.1), (128, 4096, 11008, 50.2, 62.9),
    (72, 4096, 14336, 52.3, 79.3), (128, 4096, 14336, 62.8, 81.1), (256, 1024, 4096, 15.1, 26.9),
    (256, 2048, 2048, 16.0, 19.0), (192, 256, 4096, 8.5, 28.6), (72, 12288, 640, 11.6, 16.1), (256, 12288, 640, 27.9, 20.5),
    (200, 14336, 512, 23.5, 18.4), (128, 8192, 640, 10.8, 14.2), (256, 28672, 1024, 78.6, 37.7), (96, 5120, 2560, 18.7, 22.8),
    (256, 4096, 512, 9.7, 14.0), (128, 1024, 1024, 7.6, 16.4), (96, 12288, 4096, 52.1, 40.1), (80, 14336, 4096, 56.4, 43.1),
    (160, 4096, 11008, 72.8, 63.4), (144, 5120, 2560, 21.1, 25.6),
    (192, 16384, 2048, 57.0, 35.4), (128, 16384, 2048, 39.3, 29.8), (72, 18944, 3584, 52.3, 45.8),
    (144, 9216, 3072, 46.8, 31.1), (256, 2304, 9216, 44.2, 50.3)]

# Ragged N, rows of the weight of 4096 to 8192 elements, and other group sizes: M, N, K, group size, streaming kernel, FP4 route
MEASURED_OTHERS = [
    (197, 2645, 4864, 16, 33.5, 46.5), (192, 4781, 2688, 16, 28.2, 37.5), (96, 7424, 4864, 16, 39.2, 43.1), (225, 7279, 768, 64, 17.5, 24.9),
    (256, 4327, 2304, 32, 23.3, 27.6), (74, 13017, 1280, 64, 22.4, 27.7), (192, 8287, 1664, 32, 28.7, 32.1), (189, 12907, 896, 32, 28.4, 39.6),
    (128, 27658, 768, 64, 30.5, 48.7), (104, 4081, 3840, 32, 22.7, 30.6), (192, 20844, 1920, 32, 71.8, 62.3), (132, 13625, 4352, 32, 87.6, 73.4),
    (239, 14618, 3456, 32, 97.9, 66.1), (192, 8799, 3584, 32, 51.2, 43.8), (192, 8254, 7040, 64, 90.1, 72.1), (192, 11776, 3840, 128, 61.9, 44.9),
    (148, 8786, 6016, 16, 92.2, 66.8), (175, 9112, 1152, 128, 22.7, 18.9)]


@pytest.mark.parametrize("M,N,K,gs,rows_us,fp4_us", MEASURED_OTHERS)
def test_auto_takes_the_faster_kernel_ragged_or_other_groups(M, N, K, gs, rows_us, fp4_us):
    want = amx.GEMM_ROWS if rows_us < fp4_us else amx.GEMM_FP4
    assert amx.lib().amx_gemm_kernel_for(M, N, K, gs, amx.GEMM_AUTO) == want


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
@pytest.mark.parametrize("N,K", [(512, 512), (1024, 4096), (4096, 4096), (12288, 4096), (28672, 1024), (28672, 512), (4096, 14336), (768, 8192), (4781, 2688), (11472, 4224),
                                 (16384, 2048), (5120, 2560)])
def test_the_choice_changes_once_as_rows_are_added(N, K, gs):
    """And within the streaming kernel's range no call needs more scratch than one of more rows."""
    L = amx.lib()
    kernels = [L.amx_gemm_kernel_for(M, N, K, gs, 0) for M in range(1, 257)]
    assert kernels == sorted(kernels, reverse=True)                     # GEMM_ROWS (0x100), then GEMM_FP4 (0x40)
    need = [L.amx_quant_gemm_workspace_bytes(M + 1, N, K, gs, 0) for M, k in enumerate(kernels) if k == amx.GEMM_ROWS]
    assert need == sorted(need)


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
def test_the_tested_shapes_cover_the_layouts(gs):
    diag = amx.lib().amx_diag_rows_layout
    diag.argtypes = [ctypes.c_int64] * 3 + [ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    taken = set()
    for M, N, K in test_gpu_gemm_rows_layouts.SHAPES:
        layout = (ctypes.c_int * 5)()
        assert diag(M, N, K, gs, layout) == 0 and layout[0] == 1
        taken.add(tuple(layout[1:]))
    tiles, blocks, rows, ranges = (set(v) for v in zip(*taken))
    assert tiles == {1, 2, 3, 4} and {1, 4, 7} <= blocks
    assert rows >= {8, 16, 24, 32, 40, 48, 72, 80} | (set() if gs == 16 else {56, 88, 96, 104, 112})   # (groups of 16: less room)
    assert ranges == {1, 2, 4, 8}
    assert {(r, s) for _, _, r, s in taken} >= {(8, 1), (8, 4), (8, 8), (16, 1), (16, 2), (16, 4), (16, 8), (40, 1), (40, 2), (40, 4), (40, 8),
                                               (48, 1), (48, 4), (72, 1), (72, 2), (72, 8)}
