"""The weight-streaming kernel at the edges of its tiles: token tiles of 8 (1 to 8 of them, and blocks of 64 rows above),
weight rows around a CTA's 128, K ranges of unequal length and longer than the scales held at a time, every fixed group
size; rows cast inside the kernel and ahead of it; weights whose scales start at an odd half word (groups of 128)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu


def dev_bf16(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
@pytest.mark.parametrize("M,N,K", [(1, 129, 512), (3, 8, 640), (8, 1030, 1152), (9, 128, 2176), (24, 300, 896), (32, 127, 1024),
                                   (40, 257, 640), (64, 130, 1408), (65, 140, 512), (130, 1024, 1024), (256, 260, 768),
                                   (2, 20, 33920)])
def test_few_rows_against_oracle(M, N, K, gs):
    a_bits = inputs.random_groups(3000 + M, M, K, "mixed" if gs % 32 == 0 else "normal")
    w_bits = inputs.random_groups(3100 + N, N, K, "normal")
    qa, qw = oracle.quantize(a_bits, gs), oracle.quantize(w_bits, gs)
    ref = oracle.gemm(*qa, *qw, gs)
    dev = [torch.from_numpy(t).cuda() for t in (*qa, *qw)]
    assert amx.lib().amx_gemm_kernel_for(M, N, K, gs, amx.GEMM_AUTO) == amx.GEMM_ROWS
    wide = torch.full((M, N + 3), 5.0, dtype=torch.float32, device="cuda")
    got = amx.gemm(*dev, gs, out=wide[:, :N])
    assert torch.all(wide[:, N:] == 5.0)
    g = got.cpu().numpy().astype(np.float64)
    for m in range(M):                                # "mixed" rows differ by many orders of magnitude
        if np.all(np.isfinite(ref[m])) and np.linalg.norm(ref[m]) > 0:
            assert np.linalg.norm(g[m] - ref[m]) <= 1e-5 * np.linalg.norm(ref[m]), m
    strided = torch.zeros((M, K + 24), dtype=torch.bfloat16, device="cuda")
    strided[:, 8:8 + K] = dev_bf16(a_bits)
    assert torch.equal(amx.quant_gemm(strided[:, 8:8 + K], dev[2], dev[3], gs), got.contiguous())
    assert torch.equal(amx.quant_gemm(dev_bf16(a_bits), group_size=gs, w_bf16=dev_bf16(w_bits)), got.contiguous())


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
@pytest.mark.parametrize("M,N,K", [(64, 40, 20480), (57, 130, 34048)])
def test_long_ranges_of_eight_token_tiles(M, N, K, gs):
    """Eight token tiles and K ranges of 20 and 34 steps: more than the scales held at a time, which for groups of 16 take
    the most shared memory."""
    a_bits, w_bits = inputs.random_groups(3250, M, K, "normal"), inputs.random_groups(3251, N, K, "normal")
    qw = oracle.quantize(w_bits, gs)
    got = amx.quant_gemm(dev_bf16(a_bits), *(torch.from_numpy(t).cuda() for t in qw), gs, flags=amx.GEMM_ROWS)
    ref = oracle.gemm(*oracle.quantize(a_bits, gs), *qw, gs)
    assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


def test_back_to_back_calls_share_a_workspace():
    """Calls chained on one stream, every one of them on the same workspace and output: each sees its own rows."""
    N, K = 512, 4096
    w_bits = inputs.random_groups(3200, N, K, "normal")
    wc, ws = amx.quantize(dev_bf16(w_bits))
    for M in (1, 20):
        xs = [dev_bf16(inputs.random_groups(3201 + i, M, K, "normal")) for i in range(6)]
        want = [amx.quant_gemm(x, wc, ws).clone() for x in xs]
        torch.cuda.synchronize()
        work = torch.empty(amx.lib().amx_quant_gemm_workspace_bytes(M, N, K, 32, 0), dtype=torch.uint8, device="cuda")
        out = torch.empty((M, N), dtype=torch.float32, device="cuda")
        got = []
        for x in xs:
            got.append(amx.quant_gemm(x, wc, ws, out=out, workspace=work).clone())
        assert all(torch.equal(g, w) for g, w in zip(got, want))
        assert amx.gemm_status(work) == 0


@pytest.mark.parametrize("gs", [16, 64, 128])
@pytest.mark.parametrize("M,N,K", [(300, 1000, 1152), (513, 776, 1024), (257, 2048, 640), (300, 3000, 320)])
def test_other_group_sizes_on_the_fp4_kernel(M, N, K, gs):
    """Groups of 16, 64 and 128 through the FP4 kernel (AUTO, from 2^28 multiply-adds): ragged rows, K tails inside a
    64-element block of scale factors; a flushed scale sends the product to the exact kernel."""
    if K % gs:
        pytest.skip("K not a multiple of the group size")
    a_bits, w_bits = inputs.random_groups(3300 + M, M, K, "normal"), inputs.random_groups(3400 + N, N, K, "normal")
    L = amx.lib()
    want = amx.GEMM_FP4 if M * N * K >= 1 << 28 else L.amx_gemm_kernel_for(M, N, K, gs, 0)
    assert L.amx_gemm_kernel_for(M, N, K, gs, amx.GEMM_AUTO) == want
    for spread in (0, 20):                            # 20 binades between the groups of row 3: scales are flushed
        if spread:
            a_bits = a_bits.copy()
            f = inputs.bf16_bits_to_f32(a_bits)
            f[3, :gs] *= 2.0 ** 12
            f[3, gs:] *= 2.0 ** (12 - spread)
            a_bits = inputs.f32_to_bf16_bits(f)
        qa, qw = oracle.quantize(a_bits, gs), oracle.quantize(w_bits, gs)
        dev = [torch.from_numpy(t).cuda() for t in (*qa, *qw)]
        rows = np.unique(np.concatenate([[0, 3, M - 1], np.arange(0, M, 37)]))
        ref = oracle.gemm(*qa, *qw, gs, rows=rows)
        work = torch.empty(L.amx_workspace_bytes(M, N, K, gs, 0) + 256, dtype=torch.uint8, device="cuda")
        got = amx.gemm(*dev, gs, workspace=work)
        if want == amx.GEMM_FP4:
            assert amx.gemm_status(work) == 0 and (amx.gemm_flushed_scales(work) > 0) == bool(spread)
        assert np.linalg.norm(got.cpu().numpy()[rows] - ref) <= 1e-5 * np.linalg.norm(ref)
        assert torch.equal(amx.quant_gemm(dev_bf16(a_bits), dev[2], dev[3], gs), got)
        assert torch.equal(amx.quant_gemm(dev_bf16(a_bits), group_size=gs, w_bf16=dev_bf16(w_bits)), got)


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
@pytest.mark.parametrize("M,N,K", [(600, 520, 1152), (2100, 700, 128), (260, 300, 11008), (300, 257, 5504)])
def test_one_launch_prepares_both_operands(M, N, K, gs):
    """The launch that casts the activation and casts or splits the weight, at row lengths of 4 to 344 pieces (several rows
    per warp, one row, more pieces than a lane keeps in registers), ragged rows, strided rows: against the oracle on
    sampled rows, and the same bits from the bf16 and from the quantized weight."""
    a_bits, w_bits = inputs.random_groups(3500 + M, M, K, "normal"), inputs.random_groups(3600 + N, N, K, "normal")
    qw = oracle.quantize(w_bits, gs)
    wc, ws = (torch.from_numpy(t).cuda() for t in qw)
    rows = np.unique(np.concatenate([[0, 1, M - 1], np.arange(5, M, 61)]))
    ref = oracle.gemm(*oracle.quantize(a_bits[rows], gs), *qw, gs)
    got = amx.quant_gemm(dev_bf16(a_bits), wc, ws, gs)
    assert np.linalg.norm(got.cpu().numpy()[rows] - ref) <= 1e-5 * np.linalg.norm(ref)
    strided_a = torch.zeros((M, K + 8), dtype=torch.bfloat16, device="cuda")
    strided_w = torch.zeros((N, K + 40), dtype=torch.bfloat16, device="cuda")
    strided_a[:, :K], strided_w[:, 8:8 + K] = dev_bf16(a_bits), dev_bf16(w_bits)
    assert torch.equal(amx.quant_gemm(strided_a[:, :K], group_size=gs, w_bf16=strided_w[:, 8:8 + K]), got)
