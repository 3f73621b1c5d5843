"""Quantized weights that miss an alignment, between 65 and 256 rows under AUTO: taken or refused by shape alone, whichever
kernel the estimates pick, and right where taken."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu


def shifted(t, by):
    b = torch.empty(t.numel() + 16, dtype=torch.uint8, device="cuda")
    b[by:by + t.numel()] = t.reshape(-1)
    return b[by:by + t.numel()].view(t.shape)


@pytest.mark.parametrize("M,N,K,codes_by,scales_by,taken", [
    (128, 640, 1024, 4, 2, True), (72, 12288, 1024, 4, 2, True), (200, 12288, 768, 4, 2, True),    # streaming kernel, streaming, FP4
    (96, 1233, 4992, 4, 2, False), (207, 5120, 768, 8, 2, False),                                   # streaming kernel, neither alignment
    (96, 1233, 4992, 0, 2, True), (128, 12288, 1024, 0, 2, True), (128, 640, 1024, 4, 0, False)])
def test_misaligned_weights(M, N, K, codes_by, scales_by, taken):
    a_bits, w_bits = inputs.random_groups(5000 + M, M, K, "normal"), inputs.random_groups(5100 + N, N, K, "normal")
    qw = oracle.quantize(w_bits, 32)
    x = torch.from_numpy(a_bits.view(np.int16)).cuda().view(torch.bfloat16)
    wc, ws = (shifted(torch.from_numpy(t).cuda(), by) for t, by in zip(qw, (codes_by, scales_by)))
    if not taken:
        with pytest.raises(amx.AmxError, match="misaligned"):
            amx.quant_gemm(x, wc, ws)
        return
    got = amx.quant_gemm(x, wc, ws)
    rows = np.array([0, M // 2, M - 1])
    ref = oracle.gemm(*oracle.quantize(a_bits[rows], 32), *qw, 32)
    assert np.linalg.norm(got.cpu().numpy()[rows] - ref) <= 1e-5 * np.linalg.norm(ref)
