"""The exact kernel behind an FP4 product of few tiles adds its K ranges by a launch of fewer blocks than results / 256 when it is
gated: sizes around one round of that launch (1184 blocks of 256), a ragged last one, a result with gaps between its rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(257, 1179), (257, 1180), (300, 6001)])
def test_wide_scales_reach_the_exact_kernel_whatever_the_size(M, N, K=1024):
    rng = np.random.default_rng(M + N)
    a = (2.0 ** -10 * np.abs(rng.standard_normal((M, K)))).astype(np.float32)
    a[:, :32] = 0.0
    a[:, 0] = 2.0 ** 10                                 # 15 binades and more above the rest of its row: flushed there
    w = rng.standard_normal((N, K)).astype(np.float32)
    w[:, 0] = 0.0
    a, w = inputs.f32_to_bf16_bits(a), inputs.f32_to_bf16_bits(w)
    assert amx.lib().amx_gemm_kernel_for(M, N, K, 32, amx.GEMM_AUTO) == amx.GEMM_FP4
    dev = lambda b: torch.from_numpy(b.view(np.int16)).cuda().view(torch.bfloat16)
    wc, ws = amx.quantize(dev(w), 32)
    wide = torch.full((M, N + 7), 3.0, dtype=torch.float32, device="cuda")
    got = amx.quant_gemm(dev(a), wc, ws, out=wide[:, :N])
    ref = oracle.gemm(*oracle.quantize(a, 32), *oracle.quantize(w, 32), 32).astype(np.float64)
    err = np.linalg.norm(got.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 1e-5 and torch.all(wide[:, N:] == 3.0)
    assert np.all(np.isfinite(ref)) and np.linalg.norm(ref) > 0
    explicit = amx.quant_gemm(dev(a), wc, ws, flags=amx.GEMM_FP4).cpu().numpy()
    assert np.linalg.norm(explicit - ref) / np.linalg.norm(ref) > 0.5     # the FP4 kernel alone loses these groups
