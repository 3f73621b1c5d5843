"""Tiles of 256 x 256 computed by pairs of CTAs at their edges: an odd number of 128-row blocks (half a pair has no rows),
a last block of a few rows, columns that end inside either CTA's half of a tile, K of a few blocks and of a part of one;
two planes per operand and one."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu


def dev_bf16(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


@pytest.mark.parametrize("fmt,mode", [(amx.FMT_AMXFP4, 0), (amx.FMT_MXFP4, oracle.MXFP4)])
@pytest.mark.parametrize("M,N,K", [(1900, 2600, 96), (1924, 2816, 288), (2177, 2305, 416), (300, 38000, 1056)])
def test_pairs_against_oracle(fmt, mode, M, N, K):
    a_bits = inputs.random_groups(5100 + M, M, K, "normal")
    w_bits = inputs.random_groups(5200 + N, N, K, "normal")
    _, _, pa = amx.quantize_prepared(dev_bf16(a_bits), False, fmt=fmt)
    wc, ws, pw = amx.quantize_prepared(dev_bf16(w_bits), True, fmt=fmt)
    work = torch.full((amx.lib().amx_gemm_prepared_workspace_bytes(M, N, K, 32),), 0xFF, dtype=torch.uint8, device="cuda")
    wide = torch.full((M, N + 5), -3.0, dtype=torch.float32, device="cuda")
    got = amx.gemm_prepared(pa, pw, M, N, K, out=wide[:, :N], workspace=work, sym=mode != 0)
    assert amx.gemm_status(work) == 0
    assert torch.all(wide[:, N:] == -3.0)
    rows = np.unique(np.r_[0:3, 126:130, 254:258, M - 130:M - 124, M - 3:M])
    qa = oracle.quantize_variant(a_bits[rows], 32, mode) if mode else oracle.quantize(a_bits[rows], 32)
    ref = oracle.gemm(*qa, wc.cpu().numpy(), ws.cpu().numpy(), 32)
    g = got[torch.from_numpy(rows).cuda()].cpu().numpy().astype(np.float64)
    for i in range(len(rows)):
        assert np.linalg.norm(g[i] - ref[i]) <= 1e-5 * np.linalg.norm(ref[i]), rows[i]
