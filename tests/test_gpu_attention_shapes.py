"""Attention at the edges of what its kernels tile: sequences that are no multiple of 128 and head dimension 64 through the
fused kernel (padding, masked last key tile, causal diagonal in a partial block), grouped queries, the batched launches
of short sequences, and the device-side fallback for scales the FP4 kernel cannot represent."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu


def bf(rng, shape, outliers=True):
    x = rng.standard_normal(shape).astype(np.float32)
    if outliers:
        x[..., :2] *= 20.0
    return inputs.f32_to_bf16_bits(x)


def dev(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


def rows_agree(O, ref):
    """Row by row.  The oracle's exponentials are fp64 ones, so a probability may round to the neighbouring bf16 value, which
    can move its group's scale by a step and with it the row (none of 44 000 rows of these inputs, drawn three times); the
    other rows differ by fp32 additions alone, 1e-7.  Anything wrong at the edge of a tile moves a row of every head."""
    err = np.linalg.norm(O - ref, axis=1) / np.linalg.norm(ref, axis=1)
    return np.sum(err > 1e-5) <= len(err) // 500 and np.max(err) < 0.5


def reference(q, k, v, causal):
    d = q.shape[1]
    S = oracle.gemm(*oracle.quantize(q, 32), *oracle.quantize(k, 32), 32)
    P = oracle.softmax_bf16(S, d ** -0.5, causal_row0=0) if causal else oracle.softmax_bf16(S, d ** -0.5)
    return oracle.gemm(*oracle.quantize(P, 32), *oracle.quantize(np.ascontiguousarray(v.T), 32), 32).astype(np.float64)


@pytest.mark.parametrize("causal", [0, amx.ATTN_CAUSAL])
@pytest.mark.parametrize("heads,kv,L,d,flags", [(2, 1, 544, 128, amx.GEMM_AUTO), (2, 2, 736, 64, amx.GEMM_AUTO), (3, 3, 768, 64, amx.GEMM_AUTO),
                                                (1, 1, 1056, 128, amx.GEMM_AUTO), (4, 2, 32, 128, amx.GEMM_FP4), (2, 1, 160, 64, amx.GEMM_FP4),
                                                (5, 5, 96, 64, amx.GEMM_AUTO), (12, 3, 224, 128, amx.GEMM_AUTO), (2, 2, 256, 96, amx.GEMM_AUTO)])
def test_attention_shapes_against_oracle_pipeline(heads, kv, L, d, flags, causal):
    rng = np.random.default_rng(heads * 1000 + L + d)
    q, k, v = bf(rng, (heads, L, d)), bf(rng, (kv, L, d)), bf(rng, (kv, L, d))
    O = amx.attention_heads(dev(q), dev(k), dev(v), flags | causal).cpu().numpy()
    assert np.all(np.isfinite(O))
    for h in range(heads):
        kvh = h // (heads // kv)
        ref = reference(q[h], k[kvh], v[kvh], causal)
        assert rows_agree(O[h], ref), h


@pytest.mark.parametrize("causal", [0, amx.ATTN_CAUSAL])
@pytest.mark.parametrize("L,d", [(544, 128), (768, 64)])
def test_flushed_scales_send_attention_to_the_exact_kernel(L, d, causal):
    """One row of K spans 20 binades between its groups: the FP4 kernel could not hold its small groups, which carry the
    logits here.  AUTO computes the call exactly; asked for explicitly, the FP4 kernel is visibly off."""
    rng = np.random.default_rng(7)
    q, k, v = (inputs.bf16_bits_to_f32(bf(rng, (2, L, d), False)) for _ in range(3))
    k[:, 5, :32] = 0.0
    k[:, 5, 0] = 2.0 ** 15
    k[:, 5, 32:] *= 2.0 ** -3
    q[:, :, 0] = 0.0                                  # the huge element meets a zero
    q, k, v = (inputs.f32_to_bf16_bits(t) for t in (q, k, v))
    O = amx.attention_heads(dev(q), dev(k), dev(v), causal).cpu().numpy()
    for h in range(2):
        ref = reference(q[h], k[h], v[h], causal)
        assert rows_agree(O[h], ref)
    # the same call without the wide row stays on the fused kernel: equal to the explicit FP4 call bit for bit
    k2 = inputs.bf16_bits_to_f32(k)
    k2[:, 5] = 0.5
    k2 = inputs.f32_to_bf16_bits(k2)
    assert torch.equal(amx.attention_heads(dev(q), dev(k2), dev(v), causal), amx.attention_heads(dev(q), dev(k2), dev(v), causal | amx.GEMM_FP4))
