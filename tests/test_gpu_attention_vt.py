"""The cast of V beside those of Q and K: its keys come in passes of 2048 with the last one short, head dimension 64 leaves half of a
head's operand rows empty, and from 8224 keys on a row's scales are read back instead of kept.  Also more query blocks than the
exact kernel has CUDA blocks."""
import numpy as np
import pytest
import torch

from paper_2411_09909_b200 import amx, inputs
from test_gpu_attention_shapes import bf, dev, reference, rows_agree

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,kv,L,d", [(2, 1, 2048, 64), (1, 1, 2080, 128), (2, 2, 4064, 64), (1, 1, 8192, 64), (1, 1, 8224, 128)])
def test_key_passes_of_v(heads, kv, L, d):
    rng = np.random.default_rng(L + d)
    q, k, v = bf(rng, (heads, L, d)), bf(rng, (kv, L, d)), bf(rng, (kv, L, d))
    O = amx.attention_heads(dev(q), dev(k), dev(v), amx.GEMM_FP4 | amx.ATTN_CAUSAL).cpu().numpy()
    for h in range(heads):
        assert rows_agree(O[h], reference(q[h], k[h // (heads // kv)], v[h // (heads // kv)], True)), h


@pytest.mark.parametrize("which", ["v", "k"])
def test_exact_kernel_walks_over_many_blocks(which):
    """48 heads of 34 query blocks each, sent to the exact kernel by one wide row of K or of V^T."""
    rng = np.random.default_rng(11)
    heads, L, d = 48, 544, 64
    t = {n: inputs.bf16_bits_to_f32(bf(rng, (heads, L, d), False)) for n in "qkv"}
    if which == "k":
        t["k"][3, 5, :32], t["k"][3, 5, 32:] = 0.0, t["k"][3, 5, 32:] * 2.0 ** -3
        t["k"][3, 5, 0], t["q"][:, :, 0] = 2.0 ** 15, 0.0
    else:
        t["v"][3, :32, 7], t["v"][3, 32:, 7] = 2.0 ** 15, t["v"][3, 32:, 7] * 2.0 ** -3
    q, k, v = (inputs.f32_to_bf16_bits(t[n]) for n in "qkv")
    O = amx.attention_heads(dev(q), dev(k), dev(v), amx.ATTN_CAUSAL).cpu().numpy()
    assert not torch.equal(torch.from_numpy(O[3]), amx.attention_heads(dev(q), dev(k), dev(v), amx.ATTN_CAUSAL | amx.GEMM_FP4)[3].cpu())
    for h in (0, 3, 29, heads - 1):
        assert rows_agree(O[h], reference(q[h], k[h], v[h], True)), h
