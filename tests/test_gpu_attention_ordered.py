"""The fused attention kernel's ordered statistics give the attention map's bits as the stored path has them: logits in
global memory, softmax kernel, cast.  A row sum or an exponent that is rounded elsewhere moves a bf16 probability now and
then, with it the step of its group's scale, and with that a whole row of the result."""
import numpy as np
import pytest
import torch

from paper_2411_09909_b200 import amx

pytestmark = pytest.mark.gpu

# The two paths' results differ by the order of the fp32 additions of P V alone: at most L roundings (tensor cores: truncations,
# 2^-23) of partial sums no larger than the sum of |P V| over the keys, which with P >= 0 summing to about 1 is at most the
# largest |V| of the column.  Random signs: sqrt(L) of them, and a row's norm is of the size of its larger terms.
TOL = 2.0 ** -23 * 8192 ** 0.5


@pytest.mark.parametrize("causal", [0, amx.ATTN_CAUSAL])
@pytest.mark.parametrize("heads,kv,L,d,flags", [(32, 32, 1056, 128, amx.GEMM_AUTO),     # 9 key tiles: 8 + 1, ragged last tile
                                                (32, 8, 1024, 128, amx.GEMM_AUTO),      # whole blocks, short
                                                (16, 16, 736, 64, amx.GEMM_AUTO),       # 6 tiles, the last of 96 keys
                                                (4, 4, 2080, 128, amx.GEMM_AUTO),       # 17 tiles: 2 x 8 + 1
                                                (4, 4, 2560, 64, amx.GEMM_AUTO),        # 20 whole tiles
                                                (2, 1, 8192, 64, amx.GEMM_AUTO),        # all 256 groups of the softmax kernel
                                                (64, 16, 416, 128, amx.GEMM_FP4),       # 256 items of 4 tiles: two per CTA
                                                (64, 64, 32, 128, amx.GEMM_FP4), (64, 64, 160, 64, amx.GEMM_FP4)])
def test_fused_attention_equals_the_stored_path(heads, kv, L, d, flags, causal):
    for seed in range(2):
        g = torch.Generator(device="cuda")
        g.manual_seed(1000 * seed + L + d)
        q, k, v = (torch.randn(h, L, d, device="cuda", generator=g) for h in (heads, kv, kv))
        for x in (q, k, v):
            x[:, :, torch.randperm(d, device="cuda", generator=g)[:2]] *= 20.0
        q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
        got = amx.attention_heads(q, k, v, flags | causal).double()
        want = amx.attention_heads(q, k, v, amx.GEMM_TC | causal).double()
        err = (got - want).norm(dim=2) / want.norm(dim=2)
        assert err.max().item() <= TOL, (seed, err.max().item(), (err > TOL).nonzero()[:8].tolist(), int((err > TOL).sum()))


@pytest.mark.parametrize("causal", [0, amx.ATTN_CAUSAL])
@pytest.mark.parametrize("L,d", [(8224, 128), (9216, 64)])
def test_rows_past_the_ordered_sums(L, d, causal):
    """Past 8192 keys both paths add in orders of their own: a row may take another bf16 value (up to 1 in 10 000 above; here
    1 in 1000), anything wrong with the one block of sums moves all of them."""
    g = torch.Generator(device="cuda")
    g.manual_seed(L)
    q, k, v = (torch.randn(1, L, d, device="cuda", generator=g).to(torch.bfloat16) for _ in range(3))
    got = amx.attention_heads(q, k, v, causal).double()
    want = amx.attention_heads(q, k, v, amx.GEMM_TC | causal).double()
    err = (got - want).norm(dim=2) / want.norm(dim=2)
    assert (err > TOL).double().mean().item() <= 1e-3 and err.max().item() < 0.5


def test_scratch_of_long_rows_stays_linear():
    need = [amx.lib().amx_attention_workspace_bytes_for(L, 64, 0) for L in (65536, 131072)]
    assert need[1] <= 2.1 * need[0]


@pytest.mark.parametrize("causal", [0, amx.ATTN_CAUSAL])
def test_exact_attention_kernel_equals_the_stored_path(causal):
    """A scale the FP4 kernel cannot hold sends AUTO to the kernel on CUDA cores: the same softmax once more.  The wide row's
    largest element meets zeros in Q, so that the logits are sums of few binades: the same numbers in any order."""
    L, d = 1056, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    q, k, v = (torch.randn(4, L, d, device="cuda", generator=g) for _ in range(3))
    q[:, :, 40:42] *= 20.0
    q[:, :, 0] = 0.0
    k[:, 5, :32] = 0.0
    k[:, 5, 0] = 2.0 ** 15
    k[:, 5, 32:] *= 2.0 ** -3
    q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
    got = amx.attention_heads(q, k, v, causal).double()
    want = amx.attention_heads(q, k, v, amx.GEMM_TC | causal).double()
    assert not torch.equal(got, amx.attention_heads(q, k, v, amx.GEMM_FP4 | causal).double())
    err = (got - want).norm(dim=2) / want.norm(dim=2)
    assert err.max().item() <= TOL, (err.max().item(), int((err > TOL).sum()))
