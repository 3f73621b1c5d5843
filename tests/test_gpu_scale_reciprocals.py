"""Every scale a cast can store: the reciprocals the elements are multiplied by and the scale factors of the prepared form.  Groups
hold the scale's midpoints between neighbouring codes, where a reciprocal that is off by its last bit moves a code."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_09909_b200 import amx, inputs

pytestmark = pytest.mark.gpu

TIES = np.array([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0, 6.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 5.5, 0.0])


def groups():
    """One group of 32 per pair of scale bytes: multiples of the positive one, negative multiples of the other."""
    b = np.arange(1, 0x7C, dtype=np.uint16)
    s = (b << 8).view(np.float16).astype(np.float64)
    pos = s[:, None] * TIES
    neg = -s[::-1, None] * TIES
    x = np.concatenate([pos, neg], 1).astype(np.float32)             # exact in bf16: at most 6 significant bits
    assert np.array_equal(inputs.bf16_bits_to_f32(inputs.f32_to_bf16_bits(x)), x)
    return x


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
def test_codes_and_scales_of_every_scale(gs):
    x = np.tile(groups(), (1, max(1, gs // 32)))                     # every scale is some group's largest, whatever the size
    bits = inputs.f32_to_bf16_bits(x)
    dev = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
    codes, scales = amx.quantize(dev, gs)
    rc, rs = oracle.quantize(bits, gs)
    assert np.array_equal(codes.cpu().numpy(), rc) and np.array_equal(scales.cpu().numpy(), rs)


@pytest.mark.parametrize("gs", [16, 32, 64, 128])
def test_nan_among_the_elements(gs):
    """Outside the format, but always the same: the NaN's side gets the scale byte 0x7F, read as 1.75 x 2^16, under which its other
    elements here are zero; a NaN of either sign gets code 7.  The other side and the other groups do not notice."""
    K = 256
    bits = inputs.f32_to_bf16_bits(np.random.default_rng(gs).standard_normal((4, K)).astype(np.float32))
    nans = [(0, 5, 0x7FC0), (1, 70, 0xFFC0), (2, 130, 0x7FFF), (2, 131, 0xFF81), (3, 255, 0x7F81)]
    clean = bits.copy()
    for r, k, b in nans:
        bits[r, k], clean[r, k] = b, 0
    codes, scales = oracle.quantize(clean, gs)
    nib = np.stack([codes & 15, codes >> 4], -1).reshape(4, K)
    scales = scales.reshape(4, K // gs, 2).copy()
    for r, k, b in nans:
        side, group = b >> 15, slice(k // gs * gs, (k // gs + 1) * gs)
        scales[r, k // gs, side] = 0x7F
        of_side = (clean[r, group] >> 15) == side
        nib[r, group][of_side] = side << 3
    for r, k, b in nans:
        nib[r, k] = 7
    want = (nib[:, 0::2] | (nib[:, 1::2] << 4)).astype(np.uint8)
    dev = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
    got = [amx.quantize(dev, gs)] + ([amx.quantize_prepared(dev, False)[:2]] if gs == 32 else [])
    for c, s in got:
        c, s = c.cpu().numpy(), s.cpu().numpy().reshape(4, K // gs, 2)
        assert np.array_equal(s, scales)
        assert np.array_equal(c.reshape(want.shape), want)


@pytest.mark.parametrize("rows,K", [(123, 32), (30, 128), (3, 1280)])
def test_prepared_form_of_every_scale(rows, K):
    """Scales and count of flushed ones through the FP4 route, and the product where nothing is flushed."""
    x = groups()[: rows * K // 32].reshape(rows, K)
    bits = inputs.f32_to_bf16_bits(x)
    dev = torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)
    codes, scales, prepared = amx.quantize_prepared(dev, False)
    rc, rs = oracle.quantize(bits, 32)
    assert np.array_equal(codes.cpu().numpy(), rc) and np.array_equal(scales.cpu().numpy(), rs)
    s = (rs.reshape(rows, -1).astype(np.uint16) << 8).view(np.float16).astype(np.float64)
    exp = np.where(s > 0, np.floor(np.log2(np.where(s > 0, s, 1.0))), -99)
    want = int(np.sum((s > 0) & (exp.max(1, keepdims=True) - exp >= 15)))
    assert amx.prepared_flushed_scales(prepared, rows, K, is_weight=False) == want
    w = inputs.f32_to_bf16_bits(np.random.default_rng(K).standard_normal((256, K)).astype(np.float32))
    wc, ws, wp = amx.quantize_prepared(torch.from_numpy(w.view(np.int16)).cuda().view(torch.bfloat16), True)
    got = amx.gemm_prepared(prepared, wp, rows, 256, K).cpu().numpy().astype(np.float64)
    ref = oracle.gemm(rc, rs, *oracle.quantize(w, 32), 32).astype(np.float64)
    whole = ~np.any((s > 0) & (exp.max(1, keepdims=True) - exp >= 15), 1)
    err = np.linalg.norm(got - ref, axis=1)[whole] / np.linalg.norm(ref, axis=1)[whole]
    assert np.all(err <= 1e-5)                                       # up to 1280 fp32 additions: at random signs some 36 x 2^-23


@pytest.mark.parametrize("gs", [16, 32])
def test_error_of_every_scale(gs):
    """Group by group, so that no large scale hides a small one: decoded values down to the smallest subnormals of the format the
    kernel multiplies in, elements off their codes, clamped ones wherever the scale was rounded down."""
    for factor in (1.06, 1.11):
        bits = inputs.f32_to_bf16_bits((factor * groups()).astype(np.float32))
        codes, scales = oracle.quantize(bits, gs)
        clamped = 0
        for i in range(len(bits)):
            one = [np.ascontiguousarray(t[i:i + 1]) for t in (bits, codes, scales)]
            dev = torch.from_numpy(one[0].view(np.int16)).cuda().view(torch.bfloat16)
            got = amx.quant_error(dev, torch.from_numpy(one[1]).cuda(), torch.from_numpy(one[2]).cuda(), gs).cpu().numpy()
            ref = oracle.quant_error(*one, gs)
            assert got[3] == ref[3] and np.allclose(got[:3], ref[:3], rtol=2.0 ** -20, atol=0), (i, got, ref)
            clamped += ref[3]
        assert clamped > 0 and 0 < ref[1] < ref[0]
