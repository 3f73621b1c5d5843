"""The per-layer functions refuse what is not the matrix they take, before anything runs.  (Shapes are checked before the
device, so that this needs none.)"""
import pytest
import torch

from paper_2411_09909_b200 import amx


def bf16(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16)


@pytest.mark.parametrize("a", [bf16(2, 3, 64), bf16(64), bf16(1, 2, 64, 64)])
def test_quant_gemm_refuses_an_activation_that_is_no_matrix(a):
    codes, scales = torch.zeros((8, 32), dtype=torch.uint8), torch.zeros((8, 2, 2), dtype=torch.uint8)
    with pytest.raises(ValueError, match="a must be a matrix"):
        amx.quant_gemm(a, codes, scales)
    with pytest.raises(ValueError, match="a must be a matrix"):
        amx.quant_gemm(a, w_bf16=bf16(8, 64))


def test_operands_on_the_host_are_refused():
    with pytest.raises(amx.AmxError, match="CUDA"):
        amx.quant_gemm(bf16(4, 64), w_bf16=bf16(8, 64))


def test_gemm_prepared_refuses_a_result_type_it_does_not_have():
    a = torch.zeros(256, dtype=torch.uint8)
    with pytest.raises(amx.AmxError, match="out must be a CUDA tensor"):
        amx.gemm_prepared(a, a, 128, 128, 128, out_dtype=torch.float16)


@pytest.mark.gpu
@pytest.mark.parametrize("w", [(8, 1, 64), (8, 2, 64), (8,)])
def test_quant_gemm_refuses_a_weight_that_is_no_matrix(w):
    with pytest.raises(ValueError, match="w_bf16 must be a matrix"):
        amx.quant_gemm(bf16(4, 64).cuda(), w_bf16=bf16(*w).cuda())


@pytest.mark.gpu
def test_quant_gemm_refuses_a_weight_of_other_columns():
    for k in (32, 128):
        with pytest.raises(AssertionError, match="columns of a"):
            amx.quant_gemm(bf16(4, 64).cuda(), w_bf16=bf16(8, k).cuda())


@pytest.mark.gpu
@pytest.mark.parametrize("codes,scales", [((8, 16), (8, 2, 2)), ((8, 32), (8, 1, 2))])
def test_quant_gemm_refuses_a_quantized_weight_of_fewer_columns(codes, scales):
    with pytest.raises(AssertionError, match="fewer columns"):
        amx.quant_gemm(bf16(4, 64).cuda(), *(torch.zeros(s, dtype=torch.uint8, device="cuda") for s in (codes, scales)))
