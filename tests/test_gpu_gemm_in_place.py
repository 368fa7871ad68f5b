"""nsk_gemm_bf16 with the activations written over its own input rows: the same values as out of place."""
import pytest
import torch

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,width", [(128, 64), (1000, 128), (4096, 256), (40000, 256), (777, 144), (4096, 240)])
def test_hidden_layer_in_place(gpu, rows, width):
    g = torch.Generator().manual_seed(rows + width)
    A = (0.5 * torch.randn((rows, width), generator=g)).bfloat16().to(gpu)
    B = (torch.randn((width, width), generator=g) / width**0.5).bfloat16().to(gpu)
    bias = torch.randn(width, generator=g).to(gpu)
    h = torch.empty_like(A)
    assert nsk.gemm_bf16(A, B, epilogue=2, bias=bias, hout=h) == 0
    assert nsk.gemm_bf16(A, B, epilogue=2, bias=bias, hout=A) == 0
    torch.cuda.synchronize()
    if width % 64 == 0:  # the same MMAs in the same order
        assert torch.equal(A, h)
    else:  # the kernel that streams both operands: FP32 sums of another kernel, one BF16 rounding apart at most
        assert ((A.float() - h.float()).abs() <= 2.0**-7 * h.float().abs() + 1e-6).all()
