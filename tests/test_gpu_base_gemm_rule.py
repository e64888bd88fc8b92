"""Base layer without adapters: both sides of the line between the token-wide GEMM and the CTA pairs, pairs with fewer rows than
one CTA has among them."""
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV

pytestmark = pytest.mark.gpu


# 262144 + 160 d_in products of tokens and features; 64 and 512 tokens
@pytest.mark.parametrize("T,d_in,d_out", [(64, 64, 4264), (65, 64, 4184), (65, 64, 4192), (129, 64, 2112), (129, 64, 2104),
                                          (512, 64, 536), (512, 64, 528), (300, 768, 1288), (300, 768, 1280), (100, 2048, 8000)])
def test_both_sides(T, d_in, d_out):
    x, W = mi.normal_bf16((T, d_in), 1.0, 17, T, device=DEV), mi.normal_bf16((d_out, d_in), 0.02, 18, d_out, device=DEV)
    guard = torch.full((T + 2, d_out), 7.0, dtype=torch.bfloat16, device=DEV)
    y = guard[1:T + 1]
    moin.lora_linear(None, x, W, None, 0.0, y=y)
    ref = x.double() @ W.double().T
    # one rounding to bf16 (2^-9 of the value) on top of fp32 sums of at most 2048 products of size 0.02
    assert ((y.double() - ref).abs() <= ref.abs() * 2 ** -8 + 2e-5).all()
    assert (guard[0] == 7).all() and (guard[T + 1] == 7).all()
    assert moin.device_status()["timeout_flag"] == 0
