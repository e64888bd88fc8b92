"""silu(gate) * up over the whole range of the gate, in the GEMM's epilogue (more than 512 tokens) and in the pass of its own
(fewer): far below zero the quotient is small but not zero, and a large `up` brings it back."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [40, 520])
def test_silu_of_large_gates(T):
    H = F = 256
    gates = np.resize([-88.5, -88.0, -87.5, -87.0, -80.0, -30.0, -1.0, -0.0078125, 0.0, 0.5, 20.0, 88.5], F)
    cfg = mi.DecoderConfig(n_layers=1, hidden=H, n_heads=4, n_kv_heads=4, head_dim=64, ffn=F, vocab=64, E=1, r=8, scale=1.0)
    ones, b16 = torch.ones(H), lambda t: t.to(torch.bfloat16).to(DEV).contiguous()
    up = np.where(gates < -60, 2.0 ** 100, 2.0 ** 20)
    W = {p: b16(torch.zeros(H, H)) for p in ("q", "k", "v", "o")}   # nothing is attended to: the block is its MLP
    # the normalised hidden state is all ones, so a projection is its weights' row sum (exact in bf16)
    W["gate"] = b16(torch.from_numpy(gates / H)[:, None].expand(F, H))
    W["up"] = b16(torch.from_numpy(up / H)[:, None].expand(F, H))
    down = np.where(gates < -60, 2.0 ** 20, 2.0 ** -20)
    W["down"] = b16(torch.diag(torch.from_numpy(down)))
    model = moin.DecoderModel(cfg, b16(torch.zeros(64, H)), b16(torch.zeros(64, H)), b16(ones), [b16(ones)], [b16(ones)], [W],
                              None, 1, 1.0)
    hin = torch.ones(T, H, dtype=torch.float32, device=DEV)
    hid = torch.empty_like(hin)
    cu = torch.tensor([0, T], dtype=torch.int32, device=DEV)
    moin.decoder_forward(model, torch.zeros(T, dtype=torch.int32, device=DEV), cu, None, T, logits_mode=moin.LOGITS_NONE,
                         hidden_in=hin, hidden_out=hid)
    got = (hid - hin).double().cpu().numpy()
    want = gates / (1.0 + np.exp(-gates)) * up * down
    # two roundings to bf16 (the product, the down projection) and one to fp32 at the residual's 1.0
    assert (np.abs(got - want) <= 2.0 ** -7 * np.abs(want) + 2.0 ** -22).all(), np.abs(got - want).max(axis=0)
    assert moin.device_status()["timeout_flag"] == 0
