"""Attention on the tensor cores: item and key-tile edges, the two key streams (no tile for one of them, odd and even
numbers of tiles), head groups of 1 to 8, and scores that grow along the keys, so that running maxima are overtaken and the
accumulator is rescaled."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV
from test_gpu_decoder import gpu_model, oracle_weights, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,kv", [(8, 1), (4, 1), (4, 4)])
@pytest.mark.parametrize("gain", [1.0, 12.0])
@pytest.mark.parametrize("lengths", [[1, 15, 16, 17], [63, 64, 65, 66], [128, 129, 193], [577]])
def test_attention_block(heads, kv, gain, lengths):
    cfg = mi.DecoderConfig(n_layers=1, hidden=64 * heads, n_heads=heads, n_kv_heads=kv, head_dim=64, ffn=64, vocab=512, E=2, r=8, scale=2.0)
    model = mi.decoder_model(cfg, seed=12)
    for p in ("q", "k"):   # scores gain^2 times as wide: tens of powers of two for the larger gain
        model.W[0][p] = (model.W[0][p].float() * gain).to(torch.bfloat16)
    orc = oracle.DecoderOracle(cfg, oracle_weights(model))
    batch = mi.decoder_batch(cfg, lengths, seed=12, req_expert=[i % 2 for i in range(len(lengths))])
    args = (batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy())
    h_in = orc.forward(*args, layer_begin=0, layer_end=0, want_hidden=True, want_logits=False)["hidden"]
    rnd, exact = (orc.forward(*args, layer_begin=0, layer_end=1, round_storage=r, hidden_in=h_in, want_hidden=True,
                              want_logits=False)["hidden"] - h_in for r in (True, False))
    hin = torch.from_numpy(h_in).to(torch.float32).to(DEV)
    hid = torch.empty(batch.T, cfg.hidden, dtype=torch.float32, device=DEV)
    moin.decoder_forward(gpu_model(model), batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths),
                         logits_mode=moin.LOGITS_NONE, hidden_in=hin, hidden_out=hid)
    d = hid.double().cpu().numpy() - hin.double().cpu().numpy()
    # no further from the definition than storing the declared tensors in bf16 costs
    e_exact, e_storage = rel(d, exact), rel(rnd, exact)
    print(f"heads {heads}/{kv}, gain {gain}, lengths {lengths}: vs fp64 {e_exact:.2e}, storage rounding alone {e_storage:.2e}")
    assert e_exact <= 1.1 * e_storage + 1e-3
    assert moin.device_status()["timeout_flag"] == 0
