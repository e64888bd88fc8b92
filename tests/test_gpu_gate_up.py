"""Long runs: the gate and up projections with their product in one GEMM.  Edges: columns that end inside a tile, ranks of
one and two 64-wide blocks, row tiles of two experts or of none under one CTA pair, an up pool whose slots are not the gate
pool's, no adapters at all, and the smallest batches that take the path; a few that go in segments."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, REL_FRO, kernel_launches
from test_gpu_decoder import oracle_weights, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fused,ffn,r,lengths,experts", [
    (False, 512, 16, [64], [1]), (False, 576, 8, [130, 77, 300], [0, 2, -1]), (True, 1088, 72, [65, 600], [3, 3]),
    (False, 64, 128, [200, 129], [1, 0]), (False, 704, 64, [1, 255, 128, 3, 260], [0, 1, 1, 2, 3]), (True, 832, 0, [513], None),
    (True, 832, 0, [500, 700], None), (True, 512, 16, [629], [1]), (True, 576, 8, [260, 154, 601], [0, 2, -1]),
    (True, 64, 128, [406, 229], [1, 0]), (True, 704, 64, [1, 511, 256, 3, 521], [0, 1, 1, 2, 3]), (False, 832, 0, [512], None)])
def test_block_with_fused_product(fused, ffn, r, lengths, experts):
    cfg = mi.DecoderConfig(n_layers=1, hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, ffn=ffn, vocab=512, E=4, r=max(r, 8), scale=2.0)
    model = mi.decoder_model(cfg, seed=8, missing=(2,))
    w = oracle_weights(model)
    orc = oracle.DecoderOracle(cfg, w)
    pools = None
    if experts is not None:
        pools = [{}]
        for p in oracle.PROJ_ORDER:
            m = model.pools[0][p]
            A, B, slot = m.A, m.B, m.slot_of_expert
            if p == "up":   # the same adapters in another order
                perm = torch.arange(A.shape[0] - 1, -1, -1)
                A, B = A[perm].contiguous(), B[perm].contiguous()
                slot = torch.where(slot >= 0, (A.shape[0] - 1 - slot).to(slot.dtype), slot)
            pools[0][p] = moin.Pool(A.to(DEV), B.to(DEV), slot.to(DEV))
    gm = moin.DecoderModel(cfg, model.embed.to(DEV), model.lm_head.to(DEV), model.final_norm.to(DEV),
                           [t.to(DEV) for t in model.attn_norm], [t.to(DEV) for t in model.mlp_norm],
                           [{p: model.W[0][p].to(DEV) for p in oracle.PROJ_ORDER}], pools, cfg.E, cfg.scale)
    batch = mi.decoder_batch(cfg, lengths, seed=8, req_expert=experts if experts is not None else [-1] * len(lengths))
    args = (batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy())
    h_in = orc.forward(*args, layer_begin=0, layer_end=0, want_hidden=True, want_logits=False)["hidden"]
    want = orc.forward(*args, layer_begin=0, layer_end=1, round_storage=True, hidden_in=h_in, want_hidden=True, want_logits=False)["hidden"]
    hin = torch.from_numpy(h_in).to(torch.float32).to(DEV)
    hid = torch.empty(batch.T, cfg.hidden, dtype=torch.float32, device=DEV)
    n = kernel_launches(lambda: moin.decoder_forward(
        gm, batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV) if pools else None, max(lengths),
        logits_mode=moin.LOGITS_NONE, hidden_in=hin, hidden_out=hid))
    assert n["decoder_glue"] == 7 - fused   # meta 2, three norms, rotation, the SwiGLU where it is a launch of its own
    assert ("lora_fused_tc" in n) == (fused and pools is not None)
    e = rel(hid.double().cpu().numpy() - hin.double().cpu().numpy(), want - h_in)
    # the layer's tolerance: storage rounded to bf16 where the oracle rounds it
    assert e <= REL_FRO, e
    assert moin.device_status()["timeout_flag"] == 0
