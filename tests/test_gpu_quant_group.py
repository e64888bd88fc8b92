"""A base of which some projections are 8-bit codes and some bf16: the codes of a group are converted together (long
runs), so a matrix has to end up in the slot its projection reads whichever of the group's matrices are converted."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, REL_FRO
from test_gpu_quant import quantise

pytestmark = pytest.mark.gpu


def _decoder(cfg, model, W, W8=None, Ws=None):
    pools = [{p: moin.Pool(model.pools[l][p].A.to(DEV), model.pools[l][p].B.to(DEV),
                           model.pools[l][p].slot_of_expert.to(DEV)) for p in oracle.PROJ_ORDER} for l in range(cfg.n_layers)]
    return moin.DecoderModel(cfg, model.embed.to(DEV), model.lm_head.to(DEV), model.final_norm.to(DEV),
                             [t.to(DEV) for t in model.attn_norm], [t.to(DEV) for t in model.mlp_norm], W, pools, cfg.E,
                             cfg.scale, W8=W8, W_scale=Ws)


@pytest.mark.parametrize("coded", [oracle.PROJ_ORDER, ("k", "up", "down"), ("q", "v", "gate", "o")])
def test_some_projections_coded(coded):
    cfg = mi.DecoderConfig(n_layers=1, hidden=320, n_heads=5, n_kv_heads=1, head_dim=64, ffn=576, vocab=512, E=4, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=3)
    q = {p: quantise(model.W[0][p]) for p in coded}
    plain = {p: model.W[0][p].to(DEV) for p in oracle.PROJ_ORDER}
    same = dict(plain)   # the same weights, converted by the oracle
    for p in coded:
        same[p] = torch.from_numpy(oracle.dequant_fp8(q[p][0].numpy(), q[p][1].numpy()).view(np.int16)).view(torch.bfloat16).to(DEV)
    mixed = _decoder(cfg, model, [{p: plain[p] for p in plain if p not in coded}], [{p: q[p][0].to(DEV) for p in coded}],
                     [{p: q[p][1].to(DEV) for p in coded}])
    ref = _decoder(cfg, model, [same])
    for lengths in ([130, 77], [600, 9], [700, 403]):   # segments; tiles on either base
        batch = mi.decoder_batch(cfg, lengths, seed=5, req_expert=[0, 2])
        args = (batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths))
        # the same bf16 weights through the same kernels
        assert torch.equal(moin.decoder_forward(mixed, *args), moin.decoder_forward(ref, *args))


@pytest.mark.parametrize("T", [1, 16, 17, 33, 64, 65, 128, 129, 300, 512, 513])
@pytest.mark.parametrize("adapters", [True, False])
def test_few_tokens(T, adapters):
    """Short segments: the GEMM converts the codes itself; edges of its token tile and of the rule that takes it."""
    cfg = mi.DecoderConfig(n_layers=1, hidden=320, n_heads=5, n_kv_heads=1, head_dim=64, ffn=1088, vocab=512, E=4, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=4)
    q = {p: quantise(model.W[0][p]) for p in oracle.PROJ_ORDER}
    same = {p: torch.from_numpy(oracle.dequant_fp8(c.numpy(), s.numpy()).view(np.int16)).view(torch.bfloat16).to(DEV)
            for p, (c, s) in q.items()}
    coded = _decoder(cfg, model, [{}], [{p: c.to(DEV) for p, (c, s) in q.items()}], [{p: s.to(DEV) for p, (c, s) in q.items()}])
    ref = _decoder(cfg, model, [same])
    lengths = [min(37, T - i) for i in range(0, T, 37)]
    batch = mi.decoder_batch(cfg, lengths, seed=6, req_expert=[i % 4 for i in range(len(lengths))])
    args = [batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV) if adapters else None, max(lengths)]
    got, want = (moin.decoder_forward(m, *args).double() for m in (coded, ref))
    # the same bf16 weights, sums of 32-bit products in another order: two bf16 roundings of a chain of four projections
    assert torch.isfinite(got).all()
    assert ((got - want).norm() / want.norm()).item() <= REL_FRO * 2 ** 0.5
    assert moin.device_status()["timeout_flag"] == 0
