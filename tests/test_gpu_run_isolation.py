"""Experts do not interact: an adapter that holds infinities or NaN spoils the tokens of its own runs and no others, also
where runs share a row tile of the long-run GEMM or meet in a CTA pair."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, gpu_pool, kernel_launches, oracle_layer
from test_gpu_decoder import oracle_weights

pytestmark = pytest.mark.gpu


def _spoil(pool, slot, where):
    t = getattr(pool, where)
    t[slot, 0, 0], t[slot, -1, -1] = float("inf"), float("nan")
    t[slot, t.shape[1] // 2] = float("-inf")


@pytest.mark.parametrize("where", ["A", "B"])
@pytest.mark.parametrize("lengths,experts,r", [
    ([100, 200], [0, 1], 64),                               # two runs in a tile
    ([60, 300, 70], [1, 2, 1], 16),                         # runs in front of and behind others in both CTAs of a pair
    ([32] * 9 + [7], [1, 0, 2, 1, 3, 0, 1, 2, -1, 1], 24),  # more runs than a tile takes, some without an adapter
    ([128, 128, 1], [1, 0, 1], 72),                         # a CTA each
])
def test_layer(lengths, experts, r, where):
    te = np.repeat(np.asarray(experts, np.int32), lengths)
    E, d_in, d_out = 4, 128, 264
    pool = mi.make_pool(E, r, d_in, d_out, 55, r, missing=(3,))
    case = mi.layer_case("isolation", len(te), d_in, d_out, pool, te, 2.0, 55, r)
    rows = np.nonzero(te != 1)[0]
    ref = oracle_layer(case, rows)
    _spoil(pool, 1, where)
    x, W, p = case.x.to(DEV), case.W.to(DEV), gpu_pool(pool)
    for mode in (moin.PLAN_TILES, moin.PLAN_SEGMENTS):
        y = moin.lora_linear(moin.plan_build(torch.from_numpy(te).to(DEV), E, mode), x, W, p, 2.0)
        assert_layer_close(y[torch.from_numpy(rows).to(DEV)], ref, f"mode {mode}")
        assert not torch.isfinite(y[torch.from_numpy(np.nonzero(te == 1)[0]).to(DEV)]).all(dim=1).any()


@pytest.mark.parametrize("lengths,fused", [([290, 330, 275], True), ([90, 130, 75], False)])   # tiles / segments
def test_block_with_fused_product(lengths, fused):
    cfg = mi.DecoderConfig(n_layers=1, hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, ffn=576, vocab=512, E=3, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=18)
    experts = [0, 1, 2]
    batch = mi.decoder_batch(cfg, lengths, seed=18, req_expert=experts)
    args = (batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy())
    orc = oracle.DecoderOracle(cfg, oracle_weights(model))
    h_in = orc.forward(*args, layer_begin=0, layer_end=0, want_hidden=True, want_logits=False)["hidden"]
    want = orc.forward(*args, layer_begin=0, layer_end=1, round_storage=True, hidden_in=h_in, want_hidden=True, want_logits=False)["hidden"]
    for p in ("gate", "up", "down"):   # (behind the attention, whose key tiles reach into the next request)
        _spoil(model.pools[0][p], 1, "B")
    pools = [{p: gpu_pool(model.pools[0][p]) for p in oracle.PROJ_ORDER}]
    gm = moin.DecoderModel(cfg, model.embed.to(DEV), model.lm_head.to(DEV), model.final_norm.to(DEV),
                           [t.to(DEV) for t in model.attn_norm], [t.to(DEV) for t in model.mlp_norm],
                           [{p: model.W[0][p].to(DEV) for p in oracle.PROJ_ORDER}], pools, cfg.E, cfg.scale)
    hin = torch.from_numpy(h_in).to(torch.float32).to(DEV)
    hid = torch.empty(batch.T, cfg.hidden, dtype=torch.float32, device=DEV)
    n = kernel_launches(lambda: moin.decoder_forward(gm, batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV),
                                                     max(lengths), logits_mode=moin.LOGITS_NONE, hidden_in=hin, hidden_out=hid))
    assert ("lora_fused_tc" in n) == fused
    d, ref = hid.double().cpu().numpy() - hin.double().cpu().numpy(), want - h_in
    own = slice(lengths[0], lengths[0] + lengths[1])
    others = np.r_[0:lengths[0], lengths[0] + lengths[1]:batch.T]
    assert np.linalg.norm(d[others] - ref[others]) <= 5e-3 * np.linalg.norm(ref[others])
    assert not np.isfinite(d[own]).all(axis=1).any()
    assert moin.device_status()["timeout_flag"] == 0
