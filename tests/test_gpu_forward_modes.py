"""Decoder forwards on both sides of the rules that choose between segments and tiles, and in segments between the kernels of
the base GEMM: tokens and mean lengths at their edges, block by block against the oracle, and the kernels that they launch."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, REL_FRO, kernel_launches
from test_gpu_decoder import gpu_model, oracle_weights, rel

pytestmark = pytest.mark.gpu


def _block(lengths, r):
    cfg = mi.DecoderConfig(n_layers=1, hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, ffn=576, vocab=512, E=9, r=r, scale=2.0)
    model = mi.decoder_model(cfg, seed=23, missing=(4,))
    orc = oracle.DecoderOracle(cfg, oracle_weights(model))
    batch = mi.decoder_batch(cfg, lengths, seed=r, req_expert=[(5 * i) % 10 - 1 for i in range(len(lengths))])
    args = (batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy())
    h_in = orc.forward(*args, layer_begin=0, layer_end=0, want_hidden=True, want_logits=False)["hidden"]
    ref = orc.forward(*args, layer_begin=0, layer_end=1, round_storage=True, hidden_in=h_in, want_hidden=True, want_logits=False)["hidden"]
    hin = torch.from_numpy(h_in).to(torch.float32).to(DEV)
    hid = torch.empty(batch.T, cfg.hidden, dtype=torch.float32, device=DEV)
    args = (gpu_model(model), batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths))
    run = lambda: moin.decoder_forward(*args, logits_mode=moin.LOGITS_NONE, hidden_in=hin, hidden_out=hid)
    run()
    assert moin.device_status()["timeout_flag"] == 0
    # as test_gpu_decoder's blocks: one block against the oracle that rounds where the library stores
    assert rel(hid.double().cpu().numpy() - hin.double().cpu().numpy(), ref - h_in) <= REL_FRO
    return kernel_launches(run)


@pytest.mark.parametrize("r", [16, 40])
@pytest.mark.parametrize("lengths", [[64] * 5 + [63], [64] * 6, [40] * 11 + [39], [40] * 12, [6] * 43, [24] * 22, [9] * 170, [28] * 73,
                                     [27] * 76, [29] * 71])
def test_block(lengths, r):
    _block(lengths, r)


# the fewest tokens that go in tiles, 605 + (14 + 160 / r) R in models this narrow, and one token less
@pytest.mark.parametrize("r,lengths", [(8, [236, 236, 235]), (16, [629]), (16, [85] * 9 + [80]), (16, [40] * 37 + [37]),
                                       (40, [79] * 9 + [74]), (128, [400, 235])])
def test_fewest_tokens_in_tiles(r, lengths):
    n = _block(lengths, r)
    assert n["lora_fused_tc"] == 4 and "lora_expand_stream" not in n
    n = _block(lengths[:-1] + [lengths[-1] - 1], r)
    assert n["lora_expand_stream"] == 4 and "lora_fused_tc" not in n


@pytest.mark.parametrize("r", [32, 48])   # tiles of 64 tokens up to rank 32
@pytest.mark.parametrize("T", [256, 257, 513, 1280, 1281, 2047, 2048, 2049])
def test_segments(T, r):
    n = _block([min(9, T - i) for i in range(0, T, 9)], r)
    assert n["lora_expand_stream"] == 4 and "lora_fused_tc" not in n
    assert n["gemm_tc"] == (4 if T <= 2048 else 7)   # a launch a group, or one a projection


@pytest.mark.parametrize("lengths", [[37] * 56, [9] * 70, [2] * 513])   # codes converted by the GEMM beyond 512 tokens, and no longer
def test_coded_base(lengths):
    from test_gpu_quant import quantise
    from test_gpu_quant_group import _decoder
    cfg = mi.DecoderConfig(n_layers=1, hidden=320, n_heads=5, n_kv_heads=1, head_dim=64, ffn=1088, vocab=512, E=4, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=4)
    q = {p: quantise(model.W[0][p]) for p in oracle.PROJ_ORDER}
    same = {p: torch.from_numpy(oracle.dequant_fp8(c.numpy(), s.numpy()).view(np.int16)).view(torch.bfloat16).to(DEV) for p, (c, s) in q.items()}
    coded = _decoder(cfg, model, [{}], [{p: c.to(DEV) for p, (c, s) in q.items()}], [{p: s.to(DEV) for p, (c, s) in q.items()}])
    batch = mi.decoder_batch(cfg, lengths, seed=6, req_expert=[i % 4 for i in range(len(lengths))])
    args = [batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths)]
    got, want = (moin.decoder_forward(m, *args).double() for m in (coded, _decoder(cfg, model, [same])))
    # the same bf16 weights, sums of 32-bit products in another order: two bf16 roundings of a chain of four projections
    assert ((got - want).norm() / want.norm()).item() <= REL_FRO * 2 ** 0.5
    assert moin.device_status()["timeout_flag"] == 0


@pytest.mark.parametrize("lengths,tiles,converted", [([94] * 12 + [86], False, False), ([94] * 12 + [87], True, True), ([8] * 256, False, False),
                                                     ([8] * 256 + [1], False, True)])
def test_coded_base_kernels(lengths, tiles, converted):
    from test_gpu_quant import quantise
    from test_gpu_quant_group import _decoder
    cfg = mi.DecoderConfig(n_layers=1, hidden=320, n_heads=5, n_kv_heads=1, head_dim=64, ffn=576, vocab=512, E=4, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=4)
    q = {p: quantise(model.W[0][p]) for p in oracle.PROJ_ORDER}
    coded = _decoder(cfg, model, [{}], [{p: c.to(DEV) for p, (c, s) in q.items()}], [{p: s.to(DEV) for p, (c, s) in q.items()}])
    orc = oracle.DecoderOracle(cfg, dict(oracle_weights(model), W=[{p: oracle.dequant_fp8(c.numpy(), s.numpy()) for p, (c, s) in q.items()}]))
    batch = mi.decoder_batch(cfg, lengths, seed=6, req_expert=[i % 4 for i in range(len(lengths))])
    args = [batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths)]
    got = moin.decoder_forward(coded, *args).double().cpu().numpy()
    want = orc.forward(batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy(), round_storage=True)["logits"]
    assert rel(got, want) <= REL_FRO * 2 ** 0.5   # as test_gpu_decoder's logits: a block and the head
    n = kernel_launches(lambda: moin.decoder_forward(coded, *args))
    assert ("lora_fused_tc" in n) == tiles and ("lora_expand_stream" in n) != tiles
    # meta 2, embedding, two norms, rotation, SwiGLU (in the GEMM where tiles are), two norms behind the block; a conversion a group
    assert n["decoder_glue"] == 9 - tiles + 4 * converted


@pytest.mark.parametrize("coded", [False, True])
@pytest.mark.parametrize("lengths", [[9] * 8, [70, 41, 30]])
def test_wide_block(lengths, coded):
    """A block of full width in segments: reductions of more k-blocks than a CTA has stages, so that what was requested before the
    wait and what follows it share the ring."""
    from test_gpu_quant import quantise
    from test_gpu_quant_group import _decoder
    cfg = mi.DecoderConfig(n_layers=1, vocab=512, E=4, r=16, scale=2.0)
    model = mi.decoder_model(cfg, seed=7)
    q = {p: quantise(model.W[0][p]) for p in oracle.PROJ_ORDER}
    W = {p: oracle.dequant_fp8(c.numpy(), s.numpy()) for p, (c, s) in q.items()}
    if coded:
        gm = _decoder(cfg, model, [{}], [{p: c.to(DEV) for p, (c, s) in q.items()}], [{p: s.to(DEV) for p, (c, s) in q.items()}])
    else:
        gm = _decoder(cfg, model, [{p: torch.from_numpy(w.view(np.int16)).view(torch.bfloat16).to(DEV) for p, w in W.items()}])
    batch = mi.decoder_batch(cfg, lengths, seed=6, req_expert=[i % 4 for i in range(len(lengths))])
    run = lambda: moin.decoder_forward(gm, batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV), max(lengths))
    orc = oracle.DecoderOracle(cfg, dict(oracle_weights(model), W=[W]))
    want = orc.forward(batch.tokens.numpy(), batch.cu_seqlens.numpy(), batch.req_expert.numpy(), round_storage=True)["logits"]
    assert rel(run().double().cpu().numpy(), want) <= REL_FRO * 2 ** 0.5 * 1.5   # as test_gpu_decoder's blocks of this width, and the head
    assert "lora_expand_stream" in kernel_launches(run)
    assert moin.device_status()["timeout_flag"] == 0
