"""One expert id per token, constant inside each request, against one per request: the same kernels and the same bits, on both
sides of the rule that chooses between segments and tiles."""
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, kernel_launches
from test_gpu_decoder import gpu_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [16, 64])
@pytest.mark.parametrize("lengths,experts", [([100] * 3, [0, 1, 2]), ([300], [1]), ([1], [-1]), ([24] * 25, [i % 5 for i in range(25)]),
                                             ([40] * 12, [i % 6 - 1 for i in range(12)]), ([128] * 6, [2, 2, -1, 0, 0, 3]),
                                             ([129, 1, 511, 64], [3, 0, 3, 9]), ([6] * 60, [i % 4 for i in range(60)]),
                                             ([700, 257], [0, 0]), ([640], [4])])
def test_constant_ids(lengths, experts, r):
    cfg = mi.DecoderConfig(n_layers=2, hidden=256, n_heads=4, n_kv_heads=2, head_dim=64, ffn=576, vocab=512, E=6, r=r, scale=2.0)
    gm = gpu_model(mi.decoder_model(cfg, seed=31, missing=(2,)))
    batch = mi.decoder_batch(cfg, lengths, seed=32, req_expert=experts)
    tok, cu, ids = batch.tokens.to(DEV), batch.cu_seqlens.to(DEV), batch.req_expert.to(DEV)
    te = torch.repeat_interleave(batch.req_expert, torch.tensor(lengths)).to(torch.int32).to(DEV)
    out = {}

    def per_request():
        out["request"] = moin.decoder_forward(gm, tok, cu, ids, max(lengths))

    def per_token():
        out["token"] = moin.decoder_forward(gm, tok, cu, None, max(lengths), token_expert=te)

    assert kernel_launches(per_request) == kernel_launches(per_token)
    assert torch.equal(out["request"], out["token"])
