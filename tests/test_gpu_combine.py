"""The weighted sum over a token's experts at the edges of its block shape: rows narrower than a block of 256 columns
(several tokens per block, the last block partly filled), exactly one block wide, and one block plus a remainder."""
import numpy as np
import pytest
import torch

import moe_check as MC
from oracle import moe as M
from oracle import nvfp4 as Q
from paper_2607_15810_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,topk", [(1, 128, 1), (17, 128, 9), (3, 1920, 2), (5, 2048, 3), (2, 2176, 2), (3, 4096, 1)])
def test_weighted_sum_at_row_widths(T, H, topk):
    from paper_2607_15810_b200 import binding as B
    sh = synth.MoEShape("combine", 900 + H + T, T, H, 16, topk, 128, 0.05, 2, 3.0, 10.0)
    x, _ = synth.activations(sh)
    lg = synth.router_logits(sh)
    w13, w2 = synth.expert_weights(sh, "w13"), synth.expert_weights(sh, "w2")
    w13o, w2o = MC.oracle_weights(w13), MC.oracle_weights(w2)
    pilot = M.moe_forward(MC.f32(x), lg.numpy(), w13o, w2o, topk, 0, 0, np.float32(1.0))
    a2 = Q.tensor_global_scale(pilot["h"])
    gw13 = B.fake_quant_weights(w13.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    gw2 = B.fake_quant_weights(w2.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    res = B.moe_w4a4_rac(x.cuda(), lg.cuda(), gw13, gw2, topk, 0, 0, torch.tensor([a2]).cuda(), export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    MC.check_moe(res, x, lg, w13o, w2o, topk, 0, 0, a2)
