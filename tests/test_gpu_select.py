"""The in-kernel channel selection (threshold search) at the sizes where it can go wrong: equal scores across
the boundary, one channel more or fewer than a tie group, nothing and everything but one selected."""
import numpy as np
import pytest
import torch

import moe_check as MC
from oracle import moe as M
from oracle import nvfp4 as Q
from paper_2607_15810_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    assert torch.cuda.is_available()
    from paper_2607_15810_b200 import binding
    return binding


@pytest.mark.parametrize("T,I,nsel2", [(5, 256, 1), (5, 256, 255), (40, 256, 77), (40, 384, 129), (333, 512, 200)])
def test_site2_selection_takes_the_lower_of_two_equal_channels(B, T, I, nsel2):
    """Features j and j + I/2 have the same weights, hence the same scores: every score occurs twice, and an odd
    boundary inside a pair must take the lower channel.  Compared with the oracle on the exported h."""
    sh = synth.MoEShape("pairs", 71 + T, T, 256, 8, 2, I, 0.05, 2, 3.0, 10.0)
    x, _ = synth.activations(sh)
    lg = synth.router_logits(sh)
    w13, w2 = synth.expert_weights(sh, "w13"), synth.expert_weights(sh, "w2")
    h = I // 2
    for base in (0, I):                                        # gate rows, up rows
        w13[:, base + h:base + I] = w13[:, base:base + h]
    gw13 = B.fake_quant_weights(w13.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    gw2 = B.fake_quant_weights(w2.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    w13o, w2o = MC.oracle_weights(w13), MC.oracle_weights(w2)
    pilot = M.moe_forward(MC.f32(x), lg.numpy(), w13o, w2o, 2, 0, 0, np.float32(1.0))
    a2 = Q.tensor_global_scale(pilot["h"])
    res = B.moe_w4a4_rac(x.cuda(), lg.cuda(), gw13, gw2, 2, 128, nsel2, torch.tensor([a2]).cuda(), export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    sel = res["sel2"].cpu().numpy()[:nsel2]
    assert np.all(np.diff(sel) > 0) and sel[0] >= 0 and sel[-1] < I
    lower, upper = set(sel[sel < h].tolist()), set((sel[sel >= h] - h).tolist())
    assert upper <= lower and len(lower) - len(upper) == nsel2 % 2
    MC.check_moe(res, x, lg, w13o, w2o, 2, 128, nsel2, a2)     # selection against the oracle's, up to 1e-6 ties


@pytest.mark.parametrize("T,I,E,nsel2", [
    (24, 2048, 4, 700),      # operand-swapped second projection: the widest it selects for itself
    (24, 2176, 4, 700),      # one step wider: a selection kernel in between
    (90, 640, 4, 639),       # K tail of half a stage, several chunks of 32 rows per expert, the last one ragged
    (1, 128, 256, 5)])       # one item: all other CTAs have no work
def test_site2_mask_applied_inside_the_second_projection(B, T, I, E, nsel2):
    sh = synth.MoEShape("mask2", 91 + T, T, 128, E, 1, I, 0.05, 2, 3.0, 10.0)
    x, _ = synth.activations(sh)
    lg = synth.router_logits(sh)
    w13, w2 = synth.expert_weights(sh, "w13"), synth.expert_weights(sh, "w2")
    gw13 = B.fake_quant_weights(w13.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    gw2 = B.fake_quant_weights(w2.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    w13o, w2o = MC.oracle_weights(w13), MC.oracle_weights(w2)
    pilot = M.moe_forward(MC.f32(x), lg.numpy(), w13o, w2o, 1, 64, 0, np.float32(1.0))
    a2 = Q.tensor_global_scale(pilot["h"])
    args = (x.cuda(), lg.cuda(), gw13, gw2, 1, 64, nsel2, torch.tensor([a2]).cuda())
    res = B.moe_w4a4_rac(*args, export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    MC.check_moe(res, x, lg, w13o, w2o, 1, 64, nsel2, a2)
    plain = B.moe_w4a4_rac(*args)
    assert torch.equal(plain["out"], res["out"])
