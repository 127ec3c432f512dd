"""The in-kernel channel selection (threshold search) at the sizes where it can go wrong: equal scores across
the boundary, one channel more or fewer than a tie group, nothing and everything but one selected."""
import numpy as np
import pytest
import torch

import moe_check as MC
from oracle import moe as M
from oracle import nvfp4 as Q
from oracle import rac as R
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


def _separated_channels(T, H, lo, hi, seed):
    """Channel c has one magnitude in every row, rising with c from lo to hi, and random signs: the scores of two
    channels differ by far more than any order of float32 additions can change."""
    g = torch.Generator().manual_seed(seed)
    mag = lo + (hi - lo) * torch.arange(H, dtype=torch.float32) / H
    return (mag * (torch.randint(0, 2, (T, H), generator=g) * 2 - 1)).to(torch.bfloat16)


# a given scale that every channel exceeds by 1.5 to 3 times (all clip), and one outlier beside which the others vanish
SCORE_RANGES = {"clipped": (4096.0, 8192.0, 1.0), "beside_an_outlier": (1e-5, 2e-5, None)}


@pytest.mark.parametrize("kind", sorted(SCORE_RANGES))
@pytest.mark.parametrize("T,K,nsel", [
    (513, 512, 33), (600, 256, 100), (1111, 640, 300), (40, 512, 33),
    (772, 3072, 900), (513, 4608, 700)])       # column groups of 256 and 512 channels
def test_site13_scores_keep_their_order_dense(B, kind, T, K, nsel):
    lo, hi, gs = SCORE_RANGES[kind]
    x = _separated_channels(T, K, lo, hi, T)
    if gs is None:
        x[:, 0] = 1e4
    _, w = synth.dense_inputs(T, T=8, K=K, N=128)
    wq = B.fake_quant_weights(w.unsqueeze(0).cuda(), want_fq=False, sf_layout=B.SF_TILED)
    res = B.dense_w4a4_rac(x.cuda(), wq, nsel, a_gs=None if gs is None else torch.tensor([gs], device="cuda"), export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    wo = MC.oracle_weights(w[None])
    o = M.dense_w4a4_rac(MC.f32(x), wo["codes"][0], wo["sf"][0], wo["gs"][0], nsel, a_gs=None if gs is None else np.float32(gs))
    MC.check_site1(res, dict(site13=o["site"]), nsel, {})


@pytest.mark.parametrize("kind", sorted(SCORE_RANGES))
@pytest.mark.parametrize("T,H,E,topk,nsel", [
    (600, 256, 8, 2, 60),        # dispatched copies
    (520, 640, 256, 8, 200),     # operand-swapped projections: masked in token order
    (1771, 1024, 8, 2, 300),     # column groups of 256 channels, 111 row ranges
    (994, 3584, 8, 1, 900)])     # of 512 channels
def test_site13_scores_keep_their_order_moe(B, kind, T, H, E, topk, nsel):
    lo, hi, gs = SCORE_RANGES[kind]
    sh = synth.MoEShape("scores", 61 + T, T, H, E, topk, 128, 0.05, 2, 3.0, 10.0)
    x = _separated_channels(T, H, lo, hi, T)
    if gs is None:
        x[:, 0] = 1e4
    lg = synth.router_logits(sh)
    gw13 = B.fake_quant_weights(synth.expert_weights(sh, "w13").cuda(), want_fq=False, sf_layout=B.SF_TILED)
    gw2 = B.fake_quant_weights(synth.expert_weights(sh, "w2").cuda(), want_fq=False, sf_layout=B.SF_TILED)
    res = B.moe_w4a4_rac(x.cuda(), lg.cuda(), gw13, gw2, topk, nsel, 64, torch.ones(1, device="cuda"),
                         a13_gs=None if gs is None else torch.tensor([gs], device="cuda"), export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    site = R.rac(MC.f32(x), nsel, None if gs is None else np.float32(gs))
    MC.check_site1(res, dict(site13=site), nsel, {})
