"""The cooperative front of larger batches (routing and quantization as two roles of one launch, then selection and
dispatch copies) at its edges: one token per routing warp and the two-token form, more than 32 tokens per routing
CTA, more tokens than the small-batch kernels take by one, channel groups of 128 / 256 / 512, slabs of 512 channels
that do not divide the row, the widest top-k, no residual, a given scale, operand-swapped GEMMs behind it."""
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


@pytest.mark.parametrize("T,H,E,topk,f13,static", [
    (513, 128, 8, 2, 0.5, False), (600, 640, 33, 3, 0.25, True), (1185, 256, 256, 1, 0.0, False), (1200, 384, 5, 5, 1.0, False),
    (2400, 768, 129, 16, 0.5, False), (2369, 1152, 64, 2, 0.0, True), (4800, 128, 16, 4, 0.5, False), (520, 256, 256, 8, 0.5, False),
    (520, 256, 256, 8, 0.0, False)])
def test_front_of_a_larger_layer(B, T, H, E, topk, f13, static):
    I = 128
    sh = synth.MoEShape("front", 700 + T, T, H, E, topk, I, 0.05, 2, 3.0, 10.0)
    x, _ = synth.activations(sh)
    lg = synth.router_logits(sh)
    lg[T // 2] = lg[T // 2].round()                            # equal logits: ties go to the lower expert
    w13, w2 = synth.expert_weights(sh, "w13"), synth.expert_weights(sh, "w2")
    w13o, w2o = MC.oracle_weights(w13), MC.oracle_weights(w2)
    nsel13, nsel2 = int(H * f13), I // 2
    a13 = np.float32(0.5) * Q.tensor_global_scale(MC.f32(x)) if static else None
    a13_d = torch.tensor([float(a13)], device="cuda") if static else None
    pilot = M.moe_forward(MC.f32(x), lg.numpy(), w13o, w2o, topk, nsel13, 0, np.float32(1.0), a13_gs=a13)
    a2 = Q.tensor_global_scale(pilot["h"])
    gw13 = B.fake_quant_weights(w13.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    gw2 = B.fake_quant_weights(w2.cuda(), want_fq=False, sf_layout=B.SF_TILED)
    args = (x.cuda(), lg.cuda(), gw13, gw2, topk, nsel13, nsel2, torch.tensor([a2]).cuda())
    res = B.moe_w4a4_rac(*args, a13_gs=a13_d, export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    MC.check_moe(res, x, lg, w13o, w2o, topk, nsel13, nsel2, a2, a13_gs=a13)
    dirty = torch.full_like(res["workspace"], 0xFF)             # nothing may depend on what the workspace held
    res2 = B.moe_w4a4_rac(*args, a13_gs=a13_d, workspace=dirty)
    assert torch.equal(res2["out"], res["out"])
