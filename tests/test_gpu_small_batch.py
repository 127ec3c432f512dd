"""The single-cluster front of a call with few tokens (routing, quantization, selection, dispatch) at the edges of
its tiling: 16 tokens per word of the assignment matrix, 256 tokens where a warp takes a second one, 512 where the
grid-wide kernels take over; channel units of 128 that do not divide over the cluster; the widest top-k.  Every
result is compared with the oracle as for any other layer (`moe_check`)."""
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
    (15, 256, 16, 4, 0.5, False), (16, 128, 8, 2, 0.25, True), (17, 384, 33, 3, 0.5, False),
    (1, 128, 256, 16, 0.5, False), (31, 640, 33, 3, 0.25, False), (32, 256, 5, 5, 1.0, True), (33, 2176, 8, 2, 0.5, False),
    (255, 384, 64, 16, 0.0, False), (256, 256, 129, 8, 0.5, True), (257, 1024, 16, 4, 0.5, False), (511, 256, 32, 2, 0.5, False),
    (512, 128, 8, 8, 0.25, False), (513, 128, 8, 8, 0.25, False)])
def test_front_of_a_small_layer(B, T, H, E, topk, f13, static):
    I = 128
    sh = synth.MoEShape("front", 900 + T, T, H, E, topk, I, 0.05, 2, 3.0, 10.0)
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
    res = B.moe_w4a4_rac(x.cuda(), lg.cuda(), gw13, gw2, topk, nsel13, nsel2, torch.tensor([a2]).cuda(), a13_gs=a13_d,
                         export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    MC.check_moe(res, x, lg, w13o, w2o, topk, nsel13, nsel2, a2, a13_gs=a13)
    dirty = torch.full_like(res["workspace"], 0xFF)             # nothing may depend on what the workspace held
    res2 = B.moe_w4a4_rac(x.cuda(), lg.cuda(), gw13, gw2, topk, nsel13, nsel2, torch.tensor([a2]).cuda(), a13_gs=a13_d,
                          workspace=dirty)
    assert torch.equal(res2["out"], res["out"])


@pytest.mark.parametrize("T,K,nsel", [(1, 2176, 7), (127, 640, 320), (129, 128, 64), (512, 1152, 1151), (513, 256, 128)])
def test_front_of_a_small_dense_projection(B, T, K, nsel):
    """Channels K/2 .. K-1 repeat channels 0 .. K/2-1, so the selection's boundary falls between equal scores
    (unless it separates two pairs): the lower channel is taken."""
    x, w = synth.dense_inputs(T + K, T=T, K=K, N=128)
    x[:, K // 2:] = x[:, :K - K // 2]
    wq = B.fake_quant_weights(w.unsqueeze(0).cuda(), want_fq=False, sf_layout=B.SF_TILED)
    res = B.dense_w4a4_rac(x.cuda(), wq, nsel, export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    wo = MC.oracle_weights(w[None])
    o = M.dense_w4a4_rac(MC.f32(x), wo["codes"][0], wo["sf"][0], wo["gs"][0], nsel)
    MC.check_site1(res, dict(site13=o["site"]), nsel, {})
    got = MC.f32(res["out"]).astype(np.float64)
    assert float((np.abs(got - o["y64"]) / MC.gemm_tol(o["absdot"], o["y64"])).max()) <= 1.0
