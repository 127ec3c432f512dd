"""The dense projection with few output tiles, at the edges of its tile width and of its split of K."""
import numpy as np
import pytest
import torch

import moe_check as MC
from oracle import moe as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K,N,nsel", [
    (1, 4096, 128, 2048),      # eight CTAs per tile
    (64, 4096, 128, 0),        # four, no residual
    (128, 4096, 256, 4096),    # four, every row of the tile
    (130, 2048, 128, 1024),    # two row tiles, two rows in the second
    (40, 640, 128, 320),       # three stages for two CTAs, the last one half full
    (17, 128, 128, 16),        # one stage
    (129, 128, 9600, 64),      # tiles of 256 columns, half of the last one missing
    (200, 4096, 128, 2048),    # behind the grid-wide front
    (1025, 2048, 384, 0),      # more rows than the CTA pairs' line, tiles in one wave
    (2049, 2176, 1152, 1088)]) # the same in tiles of 256 columns
def test_dense_tiles_and_splits(T, K, N, nsel):
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator().manual_seed(T + K + N)
    x = torch.randn(T, K, generator=g)
    x[:, 3] *= 20
    x = x.to(torch.bfloat16)
    w = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    wo = MC.oracle_weights(w[None])
    o = M.dense_w4a4_rac(MC.f32(x), wo["codes"][0], wo["sf"][0], wo["gs"][0], nsel)
    wq = B.fake_quant_weights(w.unsqueeze(0).cuda(), want_fq=False, sf_layout=B.SF_TILED)
    res = B.dense_w4a4_rac(x.cuda(), wq, nsel, export=True)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    MC.check_site1(res, dict(site13=o["site"]), nsel, {})
    got = MC.f32(res["out"]).astype(np.float64)
    assert float((np.abs(got - o["y64"]) / MC.gemm_tol(o["absdot"], o["y64"])).max()) <= 1.0


@pytest.mark.parametrize("T,K,N", [
    (1, 4096, 128),        # eight CTAs per tile
    (70, 4096, 1024),      # four
    (256, 2048, 2048),     # two, every row of both row tiles
    (129, 384, 640),       # one, one row in the second row tile
    (9000, 128, 384),      # tiles of 256 columns, half of the last one missing
    (9000, 2176, 384)])    # the same number of tiles with a longer K: pairs, fewer tiles than pairs of SMs
def test_bf16_product_of_one_wave(T, K, N):
    """Against a float64 product of the same bf16 values: float32 accumulation of K exact products is within
    K * 2^-24 * sum|a b| of it (partial sums of a split included), the result is rounded to bf16 once."""
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(T + K + N)
    x = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    w = (torch.randn(N, K, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    res = B.dense_one_sided(x, B.W16A16, w_bf16=w)
    torch.cuda.synchronize()
    assert B.moe_async_status(res["workspace"]) == 0
    want = x.double() @ w.double().t()
    mag = x.double().abs() @ w.double().abs().t()
    err = (res["out"].double() - want).abs()
    assert bool((err <= K * 2.0 ** -24 * mag + 2.0 ** -8 * want.abs() + 1e-30).all())


@pytest.mark.parametrize("T,K", [(513, 512), (2049, 4096), (2047, 4096)])      # either side of the two forms of the amax
def test_scale_of_x_and_scores_behind_either_amax(T, K):
    """The per-tensor scale and the codes are those of the stand-alone quantizer, twice in a row on one workspace (words of the
    first call must not survive)."""
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(T)
    w = B.fake_quant_weights(torch.randn(1, 128, K, device="cuda", generator=g).to(torch.bfloat16), want_fq=False, sf_layout=B.SF_TILED)
    ws = torch.empty(B.moe_workspace_bytes(T, K, 0, 1, 1, 128), dtype=torch.uint8, device="cuda").fill_(255)
    for scale in (30.0, 0.1):
        x = (torch.randn(T, K, device="cuda", generator=g) * scale).to(torch.bfloat16)
        res = B.dense_w4a4_rac(x, w, K // 4, export=True, workspace=ws)
        q, sf, gs = B.quantize_nvfp4(x)
        torch.cuda.synchronize()
        assert B.moe_async_status(ws) == 0
        assert torch.equal(res["a13_gs"], gs) and torch.equal(res["xq"], q) and torch.equal(res["xsf"], sf)
        scores = B.rac_channel_scores(x)
        kept = torch.zeros(K, dtype=torch.bool, device="cuda")
        kept[res["sel13"].long()] = True
        assert int(kept.sum()) == K // 4
        # float32 partial sums of T squares, added in float64: relative error below T * 2^-24 each
        assert float(scores[kept].min()) >= float(scores[~kept].max()) * (1 - 2 * T * 2.0 ** -24)
