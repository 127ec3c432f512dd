"""The dense projection with few output tiles, at the edges of its tile width and of its split of K; the rings of the larger
tiles; operands that the preceding kernel has only just written."""
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
    (2049, 2176, 1152, 1088),  # the same in tiles of 256 columns
    (1030, 2048, 4352, 0),     # CTA pairs without a residual: eight K steps through five stages, six rows in the last row tile
    (1030, 1664, 4352, 0),     # the same with a half-full last K step
    (1030, 1664, 4352, 832)])  # with a residual, four stages
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
    (70, 4096, 1024),      # eight, a tile of 70 rows
    (70, 1408, 512),       # four
    (256, 2048, 2048),     # two, every row of both row tiles
    (661, 2176, 640),      # two, where four would fit, too
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


def _fill(gen, t, std):
    t.copy_((torch.randn(t.shape, device="cuda", generator=gen) * std).to(torch.bfloat16))


def test_operands_written_right_before_the_call():
    """What a loader fetches ahead of the preceding kernel's end is complete all the same: weights packed or decoded, and an x computed,
    by the library's kernels immediately before the call, in buffers that hold other values every time.  A chain without a
    synchronisation against the same chain with one behind every call."""
    from paper_2607_15810_b200 import binding as B
    T, K, N = 64, 4096, 4096

    def chain(sync):
        g = torch.Generator(device="cuda").manual_seed(11)
        x, wb = (torch.empty(n, K, dtype=torch.bfloat16, device="cuda") for n in (T, N))
        packed = (None, torch.empty(1, N, K // 2, dtype=torch.uint8, device="cuda"),
                  torch.zeros(1, B.sf_tiled_bytes(N, K), dtype=torch.uint8, device="cuda"), torch.empty(1, device="cuda"))
        dec = torch.empty(1, N, K, dtype=torch.bfloat16, device="cuda")
        ws = torch.empty(B.moe_workspace_bytes(T, K, 0, 1, 1, N), dtype=torch.uint8, device="cuda")
        wait = torch.cuda.synchronize if sync else (lambda: None)
        got = []
        for _ in range(12):
            _fill(g, x, 1.0)
            _fill(g, wb, 0.02)
            wait()
            w = B.fake_quant_weights(wb.view(1, N, K), want_fq=False, sf_layout=B.SF_TILED, out=packed)
            wait()
            y = B.dense_w4a4_rac(x, w, K // 2, workspace=ws)["out"]                    # weights older than the front by one kernel
            wait()
            z = B.dense_one_sided(y, B.W4A16, w=w, workspace=ws)["out"]                # x: the result just above
            wait()
            B.dequantize_nvfp4(w["q"], w["sf"], w["gs"], N, K, sf_layout=B.SF_TILED, out=dec)
            wait()
            u = B.dense_one_sided(z, B.W16A4, w_bf16=dec[0], workspace=ws)["out"]      # weights decoded just above
            wait()
            v = B.dense_one_sided(u, B.W16A16, w_bf16=dec[0], workspace=ws)["out"]
            wait()
            t = B.dense_w4a4_rac(v, w, 0, workspace=ws)["out"]
            wait()
            got += [y, z, u, v, t]
        torch.cuda.synchronize()
        return got

    for i, (a, b) in enumerate(zip(chain(False), chain(True))):
        assert torch.equal(a, b), (i // 5, i % 5)
