"""Where a dense projection's result goes: outputs aligned to 16 bytes only, rows that end inside a row tile."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["W4A4", "W4A16", "W16A16"])
@pytest.mark.parametrize("T,K,N", [(1, 256, 128), (33, 128, 384), (130, 256, 256), (2300, 128, 1152)])
def test_output_aligned_to_16_bytes(mode, T, K, N):
    """The same bits as for an aligned output, and nothing written beside them."""
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(T + N)
    x = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    wb = (torch.randn(N, K, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    w = B.fake_quant_weights(wb.unsqueeze(0), want_fq=False, sf_layout=B.SF_TILED)
    if mode == "W4A4":
        want = B.dense_w4a4_rac(x, w, K // 2)["out"]
    else:
        want = B.dense_one_sided(x, getattr(B, mode), w=w, w_bf16=wb)["out"]
    buf = torch.full((T * N + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(B.moe_workspace_bytes(T, K, 0, 1, 1, N), dtype=torch.uint8, device="cuda")
    a = B.MoEArgs()
    a.T, a.H, a.I, a.E, a.topk, a.N = T, K, 0, 1, 1, N
    a.x, a.out = x.data_ptr(), buf.data_ptr() + 16
    a.w13_q, a.w13_sf, a.w13_gs, a.w13_bf16 = w["q"].data_ptr(), w["sf"].data_ptr(), w["gs"].data_ptr(), wb.data_ptr()
    a.rac_nsel_13 = K // 2 if mode == "W4A4" else 0
    a.operand_mode = getattr(B, mode)
    a.workspace, a.workspace_bytes = ws.data_ptr(), ws.numel()
    B.check(B.lib.quads_moe_w4a4_rac(C.byref(a), B._stream()))
    torch.cuda.synchronize()
    assert torch.equal(buf[8:8 + T * N].view(T, N), want)
    assert bool((buf[:8] == 7.0).all()) and bool((buf[8 + T * N:] == 7.0).all())
