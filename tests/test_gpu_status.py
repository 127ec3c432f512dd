"""The status word of a call: what an earlier call left in the workspace does not survive, and the time that the stream's
earlier work takes is not counted against a wait of the call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _operands(T, K, N):
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(T + K + N)
    x = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    wb = (torch.randn(N, K, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    return x, wb, B.fake_quant_weights(wb.unsqueeze(0), want_fq=False, sf_layout=B.SF_TILED)


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("mode", ["W4A4", "W4A16", "W16A4", "W16A16"])
@pytest.mark.parametrize("T,K,N", [(64, 512, 512), (513, 512, 128), (9000, 128, 384), (2300, 128, 2176)])
def test_status_of_an_earlier_call_is_cleared(mode, T, K, N, given):
    """Either scale of x in every mode; small and grid-wide fronts, the product of one wave (two widths) and of CTA pairs."""
    from paper_2607_15810_b200 import binding as B
    x, wb, w = _operands(T, K, N)
    gs = torch.tensor([0.002], device="cuda") if given else None
    ws = torch.full((B.moe_workspace_bytes(T, K, 0, 1, 1, N),), 0xFA, dtype=torch.uint8, device="cuda")
    if mode == "W4A4":
        B.dense_w4a4_rac(x, w, 0, a_gs=gs, workspace=ws)
    else:
        B.dense_one_sided(x, getattr(B, mode), w=w, w_bf16=wb, a_gs=gs, workspace=ws)
    assert B.moe_async_status(ws) == 0


def test_status_is_cleared_in_front_of_the_cooperative_quantizer(monkeypatch):
    from paper_2607_15810_b200 import binding as B
    x, wb, _ = _operands(64, 512, 512)
    monkeypatch.setenv("QUADS_QUANT_COOPERATIVE", "1")
    ws = torch.full((B.moe_workspace_bytes(64, 512, 0, 1, 1, 512),), 0xFA, dtype=torch.uint8, device="cuda")
    B.dense_one_sided(x, B.W16A4, w_bf16=wb, workspace=ws)
    assert B.moe_async_status(ws) == 0


def test_long_predecessor_is_not_a_timeout(monkeypatch):
    """W16A16 has no kernel of its own in front of the product, whose launch overlaps with whatever the stream runs before it: here a
    batched quantization that lets its successor start and then waits, on a few SMs, longer than any wait of the product may."""
    from paper_2607_15810_b200 import binding as B
    x, wb, _ = _operands(64, 512, 512)
    want = B.dense_one_sided(x, B.W16A16, w_bf16=wb)["out"].clone()
    ws = torch.empty(B.moe_workspace_bytes(64, 512, 0, 1, 1, 512), dtype=torch.uint8, device="cuda")
    small = torch.ones(2, 16, 64, dtype=torch.bfloat16, device="cuda")
    monkeypatch.setenv("QUADS_NO_RING_QUANT", "1")           # the cooperative kernel, whose wait the hook below makes run out
    B.fake_quant_weights(small)
    torch.cuda.synchronize()
    B.lib.quads_debug_set_quantize_wait.restype = None
    B.lib.quads_debug_set_quantize_wait.argtypes = [B.C.c_int64, B.C.c_int32]
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    B.lib.quads_debug_set_quantize_wait(5_000_000_000, 1)    # SM cycles: 2.5 s at 1965 MHz
    try:
        start.record()
        gs = B.fake_quant_weights(small)["gs"]
        out = B.dense_one_sided(x, B.W16A16, w_bf16=wb, workspace=ws)["out"]
        end.record()
        status = B.moe_async_status(ws)
    finally:
        B.lib.quads_debug_set_quantize_wait(0, 0)
    assert bool(torch.isnan(gs).all()) and start.elapsed_time(end) > 2200.0          # (the predecessor did take that long)
    assert status == 0 and torch.equal(out, want)
