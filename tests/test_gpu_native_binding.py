"""The binding's native calls against its ctypes path: the same results, objects and errors, each through the path it is meant for."""
from collections import OrderedDict

import pytest
import torch

pytestmark = pytest.mark.gpu


class Sub(torch.Tensor):
    pass


class Recorder:
    """The native module, with what became of each call: "done", the status of its error, or None where it was left to ctypes."""

    def __init__(self, module):
        self.module, self.seen = module, []

    def __getattr__(self, name):
        def call(*args):
            from paper_2607_15810_b200 import binding as B
            try:
                r = getattr(self.module, name)(*args)
            except B.QuadsError as e:
                self.seen.append(e.status)
                raise
            self.seen.append(None if r is None else "done")
            return r
        return call


def _both(monkeypatch, B, call):
    """The call's result (or status of its error) through either path, and what the native function made of it."""
    got = []
    assert B._native is not None
    rec = Recorder(B._native)
    for native in (rec, None):
        monkeypatch.setattr(B, "_native", native)
        try:
            r = call()
            got.append(r)
        except B.QuadsError as e:
            got.append(e.status)
    assert len(rec.seen) == 1
    return got + rec.seen


def _same(a, b):
    if isinstance(a, dict):
        assert a.keys() == b.keys()
        wa, wb = a["workspace"], b["workspace"]
        assert wa.dtype == wb.dtype and wa.shape == wb.shape and wa.device == wb.device
        return _same(a["out"], b["out"])
    if isinstance(a, tuple):
        assert len(a) == len(b)
        return all(_same(x, y) for x, y in zip(a, b))
    if isinstance(a, torch.Tensor):
        return a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)
    return a == b


def test_same_results_objects_and_errors(monkeypatch):
    from paper_2607_15810_b200 import binding as B
    g = torch.Generator(device="cuda").manual_seed(3)
    def bf(*shape):
        return (torch.randn(*shape, device="cuda", generator=g) * 0.5).to(torch.bfloat16)
    T, H, I, E = 40, 256, 128, 8
    x, lg = bf(T, H), torch.randn(T, E, device="cuda", generator=g)
    w13, w2 = (B.fake_quant_weights(bf(E, *s), want_fq=False, sf_layout=B.SF_TILED) for s in ((2 * I, H), (H, I)))
    p13, p2 = (B.fp8_quantize_weights(bf(E, *s)) for s in ((2 * I, H), (H, I)))
    wb = bf(384, H)
    w = B.fake_quant_weights(wb.unsqueeze(0), want_fq=False, sf_layout=B.SF_TILED)
    a2, gs = torch.tensor([0.01], device="cuda"), torch.tensor([0.002], device="cuda")
    wide = bf(T, 2 * H)[:, :H]                                              # a row stride
    tiled = (torch.empty(T, H // 2, dtype=torch.uint8, device="cuda"), torch.zeros(B.sf_tiled_bytes(T, H), dtype=torch.uint8, device="cuda"),
             torch.empty(1, device="cuda"))
    native = [
        lambda: B.moe_w4a4_rac(x, lg, w13, w2, 2, H // 2, I // 2, a2),
        lambda: B.moe_w4a4_rac(x, lg, w13, w2, 2, 0, 0, a2, a13_gs=gs, renormalize=False),
        lambda: B.moe_fp8_w8a8(x, lg, p13, p2, 2),
        lambda: B.dense_w4a4_rac(x, w, 64), lambda: B.dense_w4a4_rac(x, w, 0, a_gs=gs),
        lambda: B.dense_one_sided(x, B.W4A16, w=w), lambda: B.dense_one_sided(x, B.W16A4, w_bf16=wb, a_gs=gs),
        lambda: B.dense_one_sided(x, B.W16A16, w_bf16=wb), lambda: B.dense_w4a4_rac(torch.nn.Parameter(x), w, 64),
        lambda: B.quantize_nvfp4(x), lambda: B.quantize_nvfp4(x, gs=gs), lambda: B.quantize_nvfp4(wide),
        lambda: B.quantize_nvfp4(x[:1, :48]), lambda: B.quantize_nvfp4(x, sf_layout=B.SF_TILED, out=tiled)]
    refused = [
        lambda: B.dense_w4a4_rac(x, w, H + 1), lambda: B.moe_w4a4_rac(x, lg, w13, w2, 9, 0, 0, a2),
        lambda: B.moe_w4a4_rac(x, lg, w13, w2, 2, 0, 0, None), lambda: B.quantize_nvfp4(x[:, :40]),
        lambda: B.dense_w4a4_rac(x, w, 64, workspace=torch.empty(512, dtype=torch.uint8, device="cuda"))]
    left_to_ctypes = [
        lambda: B.dense_w4a4_rac(x.as_subclass(Sub), w, 64), lambda: B.dense_w4a4_rac(x, OrderedDict(w), 64), lambda: B.dense_w4a4_rac(x, w, True),
        lambda: B.moe_w4a4_rac(x, lg.as_subclass(Sub), w13, w2, 2, 0, 0, a2), lambda: B.moe_fp8_w8a8(x.as_subclass(Sub), lg, p13, p2, 2),
        lambda: B.dense_one_sided(x.as_subclass(Sub), B.W16A16, w_bf16=wb),
        lambda: B.quantize_nvfp4(x.as_subclass(Sub)), lambda: B.quantize_nvfp4(x, sf_layout=B.SF_TILED, out=list(tiled))]
    for group, calls in (("done", native), ("refused", refused), (None, left_to_ctypes)):
        for i, call in enumerate(calls):
            a, b, seen = _both(monkeypatch, B, call)
            monkeypatch.undo()
            assert _same(a, b), (group, i)
            assert seen == (a if group == "refused" else group), (group, i)
            assert (group == "refused") == isinstance(a, int), (group, i)
    for bad in (lambda: B.quantize_nvfp4(x.float()), lambda: B.quantize_nvfp4(x.t()), lambda: B.quantize_nvfp4(x.cpu())):
        rec = Recorder(B._native)
        monkeypatch.setattr(B, "_native", rec)
        with pytest.raises(AssertionError):
            bad()
        monkeypatch.undo()
        assert rec.seen == [None]
    # the caller's buffers come back as they are
    ws = torch.empty(B.moe_workspace_bytes(T, H, I, E, 2), dtype=torch.uint8, device="cuda")
    out = torch.empty(T, H, dtype=torch.bfloat16, device="cuda")
    r = B.moe_w4a4_rac(x, lg, w13, w2, 2, 0, 0, a2, workspace=ws, out=out)
    assert r["out"] is out and r["workspace"] is ws
    outs = (torch.empty(T, H // 2, dtype=torch.uint8, device="cuda"), torch.empty(T, H // 16, dtype=torch.uint8, device="cuda"),
            torch.empty(1, device="cuda"))
    assert all(p is q for p, q in zip(B.quantize_nvfp4(x, out=outs), outs))


def test_calls_on_the_current_stream():
    """A call inside torch.cuda.stream is ordered behind that stream's work."""
    from paper_2607_15810_b200 import binding as B
    x = torch.zeros(4096, 4096, dtype=torch.bfloat16, device="cuda")
    want = B.quantize_nvfp4(torch.full_like(x, 3.0))
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for _ in range(20):
            x.add_(1.0).sub_(1.0)
        x.fill_(3.0)
        got = B.quantize_nvfp4(x)
    s.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
