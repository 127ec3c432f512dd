"""The calls a program makes into this library, as cases to be timed: the MoE layer at decode, mixed and
prefill sizes, the dense projection, the one-sided projections of the learner's side, the FP8 layer the
NVFP4 one is compared with, the activation quantizer and the trainer's weight fake-quant.

A case is a dict of plain values.  `prepare` makes what a program holds before the call (inputs of a seed,
packed weights, workspace and, where a loop would keep them, output buffers), `run` makes the one public
call.  Value distributions are those of `paper_2607_15810_b200.synth`, drawn on the device."""
import math

import numpy as np
import torch

from paper_2607_15810_b200 import binding as B

# Expert layers: hidden size, SwiGLU width, weight std, heavy activation channels (count, degrees of freedom
# of their Student-t values, scale), static scale of h, the largest batch drawn for them.
LAYERS = {
    "2048": dict(H=2048, I=768, std=0.02, heavy=(20, 3.0, 10.0), a2=0.25, t_max=8192),
    "4096": dict(H=4096, I=1536, std=0.015, heavy=(20, 2.5, 16.0), a2=0.5, t_max=4096),
}
EXPERTS, TOPK = 128, 8
# Residual compensation: share of the channels at the input of W13 and of W2.
VARIANTS = {"both": (0.5, 0.5), "w13": (0.5, 0.0), "plain": (0.0, 0.0)}
# Expert weights [rows, K] of the two layers, as the trainer fake-quantizes them.
EXPERT_SHAPES = [(1536, 2048), (2048, 768), (3072, 4096), (4096, 1536)]
MAX_FAKE_QUANT_ELEMENTS = 128 * 1536 * 2048
MODES = {"w4a16": B.W4A16, "w16a4": B.W16A4, "w16a16": B.W16A16}


def listed():
    return [
        # one sequence decoding: 8 of 128 experts' weights, everything else is latency
        dict(name="moe_decode_1", kind="moe", layer="2048", T=1, variant="both", hot=0),
        # a small decode batch of an odd size, compensated where the paper deploys it
        dict(name="moe_decode_61_w13", kind="moe", layer="2048", T=61, variant="w13", hot=0),
        # the decode batch of the benchmark: all experts' weights streamed for 16 rows each
        dict(name="moe_decode_256", kind="moe", layer="2048", T=256, variant="both", hot=0),
        # one chunk of a chunked prefill, ragged: 94 rows per expert, less than a row tile
        dict(name="moe_chunk_1500_w13", kind="moe", layer="2048", T=1500, variant="w13", hot=0),
        # the prefill batch of the benchmark, a quarter of the assignments on eight hot experts
        dict(name="moe_prefill_8192", kind="moe", layer="2048", T=8192, variant="both", hot=8),
        # the larger layer at its prefill size
        dict(name="moe_large_4096", kind="moe", layer="4096", T=4096, variant="both", hot=0),
        # the FP8 layer at the decode batch, what rollout throughput is compared with
        dict(name="moe_fp8_decode_256", kind="moe_fp8", layer="2048", T=256, hot=0),
        # the smallest projection configuration: 128 x 512 -> 256, 16 channels compensated
        dict(name="dense_128", kind="dense", T=128, K=512, N=256, nsel=16),
        # a projection at model scale: 8192 x 4096 -> 4096, half of the channels compensated
        dict(name="dense_8192", kind="dense", T=8192, K=4096, N=4096, nsel=2048),
        # the asymmetric-QAT learner's forward: packed weights decoded, bf16 activations
        dict(name="w4a16_2048", kind="one_sided", mode="w4a16", T=2048, K=4096, N=4096),
        # online activation quantization of the prefill batch, per-tensor scale from the data
        dict(name="quantize_8192", kind="quantize", rows=8192, K=2048, tiled=False, given=False),
        # one layer's W13 on the trainer: fake-quant plus the packed bytes of the weight sync
        dict(name="fake_quant_128", kind="fake_quant", n=128, N=1536, K=2048, tiled=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["moe", "moe", "moe", "moe", "moe_fp8", "dense", "one_sided", "quantize", "fake_quant"])
    if kind == "moe":
        layer = rng.choice(["2048", "2048", "4096"])
        T = _log_int(rng, 1, LAYERS[layer]["t_max"])
        return dict(kind=kind, layer=layer, T=T, variant=rng.choice(["both", "both", "w13", "plain"]),
                    hot=8 if T >= 1024 and rng.random() < 0.5 else 0)
    if kind == "moe_fp8":
        T = _log_int(rng, 1, 8192)
        return dict(kind=kind, layer="2048", T=T, hot=8 if T >= 1024 and rng.random() < 0.5 else 0)
    if kind == "dense":
        K = 128 * _log_int(rng, 4, 32)
        return dict(kind=kind, T=_log_int(rng, 1, 8192), K=K, N=128 * _log_int(rng, 2, 32),
                    nsel=K * rng.choice([0, 1, 2, 4, 8]) // 8)
    if kind == "one_sided":
        return dict(kind=kind, mode=rng.choice(["w4a16", "w4a16", "w16a4", "w16a16"]), T=_log_int(rng, 64, 8192),
                    K=128 * _log_int(rng, 4, 32), N=128 * _log_int(rng, 4, 32))
    if kind == "quantize":
        return dict(kind=kind, rows=_log_int(rng, 1, 16384), K=16 * _log_int(rng, 16, 256), tiled=rng.random() < 0.5,
                    given=rng.random() < 0.4)
    N, K = rng.choice(EXPERT_SHAPES)
    return dict(kind=kind, n=_log_int(rng, 1, MAX_FAKE_QUANT_ELEMENTS // (N * K)), N=N, K=K, tiled=rng.random() < 0.7)


# ---------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _activations(gen, seed, T, K, heavy):
    """N(0, 1) with a few channels of Student-t values, bf16."""
    count, nu, scale = heavy
    x = torch.randn(T, K, device="cuda", generator=gen)
    rng = np.random.default_rng(seed + 17)
    channels = torch.from_numpy(np.sort(rng.choice(K, size=count, replace=False))).cuda()
    x[:, channels] = torch.from_numpy((rng.standard_t(nu, size=(T, count)) * scale).astype(np.float32)).cuda()
    return x.to(torch.bfloat16)


def _router_logits(gen, T, hot):
    """N(0, 1); with `hot` experts, biased until those get a quarter of the assignments."""
    logits = torch.randn(T, EXPERTS, device="cuda", generator=gen)
    if hot:
        lo, hi = 0.0, 4.0
        for _ in range(12):
            bias = 0.5 * (lo + hi)
            z = logits.clone()
            z[:, :hot] += bias
            share = (z.topk(TOPK, dim=1).indices < hot).float().mean().item()
            lo, hi = (bias, hi) if share < 0.25 else (lo, bias)
        logits[:, :hot] += bias
    return logits.contiguous()


def _weight(gen, rows, K, std):
    w = torch.empty(rows, K, dtype=torch.bfloat16, device="cuda")
    return w.normal_(0.0, std, generator=gen)


def _packed_experts(gen, N, K, std, fp8):
    """The weights of all experts, drawn and packed a few experts at a time."""
    parts = []
    for _ in range(0, EXPERTS, 16):
        w = _weight(gen, 16 * N, K, std).view(16, N, K)
        parts.append(B.fp8_quantize_weights(w) if fp8 else B.fake_quant_weights(w, want_fq=False, sf_layout=B.SF_TILED))
    return {k: torch.cat([p[k] for p in parts]) for k in parts[0] if parts[0][k] is not None}


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("moe", "moe_fp8"):
        c = LAYERS[case["layer"]]
        H, I, T = c["H"], c["I"], case["T"]
        s["x"] = _activations(gen, seed, T, H, c["heavy"])
        s["logits"] = _router_logits(gen, T, case["hot"])
        s["w13"] = _packed_experts(gen, 2 * I, H, c["std"], kind == "moe_fp8")
        s["w2"] = _packed_experts(gen, H, I, c["std"], kind == "moe_fp8")
        s["out"] = torch.empty(T, H, dtype=torch.bfloat16, device="cuda")
        if kind == "moe":
            f13, f2 = VARIANTS[case["variant"]]
            s["nsel"] = int(H * f13), int(I * f2)
            s["a2"] = torch.tensor([c["a2"]], dtype=torch.float32, device="cuda")
            s["ws"] = _bytes(B.moe_workspace_bytes(T, H, I, EXPERTS, TOPK))
        else:
            s["ws"] = _bytes(B.moe_fp8_workspace_bytes(T, H, I, EXPERTS, TOPK))
    elif kind in ("dense", "one_sided"):
        T, K, N = case["T"], case["K"], case["N"]
        s["x"] = _activations(gen, seed, T, K, (4, 3.0, 10.0))
        s["w_bf16"] = _weight(gen, N, K, 0.02)
        s["w"] = B.fake_quant_weights(s["w_bf16"].view(1, N, K), want_fq=False, sf_layout=B.SF_TILED)
        s["ws"] = _bytes(B.moe_workspace_bytes(T, K, 0, 1, 1, N))
    elif kind == "quantize":
        s["x"] = _activations(gen, seed, case["rows"], case["K"], (4, 3.0, 10.0))
        s["gs"] = torch.tensor([100.0 / 2688.0], dtype=torch.float32, device="cuda") if case["given"] else None
        s["ws"] = _bytes(B.lib.quads_quantize_workspace_bytes())
        if case["tiled"]:                      # a GEMM operand's buffers are kept; its padding scales stay zero
            rows, K = case["rows"], case["K"]
            s["outs"] = (torch.empty(rows, K // 2, dtype=torch.uint8, device="cuda"),
                         torch.zeros(B.sf_tiled_bytes(rows, K), dtype=torch.uint8, device="cuda"),
                         torch.empty(1, dtype=torch.float32, device="cuda"))
    else:
        n, N, K = case["n"], case["N"], case["K"]
        w = torch.empty(n, N, K, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.015, generator=gen)
        per = B.sf_tiled_bytes(N, K) if case["tiled"] else N * (K // 16)
        s["x"] = w
        s["outs"] = (torch.empty_like(w), torch.empty(n, N, K // 2, dtype=torch.uint8, device="cuda"),
                     torch.zeros(n, per, dtype=torch.uint8, device="cuda"), torch.empty(n, dtype=torch.float32, device="cuda"))
        s["ws"] = _bytes(B.lib.quads_fake_quant_workspace_bytes(n))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "moe":
        return B.moe_w4a4_rac(s["x"], s["logits"], s["w13"], s["w2"], TOPK, s["nsel"][0], s["nsel"][1], s["a2"],
                              workspace=s["ws"], out=s["out"])["out"]
    if kind == "moe_fp8":
        return B.moe_fp8_w8a8(s["x"], s["logits"], s["w13"], s["w2"], TOPK, workspace=s["ws"], out=s["out"])["out"]
    if kind == "dense":
        return B.dense_w4a4_rac(s["x"], s["w"], case["nsel"], workspace=s["ws"])["out"]
    if kind == "one_sided":
        return B.dense_one_sided(s["x"], MODES[case["mode"]], w=s["w"], w_bf16=s["w_bf16"], workspace=s["ws"])["out"]
    if kind == "quantize":
        return B.quantize_nvfp4(s["x"], gs=s["gs"], sf_layout=B.SF_TILED if case["tiled"] else B.SF_LINEAR,
                                out=s.get("outs"), workspace=s["ws"])
    r = B.fake_quant_weights(s["x"], sf_layout=B.SF_TILED if case["tiled"] else B.SF_LINEAR, out=s["outs"], workspace=s["ws"])
    return r["w_fq"], r["q"], r["sf"], r["gs"]


def work(case):
    """Each input read once, each output written once; the compensated share of a product counted at its
    n_sel / K of the product."""
    kind = case["kind"]
    if kind in ("moe", "moe_fp8"):
        c = LAYERS[case["layer"]]
        H, I, T = c["H"], c["I"], case["T"]
        hit = EXPERTS * (1.0 - (1.0 - TOPK / EXPERTS) ** T)              # experts that get a row
        per_weight = 1.0 if kind == "moe_fp8" else 0.5625
        f13, f2 = VARIANTS[case["variant"]] if kind == "moe" else (0.0, 0.0)
        flops = 2.0 * T * TOPK * (H * 2 * I * (1 + f13) + I * H * (1 + f2))
        return {"bytes": int(hit * 3 * H * I * per_weight + T * (4 * H + 4 * EXPERTS)), "flops": int(flops)}
    if kind == "dense":
        T, K, N = case["T"], case["K"], case["N"]
        return {"bytes": int(2 * T * K + 0.5625 * N * K + 2 * T * N), "flops": 2 * T * N * (K + case["nsel"])}
    if kind == "one_sided":
        T, K, N = case["T"], case["K"], case["N"]
        return {"bytes": int(2 * T * K + (0.5625 if case["mode"] == "w4a16" else 2) * N * K + 2 * T * N), "flops": 2 * T * N * K}
    if kind == "quantize":
        n = case["rows"] * case["K"]
        return {"bytes": int(2.5625 * n), "flops": n}
    n = case["n"] * case["N"] * case["K"]
    return {"bytes": int(4.5625 * n), "flops": n}


def tolerance(case):
    """Relative 2-norm errors: about four times what the path shows against float64 (0.0017 for a bf16 result of
    exact products, 0.0026 for a layer, whose hidden activations are rounded to bf16 and quantized on the way)."""
    kind = case["kind"]
    if kind in ("quantize", "fake_quant"):
        return "exact"                                                   # codes, scale bytes and their exact decode
    return {"rel": 1e-2 if kind in ("moe", "moe_fp8") else 7e-3}
