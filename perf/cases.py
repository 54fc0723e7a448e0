"""The work that users of this package have it do, as measured cases: the verify step on device and on host data, the
LM-head statistics alone, and the making of a quantised head, over the range of shapes and weight modes they support.

`listed()` names the cases, `draw()` gives more of the same ranges; `prepare()` builds what a serving loop holds before a
call (inputs from a seed, the resident head in its storage form, the context, the output buffers of a loop that reuses
them), and `run()` is one pass through the public entry points.
"""
from __future__ import annotations

import math

import torch

from paper_2506_18952_b200 import binding, workloads

# Proportions in which groups of 256 vocabulary rows end up at 4, 8 and 16 bits (the widths bench.py draws).
WIDTH_SHARES = ((4, 0.2), (8, 0.7), (16, 0.1))


def _case(name, entry, B, k, H, V, **options):
    c = {"name": name, "entry": entry, "B": B, "k": k, "H": H, "V": V, "weights": "bf16", "q": "bf16", "gate": "target",
         "fallback": "sample", "logits": False, "reuse_out": True, "inputs": "spread"}
    c.update(options)
    return c


def listed():
    return [
        # a toy model: every call is launches, latency and host work
        _case("tiny", "verify", 1, 4, 64, 1000, q="f32", inputs="gauss"),
        # one user on a 7B-class head, bf16: the head streams from HBM once per round of a decode loop; the logits are
        # kept for the caller's log-probabilities
        _case("edge", "verify", 1, 4, 4096, 32000, logits=True, inputs="gauss"),
        # the same head with the mixed 4 / 8 / 16-bit storage that the quantiser makes for small devices
        _case("edge_mixed", "verify", 1, 4, 4096, 32000, weights="mixed", logits=True, inputs="gauss"),
        # a small serving batch that gates on the draft model's own entropy
        _case("serve_b16_draft_gate", "verify", 16, 5, 4096, 32000, gate="draft", inputs="gauss"),
        # a full serving batch; the caller also wants the logits (log-probabilities for its clients)
        _case("batched_logits", "verify", 64, 5, 4096, 32000, logits=True, inputs="gauss"),
        # large vocabulary, half batch, the mixed-width head expanded on chip
        _case("large_vocab_b32_mixed", "verify", 32, 5, 4096, 128256, weights="mixed"),
        # large vocabulary, half batch, 8-bit weights and hidden rows, greedy verifier
        _case("large_vocab_b32_w8a8", "verify", 32, 5, 4096, 128256, weights="w8a8", fallback="greedy"),
        # large vocabulary, full batch: the headline shape
        _case("large_vocab", "verify", 64, 5, 4096, 128256),
        # 70B-class head, the largest batch: several passes of the verify rows over the head
        _case("wide", "verify", 256, 8, 8192, 128256, inputs="peaked"),
        # an engine whose per-step data lives in pinned host memory: copies in, step, results out
        _case("host_batched", "host", 64, 5, 4096, 32000, inputs="gauss"),
        # statistics and logits only, odd sizes (no multiple of 4 in the vocabulary, a ragged last K block), fresh outputs
        _case("lm_head_ragged", "lm_head", 23, 3, 1032, 50003, logits=True, reuse_out=False),
        # loading a model: the bf16 head is turned into the mixed-width form
        _case("quantize_mixed", "quantize", 1, 1, 4096, 32000, weights="mixed", inputs="gauss"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choices(["verify", "host", "lm_head", "quantize"], [70, 10, 10, 10])[0]
    weights = "mixed" if entry == "quantize" else (
        rng.choices(["bf16", "mixed", "int8", "w8a8", "w8a16"], [50, 20, 8, 12, 10])[0] if entry == "verify" else "bf16")
    step = {"bf16": 8, "mixed": 128}.get(weights, 16)
    while True:
        B, k = _log_int(rng, 1, 256), rng.randint(1, 8)
        V = _log_int(rng, 1000, 128256)
        if rng.random() < 0.5:
            V += -V % 4
        H = max(step, _log_int(rng, 64, 8192) // step * step)
        macs = B * (k + 1) * V * H
        # no dearer than the largest listed case: bf16 anywhere in the range, the other modes and the host entry less
        limit = 256 * 9 * 128256 * 8192 if weights == "bf16" else 256 * 9 * 128256 * 8192 // 4
        if entry == "host" and B * k * V > 64 * 5 * 128256:
            continue
        if macs <= limit and V <= 128256:
            break
    if entry == "quantize":
        B, k = 1, 1
    logits = entry == "lm_head" or (entry == "verify" and rng.random() < 0.25)
    gate = "draft" if entry == "verify" and rng.random() < 0.2 else "target"
    fallback = "greedy" if entry in ("verify", "host") and rng.random() < 0.2 else "sample"
    c = _case("", entry, B, k, H, V, weights=weights, q=rng.choice(["bf16", "bf16", "f32"]), gate=gate,
              fallback=fallback, logits=logits, reuse_out=rng.random() < 0.7,
              inputs="gauss" if entry == "quantize" else rng.choice(["spread", "gauss"]))
    del c["name"]
    return c


def _inputs(case, seed, device):
    B, k, H, V = case["B"], case["k"], case["H"], case["V"]
    q_dtype = torch.float32 if case["q"] == "f32" else torch.bfloat16
    # logits keep the spread of a trained head whatever H is: std 1.28, as N(0,1) rows on 0.02 N(0,1) weights at H = 4096
    w_std = 1.28 / math.sqrt(H)
    if case["inputs"] == "gauss":
        # half the sequences with a draft model close to the verifier, half with one that is off
        return workloads.gaussian_head("perf", B, k, H, V, seed=seed, device=device, w_std=w_std, sigma=0.1,
                                       sigma_far=2.0, q_dtype=q_dtype)
    if case["inputs"] == "peaked":
        return workloads.peaked_flat_head("perf", B, k, H, V, seed=seed, device=device, q_dtype=q_dtype)
    return workloads.entropy_spread_head("perf", B, k, H, V, seed=seed, device=device, w_std=w_std, q_dtype=q_dtype,
                                         tau=2.0)


def _widths(V):
    g = torch.Generator().manual_seed(V)          # a property of the model, not of the inputs
    shares = torch.tensor([s for _, s in WIDTH_SHARES])
    at = torch.multinomial(shares, -(-V // binding.GROUP_ROWS), replacement=True, generator=g)
    return [WIDTH_SHARES[i][0] for i in at.tolist()]


def prepare(case, seed):
    device = torch.device("cuda", torch.cuda.current_device())
    s = {"case": case}
    if case["entry"] == "quantize":
        g = torch.Generator(device=device).manual_seed(seed)
        s["W"] = (torch.randn((case["V"], case["H"]), generator=g, device=device) * 0.02).to(torch.bfloat16)
        s["widths"] = _widths(case["V"])
        return s
    w = _inputs(case, seed, device)
    s.update(hidden=w.hidden, tok=w.draft_tok, q=w.draft_q, u=w.uniforms, tau=w.tau, W=w.W_lm, w_scale=None)
    if case["weights"] == "mixed":
        s["W"] = binding.hola_quantize_mixed(w.W_lm, _widths(case["V"]))
    elif case["weights"] != "bf16":
        s["W"], s["w_scale"] = binding.hola_quantize_w8(w.W_lm)
    s["a8"] = {"w8a8": True, "w8a16": "a16"}.get(case["weights"], False)
    s["ctx"] = binding.HolaVerify(case["B"], case["k"], case["H"], case["V"])
    if case["entry"] == "host":
        for name in ("hidden", "tok", "q", "u"):
            s[name] = s[name].cpu().pin_memory()
        s["out"] = s["ctx"].alloc_outputs(case["B"], case["k"], False, device=torch.device("cpu"))
    else:
        s["out"] = s["ctx"].alloc_outputs(case["B"], case["k"], case["logits"]) if case["reuse_out"] else None
    return s


def run(s):
    case = s["case"]
    if case["entry"] == "quantize":
        head = binding.hola_quantize_mixed(s["W"], s["widths"])
        return {"W16": head.W16, "W8": head.W8, "W4": head.W4, "shift4": head.shift4, "w_scale": head.w_scale}
    ctx = s["ctx"]
    if case["entry"] == "lm_head":
        out = ctx.hola_lm_head_entropy(s["hidden"], s["W"], out=s["out"], want_logits=True, w_scale=s["w_scale"],
                                       a8=s["a8"])
        return {"entropy": out.entropy, "logZ": out.logZ, "logits": out.logits}
    options = dict(gate_source=binding.HOLA_GATE_DRAFT_ENTROPY if case["gate"] == "draft" else binding.HOLA_GATE_TARGET_ENTROPY,
                   fallback=binding.HOLA_FALLBACK_GREEDY if case["fallback"] == "greedy" else binding.HOLA_FALLBACK_SAMPLE,
                   w_scale=s["w_scale"], a8=s["a8"])
    if case["entry"] == "host":
        out = ctx.hola_verify_host(s["hidden"], s["W"], s["tok"], s["q"], s["u"], s["tau"], out=s["out"], **options)
    else:
        out = ctx.hola_verify(s["hidden"], s["W"], s["tok"], s["q"], s["u"], s["tau"], out=s["out"],
                              want_logits=case["logits"], **options)
    got = {"accept_len": out.accept_len, "next_tok": out.next_tok, "entropy": out.entropy, "logZ": out.logZ}
    if case["logits"]:
        got["logits"] = out.logits
    if case["gate"] == "draft":
        got["draft_entropy"] = out.draft_entropy
    return got


def work(case):
    B, k, H, V = case["B"], case["k"], case["H"], case["V"]
    M = B * (k + 1)
    per_weight = {"bf16": 2.0, "mixed": sum(share * bits / 8 for bits, share in WIDTH_SHARES)}.get(case["weights"], 1.0)
    head = V * H * per_weight
    if case["entry"] == "quantize":
        return {"bytes": V * H * 2 + head + V * 4, "flops": 0}
    n = head + (0 if case["weights"] == "bf16" else V * 4) + M * H * 2 + M * 8
    if case["logits"]:
        n += M * V * 4
    if case["entry"] != "lm_head":
        q = 4 if case["q"] == "f32" else 2
        n += B * (k + 1) * 8 + B * 8
        if case["gate"] == "draft":
            n += B * k * V * q                       # every draft row
        elif case["fallback"] == "sample":
            n += B * V * q + B * k * q               # one draft row per sequence and the draft tokens' probabilities
    return {"bytes": n, "flops": 2 * M * V * H}


def tolerance(case):
    if case["entry"] == "quantize":
        return "exact"
    # Against the same path in 64 bits (fp32 accumulation of bf16 products, fp32 softmax sums): relative error of logits /
    # entropy / logZ 6e-8 / 2e-8 / 3e-8 at H = 64, 1.0e-6 / 1.5e-6 / 0.9e-6 at 1032, 4.4e-6 / 7.0e-6 / 3.8e-6 at 4096
    # and, with rows that lead by 15, 1.1e-5 / 1.2e-5 / 2.5e-5 at 8192: it grows with the number of products.  Largest
    # single differences 5.6e-5 at 4096.  Four times that.  Whole numbers: a token may move where its uniform sits
    # within rounding of a boundary of the cumulative mass.
    rel = max(2e-6, 7e-9 * case["H"]) * (1.7 if case["inputs"] == "peaked" else 1.0)
    return {"rel": rel, "max": 8 * rel, "differ": 0.01}
