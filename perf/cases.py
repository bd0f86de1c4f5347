"""The work a user of this library has it do, as measurable cases.

One pass of a case is what a serving loop, an offline evaluation or a fitting run enqueues for one
unit of work, through the public entry points of ``paper_2502_14477_b200`` and nothing else.

Kinds of pass
  step      one ESA step of one layer: append the chunk's K/V, compress its keys, select, attend.  With
            l_C = 1 it is a decode step, with more it is a prefill chunk or a short follow-up question.
  prefill   the whole chunked prefill of one layer (every chunk a step, the last one ragged).
  two       a chunk whose attention uses the two position encodings of Section 3.2.
  host      a step with the K/V cache in pinned host memory (contexts that do not fit the GPU).
  full      the step with full-dimension scores (Eq. 3), or the per-head vote, in place of the compressed
            ones: the comparison and recall runs.
  noalloc   a decode step whose attention is the entry point that allocates nothing.
  fit       a stretch of the compressors' training (Eq. 7) that ends with the weights read back.

Shapes are those of ``esa_synth/configs.py`` (a small 8/2-head model, the Llama-3-8B attention shape with
32/8 heads, a 28/4-head model); contexts run from a thousand tokens to 256k, batches from 1 to 16.
"""
import math

import numpy as np
import torch

import paper_2502_14477_b200 as esa

# (query heads, key/value heads, head dimension)
SMALL, LLAMA, WIDE = (8, 2, 64), (32, 8, 128), (28, 4, 128)


def _case(kind, heads, d_c, B, l_C, t, l_I, l_L, k, eps=3, spread=0, per_head=False, pairs=0):
    """t: tokens cached before the pass (prefill: tokens to process); sequence b of a batch is b * spread tokens
    shorter.  pairs: query-key pairs of a fitting pass, in batches of l_C."""
    return {"kind": kind, "H": heads[0], "H_G": heads[1], "d": heads[2], "d_c": d_c, "B": B, "l_C": l_C, "t": t, "l_I": l_I,
            "l_L": l_L, "k": k, "eps": eps, "spread": spread, "per_head": per_head, "pairs": pairs}


def listed():
    named = {
        # the smallest call: a decode step of the small model, one sequence (latency and launches)
        "decode_small": _case("step", SMALL, 32, 1, 1, 4103, 4, 512, 256),
        # interactive decoding of one long conversation on the Llama-3-8B shape
        "decode_one": _case("step", LLAMA, 128, 1, 1, 32771, 128, 2048, 4096),
        # continuous batching: 16 sequences of different lengths, group of seven query heads
        "decode_batch": _case("step", WIDE, 128, 16, 1, 40009, 128, 2048, 4096, spread=2003),
        # throughput decoding: 8 sequences with 131072 cached tokens each
        "decode_long": _case("step", LLAMA, 128, 8, 1, 131072, 128, 2048, 4096),
        # a follow-up question of a few dozen tokens on a long document
        "question": _case("step", LLAMA, 128, 1, 37, 50021, 128, 2048, 4096),
        # one chunk of a 128k prefill, half way through
        "chunk": _case("step", LLAMA, 128, 1, 512, 65536, 128, 2048, 4096),
        # one chunk of a 256k prefill on the 28/4-head model, chunks of 1024
        "chunk_256k": _case("step", WIDE, 128, 1, 1024, 202752, 128, 4096, 8192),
        # a whole 30000-token prefill of one layer in chunks of 512 (the last chunk is ragged)
        "prefill_30k": _case("prefill", LLAMA, 128, 1, 512, 30000, 128, 2048, 4096),
        # a prefill chunk with the fixed-distance encoding for the initial and selected tokens
        "two_position": _case("two", LLAMA, 128, 1, 512, 40000, 128, 2048, 4096),
        # decoding with the K/V cache off-loaded to host memory
        "decode_host_kv": _case("host", LLAMA, 128, 1, 1, 65543, 128, 2048, 4096),
        # a chunk scored without dimensionality reduction (ground truth of the recall measurement)
        "chunk_full": _case("full", LLAMA, 128, 1, 512, 20480, 128, 2048, 4096),
        # 64 training steps of 128 pairs for one layer's compressors
        "fit": _case("fit", LLAMA, 128, 1, 128, 0, 128, 2048, 4096, pairs=8192),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same kinds and ranges.  Steps, the library's main use, come up most."""
    kind = rng.choice(["step"] * 8 + ["prefill", "two", "two", "host", "full", "full", "noalloc", "fit"])
    heads = rng.choice([SMALL, LLAMA, LLAMA, WIDE])
    d_c = rng.choice([32, 64] if heads is SMALL else [32, 64, 128, 128, 128, 128])
    eps = rng.choice([0, 1, 3, 3, 3, 5])
    l_I = rng.choice([4, 128]) if heads is SMALL else 128
    l_L = _log_int(rng, 512, 1024) if heads is SMALL else _log_int(rng, 1024, 4096)
    k = _log_int(rng, 256, 512) if heads is SMALL else _log_int(rng, 1024, 8192)
    t_max = 8192 if heads is SMALL else 131072
    if kind == "fit":
        return _case("fit", heads, d_c, 1, _log_int(rng, 32, 256), 0, l_I, l_L, k, eps, pairs=_log_int(rng, 1024, 8192))
    if kind == "prefill":
        return _case("prefill", heads, d_c, 1, rng.choice([256, 512, 512, 1000]), _log_int(rng, 4000, min(t_max, 20000)), l_I, l_L, k, eps)
    decode = kind == "noalloc" or rng.random() < 0.5
    if kind == "full":
        decode, t_max = False, min(t_max, 20480)
    if kind == "host":
        t_max = min(t_max, 65536)
    l_C = 1 if decode else _log_int(rng, 2, 1024 if kind != "full" else 512)
    B = 1
    if kind in ("step", "noalloc"):
        B = _log_int(rng, 1, 16) if decode else rng.choice([1, 1, 1, 2])
    t = _log_int(rng, 1000, t_max)
    spread = 0
    if B > 1:
        t = min(t, 8 * 131072 // B)
        spread = rng.randrange(0, t // B)
    return _case(kind, heads, d_c, B, l_C, t, l_I, l_L, k, eps, spread, kind == "full" and rng.random() < 0.5)


# ---------------------------------------------------------------------------- inputs
def _positions(case):
    return [case["t"] - b * case["spread"] for b in range(case["B"])]


def _tensor(gen, *shape):
    """N(0, 1) rows with a scale per head of U(0.5, 2): heads of a trained model differ in size by such factors."""
    x = torch.randn(*shape, device="cuda", dtype=torch.bfloat16, generator=gen)
    scale = 0.5 + 1.5 * torch.rand(shape[-2], 1, device="cuda", generator=gen)
    return x.mul_(scale.to(torch.bfloat16))


def _weights(case, gen):
    dH, dG = case["H"] * case["d"], case["H_G"] * case["d"]
    wq = torch.randn(case["d_c"], dH, device="cuda", generator=gen) / dH ** 0.5
    wk = torch.randn(case["d_c"], dG, device="cuda", generator=gen) / dG ** 0.5
    return wq.cpu().numpy(), wk.cpu().numpy()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    H, HG, d, dc, B, l_C = (case[n] for n in ("H", "H_G", "d", "d_c", "B", "l_C"))
    s = {"case": case}
    wq, wk = _weights(case, gen)
    if case["kind"] == "fit":
        cfg = esa.EsaConfig(H, HG, d, dc, case["l_I"], case["l_L"], case["k"], case["eps"], 1, 1, 16)
        s["fit"] = esa.EsaFit(cfg, l_C, 5e-4)
        s["fit"].set_weights(wq, None, wk, None)
        s["Q"], s["K"] = _tensor(gen, case["pairs"], H, d), _tensor(gen, case["pairs"], HG, d)
        s["loss"] = torch.zeros(-(-case["pairs"] // l_C), 1, device="cuda")
        return s
    prefill = case["kind"] == "prefill"
    n = case["t"] if prefill else case["t"] + l_C
    cfg = esa.EsaConfig(H, HG, d, dc, case["l_I"], case["l_L"], case["k"], case["eps"], l_C, B, n)
    ctx = esa.Esa(cfg)
    ctx.set_compressors(wq, None, wk, None)
    s.update(cfg=cfg, ctx=ctx, t=_positions(case))
    K, V = _tensor(gen, B, n, HG, d), _tensor(gen, B, n, HG, d)
    Kc = torch.zeros(B, n, dc, device="cuda", dtype=torch.bfloat16)
    s["idx"] = torch.zeros(B, case["k"], device="cuda", dtype=torch.int32)
    s["n_sel"] = torch.zeros(B, device="cuda", dtype=torch.int32)
    if prefill:
        # the layer's projections of the whole prompt, and empty caches
        s["Q"], s["K_new"], s["V_new"] = _tensor(gen, B, n, H, d), K, V
        K, V = torch.zeros_like(K), torch.zeros_like(V)
    else:
        s["Q"], s["K_new"], s["V_new"] = _tensor(gen, B, l_C, H, d), _tensor(gen, B, l_C, HG, d), _tensor(gen, B, l_C, HG, d)
        if case["kind"] != "full":
            # compressed keys of the cached tokens, left by the passes before this one
            for r0 in range(0, case["t"], 4096):
                r1 = min(case["t"], r0 + 4096)
                ctx.compress_keys(K[:, r0:r1].contiguous(), Kc, [r0] * B)
    if case["kind"] == "two":
        s["Q_far"], s["K_far"] = _tensor(gen, B, l_C, H, d), _tensor(gen, B, n, HG, d)
    if case["kind"] == "host":
        K[:, case["t"]:], V[:, case["t"]:] = s["K_new"], s["V_new"]
        K, V = K.cpu().pin_memory(), V.cpu().pin_memory()
        rows = case["l_I"] + case["k"] + case["l_L"] + l_C
        s["K_stage"] = torch.empty(B, rows, HG, d, device="cuda", dtype=torch.bfloat16)
        s["V_stage"] = torch.empty_like(s["K_stage"])
    s.update(K=K, V=V, Kc=Kc, O=torch.zeros_like(s["Q"]))
    return s


# ---------------------------------------------------------------------------- one pass
def _run_fit(s):
    fit, Q, K, loss, n = s["fit"], s["Q"], s["K"], s["loss"], s["case"]["l_C"]
    for i in range(loss.shape[0]):
        fit.step(Q[i * n:(i + 1) * n], K[i * n:(i + 1) * n], loss[i])
    return list(fit.get_weights()) + [loss]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fit":
        return _run_fit(s)
    ctx, t, Q, K, V, Kc, idx, n_sel, O = (s[n] for n in ("ctx", "t", "Q", "K", "V", "Kc", "idx", "n_sel", "O"))
    K_new, V_new = s["K_new"], s["V_new"]
    if kind == "prefill":
        step = case["l_C"]
        for p in range(0, case["t"], step):
            q, kn, vn = Q[:, p:p + step], K_new[:, p:p + step], V_new[:, p:p + step]
            ctx.append_kv(kn, vn, K, V, [p])
            ctx.compress_keys(kn, Kc, [p])
            ctx.select(q, Kc, [p], idx, n_sel)
            ctx.attend(q, K, V, [p], idx, n_sel, O[:, p:p + step])
        return O, Kc, idx, n_sel
    if kind != "host":
        ctx.append_kv(K_new, V_new, K, V, t)
    if kind == "full":
        ctx.select_full(Q, K, t, idx, n_sel, per_head=case["per_head"])
    else:
        ctx.compress_keys(K_new, Kc, t)
        ctx.select(Q, Kc, t, idx, n_sel)
    if kind == "two":
        ctx.attend_two_position(Q, s["Q_far"], K, s["K_far"], V, t, idx, n_sel, O)
    elif kind == "host":
        ctx.attend_host_kv(Q, K, V, t, idx, n_sel, s["K_stage"], s["V_stage"], O)
    elif kind == "noalloc":
        esa.attend_noalloc(s["cfg"], Q, K, V, t, idx, n_sel, O)
    else:
        ctx.attend(Q, K, V, t, idx, n_sel, O)
    return (O, idx, n_sel) if kind == "full" else (O, Kc, idx, n_sel)


# ---------------------------------------------------------------------------- necessary work
def _step_work(case, t, l_C):
    """(bytes, flops) of one sequence's step: every input row that matters read once, every output written once;
    one product per score (Eq. 6), the two products of the attention (Eq. 1), the two compressions (Eq. 5)."""
    H, HG, d, dc, k = case["H"], case["H_G"], case["d"], case["d_c"], case["k"]
    dH, dG = H * d, HG * d
    i_end = min(case["l_I"], t)
    l_M = max(i_end, t - case["l_L"]) - i_end
    n_att = i_end + min(k, l_M) + (t - i_end - l_M) + l_C
    scored = l_M if l_M > k else 0
    full = case["kind"] == "full"
    d_s = dH if full else dc
    byts = 4.0 * n_att * dG                                     # K and V rows attended
    byts += 2.0 * scored * (dG if full else dc)                 # keys scored
    byts += 4.0 * l_C * dH * (2 if case["kind"] == "two" else 1) + 8.0 * l_C * dG + 4.0 * min(k, l_M)
    flops = 4.0 * dH * l_C * (n_att - (l_C - 1) / 2.0) + 2.0 * d_s * l_C * scored
    if not full:
        flops += 2.0 * l_C * dc * (dG + (dH if scored else 0))
        byts += 2.0 * l_C * dc
    return byts, flops


def work(case):
    if case["kind"] == "fit":
        n, dc, dH, dG = case["l_C"], case["d_c"], case["H"] * case["d"], case["H_G"] * case["d"]
        params = dc * (dH + dG + 2)
        steps = -(-case["pairs"] // n)
        # the parameters and their two moments read and written each step, the pairs read once
        return {"bytes": steps * 24.0 * params + 2.0 * case["pairs"] * (dH + dG),
                "flops": case["pairs"] * (4.0 * dc * (dH + dG) + 2.0 * n * (dG + 3 * dc))}
    if case["kind"] == "prefill":
        parts = [_step_work(case, p, min(case["l_C"], case["t"] - p)) for p in range(0, case["t"], case["l_C"])]
    else:
        parts = [_step_work(case, t, case["l_C"]) for t in _positions(case)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    if case["kind"] == "fit":
        # fp32 sums in another order; Adam's first steps follow the sign of a gradient however small it is, so a
        # few weights with gradients near zero move by up to lr a step in another direction
        return {"rel": 1e-3, "max": 0.5}
    # bf16 products, probabilities and outputs.  Selected positions are decided on fp32 sums: two orders of summation
    # may swap a token at the k-th score, and the entries between the two shift in the ascending list
    return {"rel": 1e-2, "differ": 1e-2}
