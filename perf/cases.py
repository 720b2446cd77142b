"""Performance cases: the calls a program around a long-context model makes into this package.

`listed()` names the cases that are timed by default, `draw(rng)` gives further ones of the same ranges.  `prepare`
makes what the program already holds when it calls (keys, values, window queries, the pass or cache object with its
workspace), `run` is one call through the public entry points, `work` the bytes and operations it cannot do without.

Paths:
  pass    the compression pass at the end of prefill (`CompressionPass`): entropy -> budgets -> scores and selection ->
          ragged cache.  entry "staged" is `run`, "one_call" is `run_one_call`, "one_call_lse" the same with the
          prefill attention kernel's log-sum-exp handed in.
  evict   hidden-state eviction between two layer groups (`uncomp_evict_hidden`)
  decode  one decode step on the compressed cache (`DecodeCache.step`)
  wide    truncated entropy of hidden-state matrices (`uncomp_entropy_wide`)
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

from paper_2410_03090_b200 import binding as ub
from paper_2410_03090_b200 import synth
from paper_2410_03090_b200.compress import CompressionPass, DecodeCache, PassOutput

MAX_UNIT_TOKENS = 4 * 32 * 8 * 32768       # largest listed key cache: units x tokens of the batch-4 prefill
MAX_ROW_TOKENS = 512 * 16 * 8 * 131072     # largest listed scorer: window rows x units x tokens
MAX_CACHE_ROWS = 4 * 32 * 8 * 3080         # largest listed decode cache
MAX_HIDDEN = 4 * 32768 * 4096              # largest listed hidden-state tensor (elements)
MAX_WIDE = 4096                            # widest matrix of the wide entropy


def _pass(name, entry, B, L, H, Hq, N, w, avg_budget, dtype="bf16", like="c2", **more):
    return dict(name=name, path="pass", entry=entry, B=B, L=L, H=H, Hq=Hq, N=N, w=w, avg_budget=avg_budget,
                dtype=dtype, like=like, **more)


def listed():
    return [
        # the smallest call: one layer, a short prompt, fp32 caches (accuracy studies keep them in fp32)
        _pass("pass_fp32_512", "staged", 1, 1, 8, 8, 512, 32, 128, "fp32", "c1"),
        # one layer at a time while the prefill goes on, prompt of odd length
        _pass("pass_one_layer_7001", "one_call", 1, 1, 8, 32, 7001, 32, 384),
        # the method's own setting: Llama-2-7B heads (no grouping), 3712-token prompt, window 8, 384 tokens a head
        _pass("pass_llama2_3712", "staged", 1, 32, 32, 32, 3712, 8, 384),
        # Llama-3-8B shape, 8K-token prompt
        _pass("pass_llama3_8k", "staged", 1, 32, 8, 32, 8192, 32, 410),
        # Llama-3-8B shape, 32K tokens: the benchmarked workload
        _pass("pass_llama3_32k", "staged", 1, 32, 8, 32, 32768, 64, 1540, like="c3"),
        # the same behind an attention kernel that hands over its log-sum-exp
        _pass("pass_llama3_32k_lse", "one_call_lse", 1, 32, 8, 32, 32768, 64, 1540, like="c3"),
        # Mistral-7B shape, four sequences of 32K tokens, heavy-hitter positions
        _pass("pass_mistral_4x32k", "one_call", 4, 32, 8, 32, 32768, 32, 3080, like="c4"),
        # Llama-3-70B shape, 128K tokens, 16 of its 80 layers (one of five pipeline stages)
        _pass("pass_llama70b_128k", "staged", 1, 16, 8, 64, 131072, 64, 2621, like="c5"),
        # hidden states of a batch cut to half at a layer-group boundary
        dict(name="evict_4x32k", path="evict", B=4, H=8, Hq=32, N=32768, D=4096, n_keep=16384),
        # one decode step after an 8K-token prefill of one sequence: a latency-critical call per generated token
        dict(name="decode_llama3_8k", path="decode", B=1, L=32, H=8, Hq=32, N=8192, w=32, avg_budget=410),
        # one decode step of a batch with large caches
        dict(name="decode_mistral_4x32k", path="decode", B=4, L=32, H=8, Hq=32, N=32768, w=32, avg_budget=3080),
        # entropy of one layer's hidden states
        dict(name="wide_8192x4096", path="wide", count=1, N=8192, D=4096, k=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["pass"] * 6 + ["evict", "decode", "decode", "wide"])
    H, Hq = rng.choice([(8, 32), (8, 32), (8, 64), (32, 32)])
    if path == "pass":
        if rng.random() < 0.15:            # fp32 caches: short prompts of one or a few layers
            N, L, w = _log_int(rng, 200, 2048), rng.randint(1, 4), rng.choice([8, 16, 32])
            return dict(path="pass", entry=rng.choice(["staged", "one_call"]), B=1, L=L, H=8, Hq=rng.choice([8, 32]),
                        N=N, w=w, avg_budget=max(w + 8, int(N * rng.uniform(0.1, 0.25))), dtype="fp32", like="c1")
        N = _log_int(rng, 1000, 131072)
        w = rng.choice([8, 16, 32, 64])
        rows = Hq // H * w
        most = min(MAX_UNIT_TOKENS // (N * H), MAX_ROW_TOKENS // (rows * N * H), 128)
        L = _log_int(rng, 1, min(32, most))
        B = rng.randint(1, max(1, min(4, most // L)))
        avg = max(w + 16, int(N * rng.uniform(0.02, 0.12)))
        return dict(path="pass", entry=rng.choice(["staged", "staged", "one_call", "one_call_lse"]), B=B, L=L, H=H, Hq=Hq,
                    N=N, w=w, avg_budget=avg, dtype="bf16", like=rng.choice(["c2", "c3", "c4", "c5"]))
    if path == "evict":
        B, D = rng.randint(1, 4), rng.choice([2048, 3072, 4096, 8192])
        N = _log_int(rng, 2000, min(131072, MAX_HIDDEN // (B * D)))
        return dict(path="evict", B=B, H=H, Hq=Hq, N=N, D=D, n_keep=int(N * rng.uniform(0.3, 0.9)))
    if path == "decode":
        B = rng.randint(1, 4)
        avg = _log_int(rng, 200, min(4096, MAX_CACHE_ROWS // (B * 32 * H)))
        return dict(path="decode", B=B, L=32, H=H, Hq=Hq, N=avg * rng.randint(8, 20), w=32, avg_budget=avg)
    D = 64 * rng.randint(16, MAX_WIDE // 64)
    return dict(path="wide", count=1, N=_log_int(rng, 500, 16384), D=D, k=rng.choice([16, 32, 64]))


def _workload(case, seed):
    """The value recipe of the named workload at this case's shape."""
    base = synth.WORKLOADS[case["like"]]
    avg = case["avg_budget"]
    n_max = min(case["N"], int(round(5.0 * avg / 3.0)), 2 * avg - case["w"])
    return replace(base, name="case", B=case["B"], L=case["L"], H=case["H"], Hq=case["Hq"], N=case["N"], w=case["w"],
                   dtype=case["dtype"], avg_budget=avg, n_max=n_max, seed=int(seed))


def _prefill_lse(wl, K, Qw):
    """[B, L, Hq, w]: natural-log sum of exponentials of every window row's scaled, causally visible logits."""
    out = torch.empty(wl.B, wl.L, wl.Hq, wl.w, device=K.device)
    last = (wl.N - wl.w + torch.arange(wl.w, device=K.device)).repeat(wl.G)
    hidden = torch.arange(wl.N, device=K.device)[None, :] > last[:, None]
    for b in range(wl.B):
        for l in range(wl.L):
            for h in range(wl.H):
                q = Qw[b, l, h * wl.G:(h + 1) * wl.G].reshape(wl.G * wl.w, wl.d).float()
                s = torch.matmul(q, K[b, l, h].float().t()).mul_(wl.d ** -0.5).masked_fill_(hidden, float("-inf"))
                out[b, l, h * wl.G:(h + 1) * wl.G] = torch.logsumexp(s, dim=-1).view(wl.G, wl.w)
    return out


def _words(t):
    """Rows that are copied bit for bit, as whole numbers."""
    return t.view(torch.int16 if t.element_size() == 2 else torch.int32)


def _prepare_pass(case, seed):
    wl = _workload(case, seed)
    K, V, Qw = synth.generate(wl, "cuda")
    lse = _prefill_lse(wl, K, Qw) if case["entry"] == "one_call_lse" else None
    return dict(path="pass", entry=case["entry"], cp=CompressionPass(wl, "cuda"), K=K, V=V, Qw=Qw, lse=lse)


def _prepare_evict(case, seed):
    wl = replace(synth.WORKLOADS["c3"], name="case", B=case["B"], L=1, H=case["H"], Hq=case["Hq"], N=case["N"], w=1,
                 seed=int(seed))
    K, _, Qw = synth.generate(wl, "cuda")
    X = synth.hidden_states(wl, case["D"], "cuda")
    n = case["n_keep"]
    return dict(path="evict", ctx=ub.Context(ub.make_shape(wl.B, 1, wl.H, wl.Hq, wl.N, wl.d, 1, wl.dtype)), n_keep=n,
                K=K[:, 0], q=Qw[:, 0, :, -1, :].contiguous(), X=X,
                scores=torch.empty(wl.B, wl.N - 1, device="cuda"),
                indices=torch.empty(wl.B, n, dtype=torch.int32, device="cuda"),
                Xout=torch.empty(wl.B, n, case["D"], dtype=X.dtype, device="cuda"))


def _prepare_decode(case, seed):
    """The cache as a prefill pass leaves it: ragged budgets (half of a layer's heads above the average, half below),
    ascending kept positions, skewed window scores, keys with a few dominant directions per head."""
    wl = _workload(dict(case, dtype="bf16", like="c2"), seed)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kw = dict(generator=g, device="cuda")
    units, H, avg, d = wl.units, wl.H, wl.avg_budget, wl.d
    step = 2.0 * (wl.n_max - avg) / (H - 1)
    ladder = torch.tensor([int(wl.n_max - i * step) for i in range(H)], device="cuda")
    short = H * avg - int(ladder.sum())
    ladder[:short] += 1
    order = torch.rand(wl.B * wl.L, H, **kw).argsort(dim=1)
    budgets = ladder[order].reshape(-1)
    offsets = torch.zeros(units + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = budgets.cumsum(0)
    P, cap = wl.N - wl.w, int(budgets.max())
    indices = torch.empty(units * avg, dtype=torch.int32, device="cuda")
    Kc = torch.empty(units * avg, d, dtype=torch.bfloat16, device="cuda")
    Vc = torch.randn(units * avg, d, **kw).to(torch.bfloat16)
    qnew = torch.empty(units, wl.G, d, dtype=torch.bfloat16, device="cuda")
    knew = torch.empty(units, d, dtype=torch.bfloat16, device="cuda")
    r, per = 16, 64
    window = torch.arange(P, wl.N, device="cuda")
    slot = torch.arange(cap, device="cuda")
    for u0 in range(0, units, per):
        n = min(per, units - u0)
        b = budgets[u0:u0 + n]
        W = torch.randn(n, r, d, **kw) * (2.0 / r ** 0.5)

        def rows(m):
            return (torch.randn(n, m, r, **kw) @ W + torch.randn(n, m, d, **kw)).to(torch.bfloat16)

        keep = slot[None, :] < b[:, None]
        at = slice(int(offsets[u0]), int(offsets[u0 + n]))
        Kc[at] = rows(cap)[keep]
        # positions of the kept tokens: the lowest budget - w of a random order, ascending, then the window
        prefix = (torch.rand(n, P, **kw).argsort(dim=1)[:, :cap]).masked_fill_(slot[None, :] >= b[:, None] - wl.w, wl.N + 1)
        pos = prefix.sort(dim=1).values
        tail = (slot[None, :] - (b[:, None] - wl.w)).clamp_(0, wl.w - 1)
        indices[at] = torch.where(pos <= wl.N, pos, window[tail])[keep].to(torch.int32)
        qnew[u0:u0 + n] = rows(wl.G)
        knew[u0:u0 + n] = rows(1)[:, 0]
    scores = torch.exp(1.5 * torch.randn(wl.B, wl.L, H, P, **kw)) * (wl.G * wl.w / P)
    out = PassOutput(None, None, budgets.to(torch.int32).view(wl.B, wl.L, H), offsets, None, None, scores, indices, Kc, Vc)
    cp = CompressionPass(wl, "cuda")
    cache = DecodeCache(cp, out)
    new_pos = (wl.N + torch.arange(4096, dtype=torch.int32, device="cuda"))[:, None].repeat(1, wl.B)
    return dict(path="decode", cache=cache, step=0, new_pos=list(new_pos.unbind(0)),
                q=qnew.view(wl.B, wl.L, wl.Hq, d), k=knew.view(wl.B, wl.L, H, d),
                v=torch.randn(wl.B, wl.L, H, d, **kw).to(torch.bfloat16))


def _prepare_wide(case, seed):
    """Hidden states: a few hundred strong directions with a decaying spectrum, isotropic noise, a mean."""
    count, N, D, r = case["count"], case["N"], case["D"], 256
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    W = torch.randn(r, D, generator=g, device="cuda") * (torch.arange(1, r + 1, device="cuda") ** -0.7)[:, None]
    X = torch.empty(count, N, D, dtype=torch.bfloat16, device="cuda")
    for i in range(count):
        X[i] = (torch.randn(N, r, generator=g, device="cuda") @ W
                + 0.05 * torch.randn(N, D, generator=g, device="cuda") + 0.3).to(torch.bfloat16)
    scratch = torch.empty(ub.lib.uncomp_entropy_wide_scratch_bytes(N, D), dtype=torch.uint8, device="cuda")
    return dict(path="wide", ctx=ub.Context(ub.make_shape(1, 1, 1, 1, 256, 128, 8, "bf16")), X=X, k=case["k"],
                scratch=scratch)


def prepare(case, seed):
    return {"pass": _prepare_pass, "evict": _prepare_evict, "decode": _prepare_decode,
            "wide": _prepare_wide}[case["path"]](case, seed)


def run(state):
    path = state["path"]
    if path == "pass":
        cp = state["cp"]
        if state["entry"] == "staged":
            o = cp.run(state["K"], state["V"], state["Qw"])
        else:
            o = cp.run_one_call(state["K"], state["V"], state["Qw"], lse=state["lse"])
        return dict(entropy=o.entropy, erank=o.erank, budgets=o.budgets, offsets=o.offsets, layer_group=o.layer_group,
                    layer_ctx=o.layer_ctx, scores=o.scores, indices=o.indices, Kc=_words(o.Kc), Vc=_words(o.Vc))
    if path == "evict":
        ub.uncomp_evict_hidden(state["ctx"], state["q"], state["K"], state["X"], state["n_keep"], scores=state["scores"],
                               indices=state["indices"], Xout=state["Xout"])
        return dict(scores=state["scores"], indices=state["indices"], Xout=_words(state["Xout"]))
    if path == "decode":
        c = state["cache"]
        pos = state["new_pos"][state["step"] % 4096]
        state["step"] += 1
        evicted = c.step(state["q"], state["k"], state["v"], pos)
        return dict(evicted=evicted, lens=c.lens, pos=c.pos, cum=c.cum, Kc=_words(c.Kc), Vc=_words(c.Vc))
    ent, er, spec = ub.uncomp_entropy_wide(state["ctx"], state["X"], state["k"], scratch=state["scratch"], spectrum=True)
    return dict(entropy=ent, erank=er, spectrum=spec)


def work(case):
    """One pass's indispensable bytes (inputs once, outputs once) and operations (the symmetric half of a Gram matrix,
    one product of window rows and keys)."""
    d = 128
    if case["path"] == "pass":
        s = 4 if case["dtype"] == "fp32" else 2
        units, rows, N, b = case["B"] * case["L"] * case["H"], case["Hq"] // case["H"] * case["w"], case["N"], case["avg_budget"]
        per = N * d * s + rows * d * s + b * d * s + 2 * b * d * s + 4 * (N - case["w"]) + 4 * b + 24
        if case["entry"] == "one_call_lse":
            per += 4 * rows
        return dict(bytes=units * per, flops=units * (N * d * (d + 1) + 2 * rows * d * N))
    if case["path"] == "evict":
        B, N = case["B"], case["N"]
        return dict(bytes=B * (case["H"] * N * d * 2 + case["Hq"] * d * 2 + 2 * case["n_keep"] * case["D"] * 2 + 4 * (N - 1)
                               + 4 * case["n_keep"]), flops=2 * B * case["Hq"] * N * d)
    if case["path"] == "decode":
        units, G = case["B"] * case["L"] * case["H"], case["Hq"] // case["H"]
        rows = units * case["avg_budget"]
        return dict(bytes=rows * (2 * d + 12) + units * (2 * d * (G + 4) + 16), flops=2 * rows * G * d)
    c, N, D = case["count"], case["N"], case["D"]
    return dict(bytes=c * (2 * N * D + 8 * case["k"] + 8), flops=c * N * D * (min(N, D) + 1))


def tolerance(case):
    """fp32 accumulation and exponentials of logits that reach some tens; copied rows, positions and budgets are whole
    numbers, of which a tie between two scores may move a few."""
    if case["path"] == "wide":
        return {"rel": 1e-5}               # eigenvalues of a matrix reduced in fp32
    return {"rel": 3e-5, "differ": 0.01}
