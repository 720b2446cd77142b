"""Kernels of consecutive calls overlap at their ends (programmatic serialization).  Calls of every path issued one directly after
the other, each on inputs and outputs of its own but through one context and workspace, plain and captured, and calls
behind an event wait of the caller's, give bit for bit what calls with a synchronisation after each give."""
from dataclasses import fields, replace

import pytest
import torch

from paper_2410_03090_b200 import binding as ub
from paper_2410_03090_b200 import synth
from paper_2410_03090_b200.compress import CompressionPass, DecodeCache, PassOutput

pytestmark = pytest.mark.gpu


def _own_output(cp):
    return PassOutput(*(torch.zeros_like(getattr(cp.out, f.name)) for f in fields(PassOutput)))


class _Op:
    """A call and the tensors it writes, which `reset` puts back to what they were."""

    def __init__(self, call, tensors):
        self.call, self.tensors = call, tensors
        self.first = [t.clone() for t in tensors]

    def reset(self):
        for t, f in zip(self.tensors, self.first):
            t.copy_(f)

    def result(self):
        return [t.clone() for t in self.tensors]


def _pass_op(cp, wl, seed, how):
    K, V, Qw = synth.generate(replace(wl, seed=seed), "cuda")
    out = _own_output(cp)
    lse = torch.full((wl.B, wl.L, wl.Hq, wl.w), 9.0 + seed, device="cuda") if how == "lse" else None

    def call():
        cp.out = out
        if how == "staged":
            cp.run(K, V, Qw)
        elif how == "entropy":
            ub.uncomp_entropy(cp.ctx, K, wl.k_trunc, entropy=out.entropy, erank=out.erank, Qw=Qw if wl.dtype == "bf16" else None)
        else:
            cp.run_one_call(K, V, Qw, lse=lse)
    return _Op(call, [getattr(out, f.name) for f in fields(PassOutput)])


def _evict_op(cp, wl, seed):
    K, _, Qw = synth.generate(replace(wl, seed=seed), "cuda")
    D, n = 512, wl.N // 2
    X = torch.randn(wl.B, wl.N, D, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda").to(wl.torch_dtype)
    scores = torch.zeros(wl.B, wl.N - 1, device="cuda")
    indices = torch.zeros(wl.B, n, dtype=torch.int32, device="cuda")
    Xout = torch.zeros(wl.B, n, D, dtype=X.dtype, device="cuda")
    q, K0 = Qw[:, 0, :, -1].contiguous(), K[:, 0]
    return _Op(lambda: ub.uncomp_evict_hidden(cp.ctx, q, K0, X, n, scores=scores, indices=indices, Xout=Xout), [scores, indices, Xout])


def _decode_op(cp, wl, seed, steps=3):
    K, V, Qw = synth.generate(replace(wl, seed=seed), "cuda")
    cp.out = _own_output(cp)
    cp.run(K, V, Qw)
    cache = DecodeCache(cp)
    g = torch.Generator(device="cuda").manual_seed(seed)
    q = torch.randn(steps, wl.B, wl.L, wl.Hq, wl.d, generator=g, device="cuda").to(wl.torch_dtype)
    kv = torch.randn(2, steps, wl.B, wl.L, wl.H, wl.d, generator=g, device="cuda").to(wl.torch_dtype)
    pos = wl.N + torch.arange(steps, dtype=torch.int32, device="cuda")[:, None].repeat(1, wl.B)

    def call():
        for i in range(steps):
            cache.step(q[i], kv[0, i], kv[1, i], pos[i])
    return _Op(call, [cache.Kc, cache.Vc, cache.pos, cache.cum, cache.lens, cache.evicted])


def _wide_op(cp, scratch, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    N, D, k = 900, 512, 32
    X = (torch.randn(N, 60, generator=g, device="cuda") @ torch.randn(60, D, generator=g, device="cuda")
         + 0.1 * torch.randn(N, D, generator=g, device="cuda")).to(torch.bfloat16)[None]
    box = []

    def call():
        box[:] = ub.uncomp_entropy_wide(cp.ctx, X, k, scratch=scratch, spectrum=True)
    op = _Op(call, [])
    op.result = lambda: [t.clone() for t in box]
    return op


def _ops(path):
    name = "c1" if path == "fp32" else "c2"
    wl = synth.scaled(synth.WORKLOADS[name], N=520 if path == "fp32" else 700, L=1)
    if path == "many units":
        wl = synth.scaled(synth.WORKLOADS[name], N=260, L=40)
    cp = CompressionPass(wl, "cuda")
    scratch = torch.empty(ub.lib.uncomp_entropy_wide_scratch_bytes(900, 512), dtype=torch.uint8, device="cuda")
    make = {"staged": lambda s: _pass_op(cp, wl, s, "staged"), "one call": lambda s: _pass_op(cp, wl, s, "one call"),
            "lse": lambda s: _pass_op(cp, wl, s, "lse"), "entropy": lambda s: _pass_op(cp, wl, s, "entropy"),
            "evict": lambda s: _evict_op(cp, wl, s), "decode": lambda s: _decode_op(cp, wl, s),
            "wide": lambda s: _wide_op(cp, scratch, s)}
    if path in ("fp32", "many units", "mixed"):
        kinds = ["entropy", "staged", "entropy", "evict", "decode", "entropy", "decode", "one call", "lse", "entropy", "entropy", "evict"]
        if path == "mixed":
            kinds += ["wide", "staged", "wide", "entropy", "wide", "decode"]
    else:
        kinds = [path] * 4
    return cp, [make[kind](3 + i) for i, kind in enumerate(kinds)]


@pytest.mark.parametrize("path", ["staged", "one call", "lse", "entropy", "evict", "decode", "wide", "fp32", "many units", "mixed"])
def test_calls_directly_after_one_another(path):
    cp, ops = _ops(path)
    for op in ops:
        op.reset()
    want = []
    for op in ops:
        torch.cuda.synchronize()
        op.call()
        torch.cuda.synchronize()
        want.append(op.result())

    def check(how):
        torch.cuda.synchronize()
        assert cp.status() == 0
        for i, (op, w) in enumerate(zip(ops, want)):
            assert all(torch.equal(a, b) for a, b in zip(op.result(), w)), (how, i)

    for _ in range(3):
        for op in ops:
            op.reset()
        torch.cuda.synchronize()
        for op in ops:
            op.call()
        check("plain")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for op in ops:
            op.call()
    for _ in range(3):
        for op in ops:
            op.reset()
        graph.replay()
        check("captured")


@pytest.mark.parametrize("name,N,L", [("c1", 200, 1), ("c2", 700, 1), ("c2", 260, 40)])
@pytest.mark.parametrize("one_call", [False, True])
def test_rewritten_buffers(name, N, L, one_call):
    wl = replace(synth.scaled(synth.WORKLOADS[name], N=N, L=L), seed=3)
    inputs = [synth.generate(replace(wl, seed=s), "cuda") for s in (3, 4, 5)]
    K, V, Qw = (torch.empty_like(t) for t in inputs[0])
    cp = CompressionPass(wl, "cuda")
    run = cp.run_one_call if one_call else cp.run

    def outputs(o):
        return [t.clone() for t in (o.entropy, o.budgets, o.offsets, o.scores, o.indices, o.Kc, o.Vc)]

    def step(i, sync):
        for dst, src in zip((K, V, Qw), inputs[i]):
            dst.copy_(src)
        if sync:
            torch.cuda.synchronize()
        out = run(K, V, Qw)
        if sync:
            torch.cuda.synchronize()
        return outputs(out)

    want = [step(i, True) for i in range(3)]
    got = [step(i % 3, False) for i in range(9)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = run(K, V, Qw)
        run(K, V, Qw)
    for i in range(3):
        for dst, src in zip((K, V, Qw), inputs[i]):
            dst.copy_(src)
        graph.replay()
        got.append(outputs(out))
    torch.cuda.synchronize()
    assert cp.status() == 0
    for i, g in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(g, want[i % 3])), i


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("writer", ["copy", "kernel"])
@pytest.mark.parametrize("path", ["entropy", "staged", "one call", "evict", "wide"])
def test_behind_an_event_wait(path, writer, captured):
    """The keys (hidden states) come from another stream, late.  On the caller's stream a call of the library runs ahead of the
    wait, one whose last kernel lets the next begin early, and the call behind the wait must still see the new keys."""
    wl = synth.scaled(synth.WORKLOADS["c2"], N=700, L=1)
    cp = CompressionPass(wl, "cuda")
    old, new = (synth.generate(replace(wl, seed=s), "cuda") for s in (3, 4))
    src = [torch.cat([t.reshape(-1) for t in x]) for x in (old, new)]
    buf = src[0].clone()
    K, V, Qw = (p.view(t.shape) for p, t in zip(buf.split([t.numel() for t in old]), old))
    K0 = synth.generate(replace(wl, seed=5), "cuda")[0]
    ent0, er0 = (torch.zeros_like(cp.out.entropy) for _ in range(2))
    scratch = torch.empty(ub.lib.uncomp_entropy_wide_scratch_bytes(700, 1024), dtype=torch.uint8, device="cuda")
    outs = []

    def call():
        o = cp.out
        if path == "entropy":
            ub.uncomp_entropy(cp.ctx, K, 32, entropy=o.entropy, erank=o.erank, Qw=Qw)
            outs[:] = [o.entropy, o.erank]
        elif path == "evict":
            outs[:] = ub.uncomp_evict_hidden(cp.ctx, q, K[:, 0], K[:, 0].reshape(1, 700, 1024), 350, indices=idx, Xout=Xout)
        elif path == "wide":
            outs[:] = ub.uncomp_entropy_wide(cp.ctx, K[:, 0].reshape(1, 700, 1024), 32, scratch=scratch)
        else:
            (cp.run if path == "staged" else cp.run_one_call)(K, V, Qw)
            outs[:] = [o.entropy, o.budgets, o.scores, o.indices, o.Kc, o.Vc]

    q = Qw[:, 0, :, -1].contiguous()
    idx = torch.zeros(1, 350, dtype=torch.int32, device="cuda")
    Xout = torch.zeros(1, 350, 1024, dtype=torch.bfloat16, device="cuda")

    def both(stream, other):
        other.wait_stream(stream)
        with torch.cuda.stream(other):
            torch.cuda._sleep(2_000_000)
            buf.copy_(src[1]) if writer == "copy" else torch.mul(src[1], 1, out=buf)
            event = other.record_event()
        with torch.cuda.stream(stream):
            ub.uncomp_entropy(cp.ctx, K0, 32, entropy=ent0, erank=er0)
            stream.wait_event(event)
            call()

    buf.copy_(src[1])
    torch.cuda.synchronize()
    call()
    torch.cuda.synchronize()
    want = [t.clone() for t in outs]
    graph = None
    if captured:
        graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph):
            both(torch.cuda.current_stream(), other)
    streams = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(4):
        buf.copy_(src[0])
        for t in outs:
            t.zero_()
        torch.cuda.synchronize()
        if captured:
            graph.replay()
        else:
            both(*streams)
        torch.cuda.synchronize()
        assert cp.status() == 0
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
