"""Kernels of consecutive calls overlap at their ends (programmatic serialization): calls issued back to back on buffers that
are rewritten in between, and the same calls captured and replayed, give bit for bit what calls with a synchronisation
after each give."""
from dataclasses import replace

import pytest
import torch

from paper_2410_03090_b200 import synth
from paper_2410_03090_b200.compress import CompressionPass

pytestmark = pytest.mark.gpu


def _outputs(o):
    return [t.clone() for t in (o.entropy, o.budgets, o.offsets, o.scores, o.indices, o.Kc, o.Vc)]


@pytest.mark.parametrize("name,N,L", [("c1", 200, 1), ("c2", 700, 1), ("c2", 260, 40)])
@pytest.mark.parametrize("one_call", [False, True])
def test_rewritten_buffers(name, N, L, one_call):
    wl = replace(synth.scaled(synth.WORKLOADS[name], N=N, L=L), seed=3)
    inputs = [synth.generate(replace(wl, seed=s), "cuda") for s in (3, 4, 5)]
    K, V, Qw = (torch.empty_like(t) for t in inputs[0])
    cp = CompressionPass(wl, "cuda")
    run = cp.run_one_call if one_call else cp.run

    def step(i, sync):
        for dst, src in zip((K, V, Qw), inputs[i]):
            dst.copy_(src)
        if sync:
            torch.cuda.synchronize()
        out = run(K, V, Qw)
        if sync:
            torch.cuda.synchronize()
        return _outputs(out)

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
        got.append(_outputs(out))
    torch.cuda.synchronize()
    assert cp.status() == 0
    for i, g in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(g, want[i % 3])), i
