"""Selection at the prefix lengths where a CTA's share, the cluster and the kernel change, with ties, extreme budgets and
pool windows, against the oracle's selection of the pooled scores; budgets with more groups and units than fit a block."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
import parity
from paper_2410_03090_b200 import synth

pytestmark = pytest.mark.gpu


def _select(ub, P, H, budget, pool_kernel=1, pool_mode=0, ties=False, seed=0):
    w = 1
    wl = replace(synth.WORKLOADS["c2"], L=1, H=H, Hq=H, N=P + w, w=w, avg_budget=budget, M=1, n_max=budget, seed=seed)
    K, _, Qw = synth.generate(wl, "cuda")
    if ties:
        Qw.zero_()                                       # equal scores everywhere ...
        Qw[0, 0, 0, 0, 0] = 1.0
        K[0, 0, 0] = 0
        K[0, 0, 0, ::7, 0] = 2.0                         # ... and two levels in head 0
    ctx = ub.Context(ub.make_shape(1, 1, H, H, wl.N, 128, w, "bf16"))
    bud = torch.full((1, 1, H), budget, dtype=torch.int32, device="cuda")
    off = torch.arange(H + 1, device="cuda") * budget
    scores = torch.empty(1, 1, H, P, device="cuda")
    idx = ub.uncomp_score_select(ctx, Qw, K, bud, off, H * budget, pool_kernel, pool_mode, 0.0, scores)
    torch.cuda.synchronize()
    assert ub.uncomp_status(ctx) == 0
    parity.check_select(wl, scores, bud, off, idx, range(H))
    raw = torch.empty_like(scores)
    ub.uncomp_score_select(ctx, Qw, K, bud, off, H * budget, 1, 0, 0.0, raw)
    for u in range(min(H, 2)):
        ref = oracle.pool(raw[0, 0, u].double().cpu().numpy(), pool_kernel, pool_mode)
        np.testing.assert_allclose(scores[0, 0, u].cpu().numpy(), ref, rtol=1e-5)


@pytest.mark.parametrize("P", [1, 2, 127, 129, 2047, 2048, 2049, 4097, 8192, 8193, 16385, 32769, 65536, 65537, 131072, 131073])
def test_prefix_lengths(P):
    from paper_2410_03090_b200 import binding as ub
    _select(ub, P, 3, max(2, P // 9), seed=P)


@pytest.mark.parametrize("P,budget,pk,pm", [(5000, 2, 7, 0), (5000, 5001, 7, 0), (5000, 5000, 63, 0), (9001, 700, 7, 1),
                                            (20000, 19990, 7, 0), (4095, 64, 5, 0), (8190, 4000, 63, 1)])
def test_budgets_and_pools(P, budget, pk, pm):
    from paper_2410_03090_b200 import binding as ub
    _select(ub, P, 5, budget, pk, pm, seed=P + budget)


@pytest.mark.parametrize("P,budget", [(6000, 1000), (6000, 900), (30000, 4444), (140000, 2000)])
def test_ties(P, budget):
    from paper_2410_03090_b200 import binding as ub
    _select(ub, P, 2, budget, 1, 0, ties=True)


@pytest.mark.parametrize("P,budget,pk,pm,ties", [
    (262144, 3000, 7, 0, False),       # the longest prefix whose keys fit the shared memory of a cluster
    (262145, 3000, 7, 0, False),       # one more: radix select over global memory
    (262147, 2, 1, 0, False),          # one position
    (263000, 262999, 7, 0, False),     # all but two
    (263000, 263001, 63, 0, False),    # all
    (270001, 20000, 63, 1, False),     # mean pool
    (270001, 40000, 1, 0, True),       # the threshold among equal scores
    (270001, 9000, 7, 0, True),
])
def test_beyond_the_keys_in_shared_memory(P, budget, pk, pm, ties):
    from paper_2410_03090_b200 import binding as ub
    _select(ub, P, 2, budget, pk, pm, ties=ties, seed=P + budget)


@pytest.mark.parametrize("L,H,M,scope", [(1, 7, 3, 0), (80, 64, 5000, 1), (80, 64, 100, 1), (33, 32, 32, 0), (3, 8, 1, 1)])
def test_budget_tables(L, H, M, scope):
    from paper_2410_03090_b200 import binding as ub
    n = L * H if scope else H
    ctx = ub.Context(ub.make_shape(1, L, H, H, 4000, 128, 4, "bf16"))
    g = torch.Generator(device="cuda").manual_seed(L * H)
    er = (torch.randint(0, 50, (1, L, H), generator=g, device="cuda") + 1).float()       # many equal values
    avg, n_max = 101, 151
    bud, off, _, _ = ub.uncomp_assign_budgets(ctx, er, avg, M, n_max, scope)
    torch.cuda.synchronize()
    wl = replace(synth.WORKLOADS["c2"], L=L, H=H, Hq=H, N=4000, w=4, avg_budget=avg, M=M, n_max=n_max)
    parity.check_budgets(wl, er, bud, off, scope=scope)
    assert int(off[-1]) == L * H * avg
