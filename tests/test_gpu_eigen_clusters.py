"""Entropy of bf16 keys at the unit counts where the assembly of the covariance changes its cluster size, and at the
edges of the truncation, against the oracle."""
from dataclasses import replace

import pytest
import torch

import parity
from paper_2410_03090_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,H,N,k_trunc", [
    (1, 1, 4097, 32),      # clusters of 8
    (1, 37, 1100, 33),     # the last count of clusters of 4; more eigenvalues than one sweep of teams
    (2, 19, 1100, 1),      # 38 units: clusters of 2
    (1, 75, 2100, 128),    # clusters of one, all eigenvalues
    (2, 74, 600, 32),      # 148 units, one and two partials
    (3, 50, 2, 32),        # two tokens: rank one after centring
    (8, 37, 600, 32),      # 296 units: the last count of one kernel
    (9, 33, 700, 32),      # 297 units: a second kernel for the last 64 steps, three of four warps in its last CTA idle
    (10, 32, 300, 100),    # more eigenvalues than lanes there
])
def test_cluster_sizes(L, H, N, k_trunc):
    from paper_2410_03090_b200 import binding as ub
    wl = replace(synth.WORKLOADS["c2"], L=L, H=H, Hq=H, N=N, w=1, k_trunc=k_trunc, seed=77)
    K, _, _ = synth.generate(wl, "cuda")
    ctx = ub.Context(ub.make_shape(1, L, H, H, N, 128, 1, "bf16"))
    for center, norm in ((1, 0), (0, 1)):
        ent, er = ub.uncomp_entropy(ctx, K, k_trunc, center, norm)
        torch.cuda.synchronize()
        assert ub.uncomp_status(ctx) == 0
        units = sorted({0, wl.units // 3, wl.units - 1})
        parity.check_entropy(wl, K, ent, er, units, k_trunc=k_trunc, center=center, norm=norm)
