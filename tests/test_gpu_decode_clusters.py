"""The one-launch decode step at the cache sizes where its cluster grows, where a CTA's share is ragged or empty, and
where the logits no longer fit into shared memory (the three-launch form), against the oracle."""
import numpy as np
import pytest

import test_gpu_decode as td

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("caps,G,dtype,full", [
    ([1, 2, 3], 4, "bf16", True),                       # fewer entries than CTAs of the cluster would have
    ([255, 256, 257], 2, "bf16", True),
    ([1023, 511, 8], 8, "bf16", True),                  # 1024 entries with the new token
    ([1024, 1000], 4, "fp32", True),                    # one more: a cluster of two
    ([8200, 4100, 9], 1, "bf16", False),                # cluster of eight, appending
    ([26000, 100], 16, "bf16", True),                   # beyond shared memory
])
def test_cluster_steps(caps, G, dtype, full):
    from paper_2410_03090_b200 import binding as ub
    units = len(caps)
    caps = np.array(caps)
    lens = caps.copy() if full else np.maximum(0, caps - 2)
    ctx = ub.Context(ub.make_shape(1, 1, units, units * G, 131072, 128, 32, dtype))
    st = td.State(1, 1, units, units * G, dtype, caps, lens, seed=5, start_pos=30000)
    for _ in range(3):
        td._step_and_check(ub, ctx, st, int(caps.max()), protect=1)
    assert ub.uncomp_status(ctx) == 0


@pytest.mark.parametrize("units", [147, 296, 297, 600])
def test_cluster_choice_by_units(units):
    from paper_2410_03090_b200 import binding as ub
    rng = np.random.default_rng(units)
    caps = rng.integers(1, 700, size=units)
    caps[0] = 700
    ctx = ub.Context(ub.make_shape(1, 1, units, units * 4, 16384, 128, 32, "bf16"))
    st = td.State(1, 1, units, units * 4, "bf16", caps, caps.copy(), seed=6, start_pos=5000)
    td._step_and_check(ub, ctx, st, 700, protect=3)
    assert ub.uncomp_status(ctx) == 0
