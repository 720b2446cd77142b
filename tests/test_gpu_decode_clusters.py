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


@pytest.mark.parametrize("G,dtype", [(1, "bf16"), (2, "bf16"), (4, "bf16"), (8, "bf16"), (16, "bf16"), (1, "fp32"), (16, "fp32")])
@pytest.mark.parametrize("full", [True, False])
def test_three_launches_beyond_shared_memory(G, dtype, full):
    """Eight CTAs hold 200 KB of logits each: 51200 / G entries, less the padding.  The three launches beyond that, evicting
    and appending, beside a unit of one chunk and one of a single row."""
    from paper_2410_03090_b200 import binding as ub
    cap = 8 * 51200 // G + 8
    caps = np.array([1, cap, 1023])
    lens = caps.copy() if full else np.maximum(0, caps - 2)
    N = max(cap + 64, 150000)
    ctx = ub.Context(ub.make_shape(1, 1, 3, 3 * G, N, 128, 32, dtype))
    st = td.State(1, 1, 3, 3 * G, dtype, caps, lens, seed=G, start_pos=cap + 500)
    ub.uncomp_profile_enable(ctx, True)
    td._step_and_check(ub, ctx, st, cap, protect=1)
    launches = {name: n for name, (_, n) in ub.uncomp_profile_read(ctx).items() if n}
    assert launches == {"decode_logits": 1, "decode_accumulate": 1, "decode_commit": 1}


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
