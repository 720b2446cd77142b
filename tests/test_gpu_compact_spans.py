"""Gather of the kept rows where the rows per warp and the search over the units change, against plain indexing."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("units,keep", [(1, 32), (1, 257), (31, 33), (33, 300), (1056, 40), (1056, 301)])
def test_rows_of_uneven_units(units, keep, dtype):
    from paper_2410_03090_b200 import binding as ub

    N, t = 320, torch.float32 if dtype == "fp32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(units + keep)
    K, V = (torch.randn(1, units, 1, N, 128, generator=gen, device="cuda").to(t) for _ in range(2))
    budgets = torch.randint(32, keep + 1, (units,), generator=gen, device="cuda")     # up to 9472 rows and more: one or several steps
    offsets = torch.zeros(units + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = budgets.cumsum(0)
    total = int(offsets[-1])
    indices = torch.randint(0, N, (total,), generator=gen, device="cuda").to(torch.int32)
    unit = torch.repeat_interleave(torch.arange(units, device="cuda"), budgets)
    ctx = ub.Context(ub.make_shape(1, units, 1, 1, N, 128, 32, dtype))
    Kc, Vc = ub.uncomp_compact(ctx, K, V, indices, offsets, total)
    assert ub.uncomp_status(ctx) == 0
    assert torch.equal(Kc, K[0, unit, 0, indices.long()]) and torch.equal(Vc, V[0, unit, 0, indices.long()])
