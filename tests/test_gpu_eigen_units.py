"""Eigenvalues over the numbers of units at which the split of a unit over CTAs changes, against fp64 on the CPU."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("units", [1, 18, 19, 37, 38, 74, 75])
def test_spectrum_over_unit_counts(units, dtype):
    from paper_2410_03090_b200 import binding as ub

    N = 160
    torch.manual_seed(units)
    K = torch.randn(1, units, 1, N, 128, device="cuda") * torch.logspace(0, -2, 128, device="cuda")
    K = K.to(torch.float32 if dtype == "fp32" else torch.bfloat16)
    X = K[0, :, 0].double().cpu()
    X = X - X.mean(1, keepdim=True)
    want = torch.linalg.eigvalsh(X.transpose(1, 2) @ X).flip(1).clamp(min=0)
    ctx = ub.Context(ub.make_shape(1, units, 1, 1, N, 128, 32, dtype))
    for k in (1, 33, 128):
        spectrum = torch.empty(1, units, 1, k, dtype=torch.float64, device="cuda")
        ent, erank = ub.uncomp_entropy(ctx, K, k, spectrum=spectrum)
        assert ub.uncomp_status(ctx) == 0
        lam = spectrum[0, :, 0].cpu()
        # brackets of 1e-13 (fp32 keys) and 2e-8 of the Gershgorin radius, at most three times the largest eigenvalue of a
        # tridiagonal matrix; the reductions: 128 steps of 2^-53 and, with the fp32 partials, of 2^-24
        bound = 3e-13 + 128 * 2.0 ** -53 if dtype == "fp32" else 6e-8 + 128 * 2.0 ** -24
        assert float(((lam - want[:, :k]).abs() / want[:, :1]).max()) < bound
        p = want[:, :k] / want[:, :k].sum(1, keepdim=True)
        H = -(p * p.clamp(min=1e-300).log()).sum(1)
        assert float((ent[0, :, 0].double().cpu() - H).abs().max()) < 1e-4
        assert torch.allclose(erank, ent.exp(), rtol=1e-5)


@pytest.mark.parametrize("dtype,units", [("fp32", 8), ("fp32", 80), ("bf16", 8), ("bf16", 80), ("bf16", 300)])
@pytest.mark.parametrize("max_iters", [1 << 30, 2**31 - 1])
def test_any_number_of_rounds(dtype, units, max_iters):
    """As many rounds as fit the parameter: what the default gives, bit for bit."""
    from paper_2410_03090_b200 import binding as ub

    g = torch.Generator(device="cuda").manual_seed(units)
    K = torch.randn(1, units, 1, 150, 128, generator=g, device="cuda").to(torch.float32 if dtype == "fp32" else torch.bfloat16)
    ctx = ub.Context(ub.make_shape(1, units, 1, 1, 150, 128, 32, dtype))
    spectra = [torch.empty(1, units, 1, 32, dtype=torch.float64, device="cuda") for _ in range(2)]
    want = ub.uncomp_entropy(ctx, K, 32, spectrum=spectra[0])
    got = ub.uncomp_entropy(ctx, K, 32, max_iters=max_iters, spectrum=spectra[1])
    assert ub.uncomp_status(ctx) == 0
    assert torch.equal(spectra[0], spectra[1]) and all(torch.equal(a, b) for a, b in zip(want, got))


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("units", [4, 18, 37, 60, 74, 75, 300])
def test_keys_without_any_spread(units, dtype):
    """All zero, or the same row for every token: no eigenvalue, entropy 0 and effective rank 1, beside units like any other."""
    from paper_2410_03090_b200 import binding as ub

    N = 200
    g = torch.Generator(device="cuda").manual_seed(units)
    K = torch.randn(1, units, 1, N, 128, generator=g, device="cuda")
    K[0, 1] = 0
    K[0, 2] = torch.randint(-8, 9, (128,), generator=g, device="cuda").float()
    K[0, units - 1] = 3.0
    K = K.to(torch.float32 if dtype == "fp32" else torch.bfloat16)
    Qw = torch.randn(1, units, 1, 32, 128, generator=g, device="cuda").to(K.dtype)
    ctx = ub.Context(ub.make_shape(1, units, 1, 1, N, 128, 32, dtype))
    for k in (1, 32, 128):
        for center in (0, 1):
            for norm in (0, 1):
                for q in (None, Qw) if dtype == "bf16" else (None,):
                    ent, erank = ub.uncomp_entropy(ctx, K, k, center, norm, Qw=q)
                    assert ub.uncomp_status(ctx) == 0
                    for u in (1, 2, units - 1):        # without centring a constant row is one direction: entropy 0 as well
                        assert abs(float(ent[0, u, 0])) < 1e-4 and abs(float(erank[0, u, 0]) - 1) < 1e-4, (u, k, center, norm)
                    assert k == 1 or float(ent[0, 0, 0]) > 1
