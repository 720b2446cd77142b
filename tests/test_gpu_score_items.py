"""The persistent scorer where its variants and its work split change: numbers of window rows around 32, 64, 128 and 512,
several (unit, chunk) items per CTA with units changing inside a CTA, ragged last tiles; scores, entropies and the
log-sum-exp form against the oracle."""
from dataclasses import replace

import pytest
import torch

import parity
from paper_2410_03090_b200 import synth

pytestmark = pytest.mark.gpu


def _lse(wl, K, Qw):
    q = Qw.float().view(wl.B, wl.L, wl.H, wl.G * wl.w, wl.d)
    s = torch.einsum("blhrd,blhnd->blhrn", q, K.float()) / wl.d ** 0.5
    last = (wl.N - wl.w + torch.arange(wl.w, device="cuda")).repeat(wl.G)
    s.masked_fill_(torch.arange(wl.N, device="cuda")[None, :] > last[:, None], float("-inf"))
    return torch.logsumexp(s, dim=-1).view(wl.B, wl.L, wl.Hq, wl.w)


@pytest.mark.parametrize("L,H,G,w,N", [
    (1, 1, 1, 1, 129),        # one row, one item
    (20, 8, 4, 8, 700),       # 32 rows; 320 items, two chunks per unit
    (1, 3, 3, 11, 1300),      # 33 rows
    (19, 8, 1, 64, 640),      # 64 rows; 152 units of two chunks, the second is one full tile
    (1, 2, 5, 13, 641),       # 65 rows, one token in the last tile
    (40, 8, 4, 32, 512),      # 128 rows; 320 units of one chunk: the queries change with every item
    (20, 8, 3, 43, 520),      # 129 rows, one query buffer
    (20, 8, 8, 48, 600),      # 384 rows
    (20, 8, 8, 64, 1100),     # 512 rows
])
def test_items(L, H, G, w, N):
    from paper_2410_03090_b200.compress import CompressionPass
    avg = w + 20
    wl = replace(synth.WORKLOADS["c2"], L=L, H=H, Hq=H * G, N=N, w=w, avg_budget=avg, M=1, n_max=avg, seed=31)
    K, V, Qw = synth.generate(wl, "cuda")
    cp = CompressionPass(wl, "cuda")
    units = sorted({0, 1 % wl.units, wl.units // 2, wl.units - 1})
    for out in (lambda: cp.run(K, V, Qw), lambda: cp.run_one_call(K, V, Qw), lambda: cp.run_one_call(K, V, Qw, lse=_lse(wl, K, Qw)),
                lambda: cp.run(K, V, Qw, lse=_lse(wl, K, Qw))):
        cp.out.scores.fill_(-1)
        cp.out.entropy.fill_(-1)
        o = out()
        torch.cuda.synchronize()
        assert cp.status() == 0
        assert bool((o.scores >= 0).all()) and bool((o.entropy >= 0).all())
        parity.check_scores(wl, K, Qw, o.scores, units)
        parity.check_entropy(wl, K, o.entropy, o.erank, units)


@pytest.mark.parametrize("G,w,N", [(4, 8, 700), (1, 64, 641), (4, 32, 1300), (5, 40, 900), (6, 64, 769), (8, 64, 640)])
def test_column_sums_of_keys_with_a_mean(G, w, N):
    """Keys whose mean is ten times their spread: the covariance is what the subtraction of the column sums leaves, so the
    entropy only agrees when the sums come out of the same tiles as the Gram matrix, every feature in its place."""
    from paper_2410_03090_b200.compress import CompressionPass
    avg = w + 20
    wl = replace(synth.WORKLOADS["c2"], L=20, H=2, Hq=2 * G, N=N, w=w, avg_budget=avg, M=1, n_max=avg, seed=7)
    K, V, Qw = synth.generate(wl, "cuda")
    K = (K.float() + 10 * torch.linspace(-1, 2, wl.d, device="cuda").roll(G)).to(torch.bfloat16)
    cp = CompressionPass(wl, "cuda")
    for out in (lambda: cp.run(K, V, Qw), lambda: cp.run_one_call(K, V, Qw, lse=_lse(wl, K, Qw))):
        cp.out.entropy.fill_(-1)
        o = out()
        torch.cuda.synchronize()
        assert cp.status() == 0
        parity.check_entropy(wl, K, o.entropy, o.erank, [0, 17, wl.units - 1])


@pytest.mark.parametrize("w,how", [(32, "statistics"), (64, "statistics"), (32, "lse")])
@pytest.mark.parametrize("mean,whole", [(0, False), (1, False), (10, False), (100, False), (40, True), (100, True)])
def test_column_sums_over_the_longest_chunks(w, how, mean, whole):
    """Chunks of 8192 tokens, 512 additions into one accumulator, of keys with a mean of up to 100 times their spread, held to the
    tolerance of the entropy.  Whole numbers around 40: every sum fits 24 bits, so the covariance is exact and the entropy is
    good to the brackets of the eigenvalues (2e-8 of the largest, equal ones) and its own 24 bits."""
    from paper_2410_03090_b200 import binding as ub
    L, H, G, N, k = 32, 8, 4, 24576, 32
    g = torch.Generator(device="cuda").manual_seed(w + mean)
    K1 = torch.randn(H, N, 128, generator=g, device="cuda") * (1.0 if not whole else 1.5) + mean
    K1 = (K1.round().clamp(mean - 4, mean + 4) if whole else K1).to(torch.bfloat16)
    K = K1[None, None].expand(1, L, H, N, 128)
    Qw = torch.randn(1, L, H * G, w, 128, generator=g, device="cuda").to(torch.bfloat16)
    ctx = ub.Context(ub.make_shape(1, L, H, H * G, N, 128, w, "bf16"))
    if how == "lse":
        from paper_2410_03090_b200.compress import CompressionPass
        wl = replace(synth.WORKLOADS["c2"], L=L, H=H, Hq=H * G, N=N, w=w, avg_budget=100, M=1, n_max=100)
        cp = CompressionPass(wl, "cuda")
        cp.run_one_call(K, K, Qw, lse=torch.full((1, L, H * G, w), 20.0 + mean, device="cuda"))
        ent = cp.out.entropy
        assert cp.status() == 0
    else:
        ent, _ = ub.uncomp_entropy(ctx, K, k, Qw=Qw)
        assert ub.uncomp_status(ctx) == 0
    X = K1.double() - K1.double().mean(1, keepdim=True)
    lam = torch.linalg.eigvalsh(X.transpose(1, 2) @ X).flip(1)[:, :k]
    p = lam / lam.sum(1, keepdim=True)
    want = -(p * p.log()).sum(1)
    err = float((ent[0].double() - want).abs().max())
    assert err <= (1e-6 if whole and mean == 40 else parity.ENTROPY_RTOL * float(want.min()))
