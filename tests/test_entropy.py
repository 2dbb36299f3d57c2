"""Row entropy of the scaled softmax (Eq. 6) on the GPU against the oracle's, which is pinned in test_oracle_pins.py."""
import numpy as np
import pytest
import torch

from oracle import ahakv_oracle as orc
from paper_2506_03762_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,n,r,dtype_name,extra", [
    (1, 2, 2, 64, 512, 32, "F32", {}),
    (2, 8, 2, 128, 1500, 32, "BF16", dict(n_total=9000)),
    (1, 4, 4, 128, 4096, 64, "F16", {}),
    (1, 1, 1, 128, 300, 200, "F16", dict(scale_mode=0, scale=128 ** -0.5)),     # plain softmax, rows deep in the mask
    (1, 2, 1, 64, 129, 1, "BF16", {}),
    (1, 2, 2, 64, 700, 256, "F16", {}),                                         # the most rows a call takes
])
def test_row_entropy_matches_the_oracle(B, Hq, Hkv, d, n, r, dtype_name, extra):
    from paper_2506_03762_b200 import binding as ab
    from tests import parity
    dtype = getattr(ab, dtype_name)
    dt = {ab.F32: torch.float32, ab.F16: torch.float16, ab.BF16: torch.bfloat16}[dtype]
    g = torch.Generator().manual_seed(n + r)
    q = torch.randn((B, Hq, r, d), generator=g).to(dt).cuda()
    k = torch.randn((B, Hkv, n, d), generator=g).to(dt).cuda()
    p = ab.Params(B, Hq, Hkv, d, n, r, 16, 100, dtype=dtype, **extra)
    H = ab.ahakv_row_entropy(p, q, k).cpu().numpy().astype(np.float64)
    again = ab.ahakv_row_entropy(p, q, k).cpu().numpy()
    assert np.array_equal(H.astype(np.float32), again)                          # fixed reduction order
    op = parity.oracle_params(p)
    qn, kn = synth.to_numpy(q), synth.to_numpy(k)
    ref = np.stack([np.stack([orc.row_entropy(op, qn, kn, b, h) for h in range(Hq)]) for b in range(B)])
    assert H.shape == ref.shape == (B, Hq, r)
    # entropies are a few nats; FP32 sums of up to 4096 terms, approximate exp2 and log2
    tol = 2e-5 if dtype == ab.F32 else 1e-4
    assert np.abs(H - ref).max() <= tol * max(1.0, np.abs(ref).max()), np.abs(H - ref).max()
    assert (H >= -1e-6).all() and (H <= np.log(n) + 1e-6).all()


def test_entropy_tracks_eq10_on_gaussian_data():
    """Eq. 10: E[H_i] = ln i - lambda^2 d / 2 for unit-variance Gaussian queries and keys (an approximation that
    holds for small lambda^2 d; checked loosely), and Eq. 12's lambda brings the mean entropy near ln(budget)."""
    from paper_2506_03762_b200 import binding as ab
    B, H, d, n, r, Bud = 4, 8, 128, 8192, 32, 2048
    g = torch.Generator().manual_seed(5)
    q = torch.randn((B, H, r, d), generator=g).to(torch.float16).cuda()
    k = torch.randn((B, H, n, d), generator=g).to(torch.float16).cuda()
    lam = 0.05
    p = ab.Params(B, H, H, d, n, r, 16, Bud, dtype=ab.F16, scale_mode=ab.SCALE_FIXED, scale=lam)
    Hm = float(ab.ahakv_row_entropy(p, q, k).double().mean())
    assert abs(Hm - (np.log(n) - lam * lam * d / 2)) < 0.05, Hm
    p12 = ab.Params(B, H, H, d, n, r, 16, Bud, dtype=ab.F16)                    # Eq. 12 per row
    H12 = float(ab.ahakv_row_entropy(p12, q, k).double().mean())
    assert abs(H12 - np.log(Bud)) < 0.35, (H12, np.log(Bud))


@pytest.mark.parametrize("scale", [1e-30, 1e-12, 1e6, 1e9])
def test_row_entropy_at_the_ends_of_the_scale(scale):
    """A caller who tunes the scale may try any positive number.  A vanishing one makes every row uniform over the keys it sees
    (H_i = ln i), a huge one concentrates it on a single key (H_i = 0); masked keys weigh nothing in either."""
    from paper_2506_03762_b200 import binding as ab
    d, n, r = 64, 700, 64
    g = torch.Generator().manual_seed(11)
    q = torch.randn((1, 2, r, d), generator=g).to(torch.float16).cuda()
    k = torch.randn((1, 2, n, d), generator=g).to(torch.float16).cuda()
    p = ab.Params(1, 2, 2, d, n, r, 4, 80, dtype=ab.F16, scale_mode=ab.SCALE_FIXED, scale=scale)
    H = ab.ahakv_row_entropy(p, q, k).cpu().double()
    if scale < 1:
        want = torch.log(torch.arange(n - r + 1, n + 1, dtype=torch.float64)).expand_as(H)
    else:
        want = torch.zeros_like(H)
    assert bool(((H - want).abs() < 1e-5).all()), (H - want).abs().max()


@pytest.mark.parametrize("B,H,d,n,r,scale,sharp", [(1, 4, 128, 5000, 64, 0.3, 1.0), (1, 4, 64, 9000, 100, 1.0, 1.0), (2, 3, 128, 1100, 17, 1.0, 3.0),
                                                   (1, 1, 64, 20000, 128, 0.02, 1.0)])
def test_small_entropies_under_large_logits(B, H, d, n, r, scale, sharp):
    """Rows whose largest logit is hundreds and whose entropy is far below 1, against a float64 evaluation.  The logits are sums
    of d exact products in FP32, scaled in FP32: each is off by some ulps of its size, u = 2^-24 x (8 + |x| / ln 2) in the
    exponent, and an entropy moves by at most the mean |x - E x| of its row, itself of the order of H + its spread, times that;
    what comes on top is FP32 rounding of terms no larger than max(1, H).  Nothing may depend on the logits' own size beyond."""
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator().manual_seed(n)
    q = (sharp * torch.randn((B, H, r, d), generator=g)).to(torch.float16).cuda()
    k = torch.randn((B, H, n, d), generator=g).to(torch.float16).cuda()
    p = ab.Params(B, H, H, d, n, r, 4, 80, dtype=ab.F16, scale_mode=ab.SCALE_FIXED, scale=scale)
    got = ab.ahakv_row_entropy(p, q, k).double()
    x = float(torch.tensor(scale, dtype=torch.float32)) * q.double() @ k.double().transpose(-1, -2)
    seen = torch.arange(n, device="cuda") <= torch.arange(n - r, n, device="cuda").view(r, 1)
    x = x.masked_fill(~seen, float("-inf"))
    lse = x.logsumexp(-1, keepdim=True)
    a = (x - lse).exp()
    dev = (x - lse).masked_fill(~seen, 0)
    want = -(a * dev).sum(-1)
    spread = (a * (dev + want.unsqueeze(-1)).abs()).sum(-1)
    size = x.amax(-1).abs() / 0.6931
    bound = 2.0 ** -24 * (4 * (8 + size) * spread + 16 * want.clamp(min=1.0))
    assert bool((got >= -2.0 ** -22).all())
    assert bool(((got - want).abs() <= bound).all()), ((got - want).abs() / bound).max()


def test_entropy_scratch_for_a_large_call_serves_the_smaller_ones():
    """Scratch sized for the largest batch and context a caller has must do for every smaller call."""
    from paper_2506_03762_b200 import binding as ab
    def need(B, n, r, dtype, G=4):
        return ab.ahakv_entropy_workspace_bytes(ab.Params(B, 4 * G, 4, 128, n, r, 0, 64, dtype=dtype))
    for dtype in (ab.F16, ab.F32):
        for n in (64, 127, 128, 300, 1000, 4096, 30000):
            for r in (1, 16, 33, 64):
                sizes = [need(B, n, r, dtype) for B in range(1, 161)]
                assert sizes == sorted(sizes), (dtype, n, r)
        for B in (1, 5, 9, 37, 40, 150):
            sizes = [need(B, n, 32, dtype) for n in (*range(32, 1200, 31), 3000, 8000, 8192, 20000, 70000)]
            assert sizes == sorted(sizes), (dtype, B)
            sizes = [need(B, 5000, r, dtype) for r in range(1, 65)]
            assert sizes == sorted(sizes), (dtype, B)
