"""Refinement and selection at the sizes where a cluster of CTAs per head can go wrong: the edges of a thread's run of
tokens, of a CTA and of a cluster, rows that do not start on 16-byte boundaries, many heads, ties and scores over many
octaves.  Selection has no tolerance: the reference is a stable sort of the same float32 scores."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _expected(s, Br, Bud):
    n = s.shape[-1]
    if n <= Bud:
        return np.arange(n)
    order = np.argsort(-s[: n - Br], kind="stable")[: Bud - Br]
    return np.concatenate([np.sort(order), np.arange(n - Br, n)])


@pytest.mark.parametrize("H,n,Br,Bud", [
    (3, 1, 0, 1), (2, 7, 2, 5), (5, 511, 0, 100), (5, 513, 3, 512), (4, 1025, 0, 1), (4, 2049, 64, 300),
    (3, 4096, 128, 1024), (3, 4097, 0, 4000), (3, 8191, 1, 513), (2, 65535, 7, 3000), (2, 65537, 0, 65536),
    (1, 131072, 128, 40000), (1, 131073, 128, 40000), (160, 8200, 16, 700), (160, 4098, 0, 2000)])
@pytest.mark.parametrize("kind", ["spread", "ties", "octaves", "one_bin"])
def test_selection_equals_a_stable_sort(H, n, Br, Bud, kind):
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator().manual_seed(n * 31 + H)
    s = torch.rand((1, H, n), generator=g)
    if kind == "ties":
        s = torch.round(s * 9) / 9
    elif kind == "octaves":
        s = torch.exp2(-60 * s) * torch.where(torch.rand(s.shape, generator=g) < 0.1, -1.0, 1.0)
    elif kind == "one_bin":
        s = 1.0 + s * 2.0 ** -9                              # everything in a few bins of the first histogram
    s = s.cuda()
    p = ab.Params(1, H, H, 64, n, 1, Br, Bud, dtype=ab.F16, flags=0)
    idx = torch.full((1, H, min(n, Bud)), -7, dtype=torch.int32, device="cuda")
    ab.ahakv_select(p, s, idx)
    sn, got = s.cpu().numpy(), idx.cpu().numpy()
    for h in range(0, H, max(1, H // 4)):
        assert np.array_equal(got[0, h], _expected(sn[0, h], Br, Bud))


@pytest.mark.parametrize("H,n", [(1, 65552), (1, 98304), (1, 98305), (200, 12288), (200, 12290)])     # nine to thirteen tokens a thread
@pytest.mark.parametrize("kind", ["spread", "one_bin"])
def test_selection_around_twelve_tokens_a_thread(H, n, kind):
    test_selection_equals_a_stable_sort(H, n, 5, n // 3, kind)


@pytest.mark.parametrize("n", [130, 1027, 4100, 9001, 33001])
@pytest.mark.parametrize("pool,flags", [(1, 1), (3, 1), (7, 1), (7, 3), (31, 1)])
def test_refinement_in_the_eviction_call_equals_the_definition(n, pool, flags):
    """The refined score against Eq. 13-15 in float64 from the same raw scores (value prior off) and the same value rows;
    both sides round the norms of 64 float16 squares and a handful of products once each, so 1e-5 relative holds."""
    from paper_2506_03762_b200 import binding as ab
    B, H, d, r, Br, Bud = 1, 2, 64, 16, 8, 64
    g = torch.Generator().manual_seed(n + pool)
    q = torch.randn((B, H, r, d), generator=g).half().cuda()
    k = torch.randn((B, H, n, d), generator=g).half().cuda()
    v = (torch.randn((B, H, n, d), generator=g) * (0.2 + torch.rand((B, H, n, 1), generator=g))).half().cuda()
    prev = (torch.rand((B, H, n), generator=g) * 1e-3).cuda()
    p = ab.Params(B, H, H, d, n, r, Br, Bud, dtype=ab.F16, flags=flags, pool_kernel=pool)
    ws = ab.alloc_workspace(p)
    raw, score = torch.empty((B, H, n), device="cuda"), torch.empty((B, H, n), device="cuda")
    p.flags = 0
    ab.ahakv_score(p, q, k, None, None, raw, ws)
    p.flags = flags
    ab.ahakv_score(p, q, k, v, prev, score, ws)
    k_out, v_out, s_out, idx = ab.alloc_outputs(p)
    ab.ahakv_evict(p, q, k, v, prev, k_out, v_out, s_out, idx, ws)
    nu = v.double().square().sum(-1)
    ones = torch.ones((1, 1, pool), dtype=torch.float64, device="cuda")
    tot = torch.nn.functional.conv1d(nu.view(B * H, 1, n), ones, padding=pool // 2).view(B, H, n)
    cnt = torch.nn.functional.conv1d(torch.ones_like(nu).view(B * H, 1, n), ones, padding=pool // 2).view(B, H, n)
    gamma = tot / pool if flags & ab.FLAG_POOL_ZERO_PAD else tot / cnt
    want = raw.double() * gamma / gamma.amax(-1, keepdim=True) + prev.double()
    assert torch.allclose(score.double(), want, rtol=1e-5, atol=0)
    sn = score.cpu().numpy()
    for h in range(H):
        assert np.array_equal(idx[0, h].cpu().numpy(), _expected(sn[0, h], Br, Bud))
    assert torch.equal(s_out, score.gather(-1, idx.long()))


@pytest.mark.parametrize("d,Bud", [(64, 9), (64, 255), (64, 257), (64, 500), (128, 129), (128, 250)])
def test_rows_gathered_by_the_selecting_cta_are_the_kept_ones(d, Bud):
    """Copies: bit for bit, also where a thread's last rows are fewer than it has in flight."""
    from paper_2506_03762_b200 import binding as ab
    B, H, n, r, Br = 2, 3, 1500, 16, 8
    g = torch.Generator().manual_seed(Bud + d)
    q, k, v = (torch.randn((B, H, m, d), generator=g).half().cuda() for m in (r, n, n))
    p = ab.Params(B, H, H, d, n, r, Br, Bud, dtype=ab.F16, flags=1)
    ws = ab.alloc_workspace(p)
    k_out, v_out, s_out, idx = ab.alloc_outputs(p)
    ab.ahakv_evict(p, q, k, v, None, k_out, v_out, s_out, idx, ws)
    at = idx.long().unsqueeze(-1).expand(-1, -1, -1, d)
    assert torch.equal(k_out, k.gather(2, at)) and torch.equal(v_out, v.gather(2, at))


@pytest.mark.parametrize("H,n", [(2, 700), (3, 4096), (2, 9001), (1, 70001)])
@pytest.mark.parametrize("m", [1, 2, 63, 64, 65, 127, 129, 512, 513, 600])
def test_threshold_among_m_close_scores(H, n, m):
    """`m` distinct scores within one bin of the first histogram, the threshold in the middle of them; around the most that are
    ranked from a list."""
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator().manual_seed(n + m)
    s = torch.rand((1, H, n), generator=g) * 0.5
    for h in range(H):
        at = torch.randperm(n, generator=g)[:m]
        s[0, h, at] = 1.0 + torch.randperm(m, generator=g).float() * 2.0 ** -20
    keep = max(1, m // 2)
    p = ab.Params(1, H, H, 64, n, 1, 0, keep, dtype=ab.F16, flags=0)
    idx = torch.full((1, H, keep), -7, dtype=torch.int32, device="cuda")
    ab.ahakv_select(p, s.cuda(), idx)
    for h in range(H):
        assert np.array_equal(idx[0, h].cpu().numpy(), _expected(s[0, h].numpy(), 0, keep))


def test_time_of_a_selection_does_not_hang_on_the_distribution():
    """2048 heads that drop one of 1000 tokens each: scores over many octaves, where half of a head's tokens lie below the first
    histogram's range, may take a few passes more than uniform ones, not seven times as long as ranking them by pairs did."""
    from paper_2506_03762_b200 import binding as ab
    u = torch.rand((64, 32, 1000), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    p = ab.Params(64, 32, 32, 64, 1000, 1, 0, 999, dtype=ab.F16, flags=0)
    idx = torch.empty((64, 32, 999), dtype=torch.int32, device="cuda")

    def us(s):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(5):
            a.record()
            for _ in range(10):
                ab.ahakv_select(p, s, idx)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    assert us(torch.exp(20 * u - 30)) < 3 * us(u)
