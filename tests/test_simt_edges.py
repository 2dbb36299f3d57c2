"""The float32 scoring kernels at the edges of their 64-key tiles, 128-key blocks and 32-row chunks, grouped and pooled by
maximum, against a float64 evaluation of Eq. 1, 5, 9 on the same inputs; 1e-5 relative as for every float32 score (the
logits and shifts are formed in double; what is left is a few FP32 roundings and ex2's two units in the last place)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,n,r,flags", [
    (1, 1, 1, 64, 1, 1, 0), (1, 2, 2, 128, 63, 5, 0), (2, 2, 1, 64, 65, 16, 0), (1, 3, 1, 128, 128, 11, 4),
    (1, 4, 2, 64, 129, 33, 4), (1, 2, 2, 128, 193, 32, 0), (1, 8, 1, 64, 700, 32, 0), (1, 1, 1, 128, 1025, 256, 0)])
def test_float32_scores_at_tile_edges(B, Hq, Hkv, d, n, r, flags):
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator().manual_seed(n + r)
    q = (3 * torch.randn((B, Hq, r, d), generator=g)).cuda()
    k = torch.randn((B, Hkv, n, d), generator=g).cuda()
    v = torch.randn((B, Hkv, n, d), generator=g).cuda()
    p = ab.Params(B, Hq, Hkv, d, n, r, 0, max(1, n // 2), dtype=ab.F32, scale_mode=ab.SCALE_FIXED, scale=0.09, flags=flags)
    score = torch.empty((B, Hkv, n), device="cuda")
    ab.ahakv_score(p, q, k, v, None, score, ab.alloc_workspace(p))
    G = Hq // Hkv
    w = float(torch.tensor(0.09, dtype=torch.float32)) * q.double() @ k.double().repeat_interleave(G, 1).transpose(-1, -2)
    seen = torch.arange(n, device="cuda") <= torch.arange(n - r, n, device="cuda").view(r, 1)
    a = w.masked_fill(~seen, float("-inf")).softmax(-1).sum(2).view(B, Hkv, G, n)
    want = a.amax(2) if flags & ab.FLAG_GROUP_MAX else a.mean(2)
    assert torch.allclose(score.double(), want, rtol=1e-5, atol=1e-5 * 1e-3 * r / n)


@pytest.mark.parametrize("B,Hq,Hkv,d,n,r", [
    (1, 1, 1, 128, 65, 1),          # two CTAs, one of them with a single key
    (1, 8, 8, 128, 3001, 32),       # ten CTAs a head, four and five tiles each
    (1, 8, 2, 64, 1000, 16),        # two chunks of rows
    (2, 6, 2, 128, 900, 33),        # a last chunk of three rows
    (3, 4, 4, 128, 2000, 32),       # eight CTAs a head, four tiles each
    (4, 16, 16, 64, 1000, 32),      # four CTAs a head, two of them on an SM
    (4, 16, 16, 128, 1500, 16),     # two CTAs a head, twelve tiles each
    (1, 8, 8, 64, 1020, 20),        # sixteen CTAs a head, one tile each, two on an SM
    (1, 3, 1, 64, 513, 80),         # 240 rows
])
def test_float32_scores_by_clusters(B, Hq, Hkv, d, n, r):
    """Calls whose tiles are all on the GPU at once: one kernel does both passes, and an eviction call is two or three launches."""
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator(device="cuda").manual_seed(n + r)
    q = 3 * torch.randn((B, Hq, r, d), generator=g, device="cuda")
    k, v = (torch.randn((B, Hkv, n, d), generator=g, device="cuda") for _ in range(2))
    p = ab.Params(B, Hq, Hkv, d, n, r, 0, max(1, n // 2), dtype=ab.F32, scale_mode=ab.SCALE_FIXED, scale=0.09, flags=0)
    score = torch.empty((B, Hkv, n), device="cuda")
    before = ab.ahakv_launch_count()
    ab.ahakv_score(p, q, k, v, None, score, ab.alloc_workspace(p))
    assert ab.ahakv_launch_count() - before == 2
    G = Hq // Hkv
    w = float(torch.tensor(0.09, dtype=torch.float32)) * q.double() @ k.double().repeat_interleave(G, 1).transpose(-1, -2)
    seen = torch.arange(n, device="cuda") <= torch.arange(n - r, n, device="cuda").view(r, 1)
    want = w.masked_fill(~seen, float("-inf")).softmax(-1).sum(2).view(B, Hkv, G, n).mean(2)
    assert torch.allclose(score.double(), want, rtol=1e-5, atol=1e-5 * 1e-3 * r / n)


@pytest.mark.parametrize("where", ["key", "infinite key", "query", "head"])
def test_float32_scores_of_nan_inputs_are_the_same_by_either_path(where):
    """Four heads go by clusters, the same four among 32 through the two kernels: what is not a number counts as nothing in both."""
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator(device="cuda").manual_seed(7)
    q = torch.randn((1, 32, 32, 64), generator=g, device="cuda")
    k, v = (torch.randn((1, 32, 1000, 64), generator=g, device="cuda") for _ in range(2))
    if where == "key": k[0, 1, 300, 5] = float("nan")
    if where == "infinite key": k[0, 1, 300, 5] = float("inf")
    if where == "query": q[0, 1, 7, 3] = float("nan")
    if where == "head": k[0, 1] = float("nan")
    scores = []
    for heads, launches in ((4, 2), (32, 3)):
        p = ab.Params(1, heads, heads, 64, 1000, 32, 0, 500, dtype=ab.F32, scale_mode=ab.SCALE_FIXED, scale=0.09, flags=0)
        score = torch.empty((1, heads, 1000), device="cuda")
        before = ab.ahakv_launch_count()
        ab.ahakv_score(p, *(t[:, :heads].contiguous() for t in (q, k, v)), None, score, ab.alloc_workspace(p))
        assert ab.ahakv_launch_count() - before == launches
        scores.append(score[:, :4])
    assert torch.allclose(*scores, rtol=1e-5, atol=0) and scores[0].isfinite().all()


@pytest.mark.parametrize("n,r,Hq,Hkv,flags", [(9001, 64, 4, 4, 1), (9100, 20, 12, 4, 5)])
def test_scores_with_and_without_room_for_numerators_agree(n, r, Hq, Hkv, flags):
    """The library's own scratch is too small for these cases' softmax numerators, so that the logits are formed twice; with
    a workspace of the size asked for they are kept.  (That the two agree to the bit is tested below.)"""
    from paper_2506_03762_b200 import binding as ab
    g = torch.Generator().manual_seed(n)
    q = torch.randn((1, Hq, r, 64), generator=g).cuda()
    k, v = (torch.randn((1, Hkv, n, 64), generator=g).cuda() for _ in range(2))
    p = ab.Params(1, Hq, Hkv, 64, n, r, 4, 40, dtype=ab.F32, flags=flags)
    assert ab.ahakv_workspace_bytes(p) > ab.ahakv_static_workspace_bytes()
    a, b = (torch.empty((1, Hkv, n), device="cuda") for _ in range(2))
    ab.ahakv_score(p, q, k, v, None, a, ab.alloc_workspace(p))
    ab.ahakv_score_static(p, q, k, v, None, b)
    assert torch.allclose(a, b, rtol=1e-5, atol=0)


@pytest.mark.parametrize("large,small", [
    (dict(batch=24, n=3001), dict(batch=20, n=3001)),         # the smaller batch asks for room for its numerators, the larger does not
    (dict(batch=1, n=66000), dict(batch=1, n=20000)),
])
def test_scratch_for_a_large_call_serves_the_smaller_ones(large, small):
    from paper_2506_03762_b200 import binding as ab
    params = lambda batch, n: ab.Params(batch, 8, 8, 64, n, 32, 4, 100, dtype=ab.F32)
    p = params(**small)
    ws = ab.alloc_workspace(params(**large))
    assert ws.nbytes < ab.ahakv_workspace_bytes(p)
    g = torch.Generator(device="cuda").manual_seed(5)
    q = torch.randn((p.batch, 8, 32, 64), generator=g, device="cuda")
    k, v = (torch.randn((p.batch, 8, p.n_ctx, 64), generator=g, device="cuda") for _ in range(2))
    a, b = (torch.empty((p.batch, 8, p.n_ctx), device="cuda") for _ in range(2))
    ab.ahakv_score(p, q, k, v, None, a, ws)
    ab.ahakv_score(p, q, k, v, None, b, ab.alloc_workspace(p))
    assert torch.allclose(a, b, rtol=1e-5, atol=0)
    outs = ab.alloc_outputs(p), ab.alloc_outputs(p)
    ab.ahakv_evict(p, q, k, v, None, *outs[0], ws)
    ab.ahakv_evict(p, q, k, v, None, *outs[1], ab.alloc_workspace(p))
    assert torch.allclose(outs[0][2], outs[1][2], rtol=1e-5, atol=0)


@pytest.mark.parametrize("Hq,Hkv,n,r,flags", [(8, 8, 3001, 32, 1), (12, 4, 3300, 20, 5), (6, 2, 6100, 33, 1), (4, 4, 6007, 64, 4), (8, 8, 4099, 1, 1)])
def test_scores_do_not_depend_on_the_room_for_numerators(Hq, Hkv, n, r, flags):
    """A sequence of a ragged batch, a call on the library's own scratch and a call on scratch of another size get exactly what
    a call with all the room it asks for gets: bit for bit, whether numerators are kept or formed twice."""
    from paper_2506_03762_b200 import binding as ab
    p = ab.Params(1, Hq, Hkv, 128, n, r, 4, 300, dtype=ab.F32, flags=flags)
    need = ab.ahakv_workspace_bytes(p)
    kept = Hkv * (Hq // Hkv) * r * n * 4
    assert need > kept, "the call keeps its numerators"
    g = torch.Generator(device="cuda").manual_seed(n)
    q = 3 * torch.randn((1, Hq, r, 128), generator=g, device="cuda")
    k, v = (torch.randn((1, Hkv, n, 128), generator=g, device="cuda") for _ in range(2))
    ws = ab.alloc_workspace(p)
    a, b = (torch.empty((1, Hkv, n), device="cuda") for _ in range(2))
    ab.ahakv_score(p, q, k, v, None, a, ws)
    ab.ahakv_score(p, q, k, v, None, b, ws, ws_bytes=need - kept)
    assert torch.equal(a, b)
    outs = ab.alloc_outputs(p), ab.alloc_outputs(p)
    ab.ahakv_evict(p, q, k, v, None, *outs[0], ws)
    ab.ahakv_evict(p, q, k, v, None, *outs[1], ws, ws_bytes=need - kept)
    for x, y in zip(*outs):
        assert torch.equal(x, y)
