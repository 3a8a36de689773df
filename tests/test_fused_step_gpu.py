"""The fused step (append, score, select + FILL compaction in one call) on the cases its single-eviction path has of
its own: the token to evict is the unit's last row (nothing moves), or any other row (the last row fills the hole),
checked on the cache contents, not only on the indices."""
import pytest
import torch

import paper_2504_14051_b200 as P

pytestmark = pytest.mark.gpu
DEV = "cuda"


def make_cache(B, H, d, n, cap, dtype, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    c = P.EvictionCache(B, H, H, d, cap, 1, dtype, n, "last_query", "fill", d ** -0.5, max_evict=1, device=DEV)
    K0 = torch.randn((B, H, cap, d), generator=g).to(dtype).to(DEV)
    V0 = torch.randn((B, H, cap, d), generator=g).to(dtype).to(DEV)
    c.load(K0, V0, torch.full((B,), n, dtype=torch.int32, device=DEV))
    q = torch.randn((B, H, 1, d), generator=g).to(dtype).to(DEV)
    vn = torch.randn((B, H, 1, d), generator=g).to(dtype).to(DEV)
    return c, q, vn, g


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.float32, 64), (torch.float32, 128)])
@pytest.mark.parametrize("n", [37, 2049, 9000])
def test_new_token_with_the_lowest_score_is_evicted_in_place(dtype, d, n):
    """One head per unit; the new key points away from the query (logit -20 below zero), so the new token has by far
    the smallest weight and score: it is the unit's last row, which is evicted without a move."""
    B, H, cap = 3, 2, n + 8
    c, q, vn, _ = make_cache(B, H, d, n, cap, dtype, 100 + n)
    qf = q.float()
    kn = (-(20.0 / (d ** -0.5 * (qf * qf).sum(-1, keepdim=True))) * qf).to(dtype)
    K0, V0, pos0 = c.K.clone(), c.V.clone(), c.pos.clone()
    c.step(q, kn, vn)
    torch.cuda.synchronize()
    assert c.status() == 0
    assert c.n_evict.tolist() == [1] * B and c.lens.tolist() == [n] * B
    assert (c.evict_idx[:, :, 0] == n).all()
    assert torch.equal(c.K[:, :, :n], K0[:, :, :n]) and torch.equal(c.V[:, :, :n], V0[:, :, :n])
    assert torch.equal(c.pos[:, :, :n], pos0[:, :, :n])


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.float32, 64), (torch.float32, 128)])
@pytest.mark.parametrize("n", [37, 2049, 9000])
def test_last_row_fills_the_hole(dtype, d, n):
    """The new key is the query's direction (the largest weight by far), so some older token goes: the new token's row
    lands in its slot, every other row stays where it was."""
    B, H, cap = 3, 2, n + 8
    c, q, vn, _ = make_cache(B, H, d, n, cap, dtype, 200 + n)
    qf = q.float()
    kn = ((12.0 / (d ** -0.5 * (qf * qf).sum(-1, keepdim=True))) * qf).to(dtype)
    K0, V0, pos0 = c.K.clone(), c.V.clone(), c.pos.clone()
    c.step(q, kn, vn)
    torch.cuda.synchronize()
    assert c.status() == 0
    assert c.n_evict.tolist() == [1] * B and c.lens.tolist() == [n] * B
    scores = c.scores.clone()
    for b in range(B):
        for h in range(H):
            e = int(c.evict_idx[b, h, 0])
            assert 0 <= e < n
            # the evicted slot is the argmin of the scores this call wrote (ties: the lower position)
            sc = scores[b, h, :n + 1]
            assert float(sc[e]) == float(sc.min())
            assert e == int(torch.nonzero(sc == sc.min())[0])
            keep = torch.ones(n, dtype=torch.bool, device=DEV)
            keep[e] = False
            assert torch.equal(c.K[b, h, :n][keep], K0[b, h, :n][keep])
            assert torch.equal(c.V[b, h, :n][keep], V0[b, h, :n][keep])
            assert torch.equal(c.K[b, h, e], kn[b, h, 0]) and torch.equal(c.V[b, h, e], vn[b, h, 0])
            assert int(c.pos[b, h, e]) == n and torch.equal(c.pos[b, h, :n][keep], pos0[b, h, :n][keep])


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.float32, 64)])
@pytest.mark.parametrize("n", [300, 9000])
def test_equal_lowest_scores_go_by_position(dtype, d, n):
    """Three cached tokens of every unit are copies of one another (same key, same value) with by far the smallest
    weight, so their scores are the unit's lowest and, computed the same way, equal; positions are a permutation, so the
    copy in the highest slot can have the lowest position. The evicted slot is the arg-min over (score bits, position)
    of the scores this call wrote."""
    B, H, cap = 2, 2, n + 8
    c, q, vn, g = make_cache(B, H, d, n, cap, dtype, 300 + n)
    qf = q.float()
    low = (-(20.0 / (d ** -0.5 * (qf * qf).sum(-1, keepdim=True))) * qf).to(dtype)  # [B, H, 1, d]
    K0, V0 = c.K.clone(), c.V.clone()
    copies = [5, n // 2, n - 2]
    for j in copies:
        K0[:, :, j] = low[:, :, 0]
        V0[:, :, j] = V0[:, :, 5]
    pos0 = torch.stack([torch.stack([torch.randperm(cap, generator=g) for _ in range(H)]) for _ in range(B)]).to(torch.int32).to(DEV)
    c.load(K0, V0, torch.full((B,), n, dtype=torch.int32, device=DEV), pos=pos0)
    c.n_seen.fill_(cap)  # the new token's position: above every cached one
    kn = ((12.0 / (d ** -0.5 * (qf * qf).sum(-1, keepdim=True))) * qf).to(dtype)
    c.step(q, kn, vn)
    torch.cuda.synchronize()
    assert c.status() == 0 and c.n_evict.tolist() == [1] * B
    ties = 0
    for b in range(B):
        for h in range(H):
            sc = c.scores[b, h, :n + 1]
            cand = torch.nonzero(sc == sc.min()).flatten()
            ties += int(len(cand) > 1)
            pos_pre = torch.cat([pos0[b, h, :n], torch.tensor([cap], dtype=torch.int32, device=DEV)])
            want = int(cand[torch.argmin(pos_pre[cand])])
            assert int(c.evict_idx[b, h, 0]) == want
            assert want in copies
    assert ties > 0, "the copies' scores were expected to be equal in at least one unit"


@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, d, cap, lengths, budgets: sequences that grow, that evict one, that have no room, that would have to
    # evict two, a new token on a tile of its own, more CTAs in the cluster than tiles
    (4, 8, 2, 128, 1296, [1279, 1295, 1296, 300], [1400, 1295, 1296, 299]),
    (2, 14, 2, 128, 400, [128, 255], [128, 400]),
    (5, 8, 8, 64, 2064, [1, 127, 128, 2047, 2063], [1, 127, 500, 2047, 2063]),
    # the CUDA-core form: fp32, 16 heads per group, one tile per CTA, several, a single CTA
    (4, 4, 2, 64, 272, [1, 64, 255, 271], [1, 64, 255, 400], torch.float32),
    (8, 6, 2, 128, 2048, [2047, 1024, 700, 1, 2, 513, 65, 2046], [2047, 1024, 699, 1, 2, 513, 65, 2046], torch.float32),
    (3, 16, 1, 64, 1024, [1023, 513, 512], [1023, 513, 511], torch.float32),
    (2, 3, 1, 128, 64, [63, 64], [63, 64], torch.float32),
    (3, 32, 2, 128, 512, [511, 449, 448], [511, 449, 447]),
    (2, 16, 1, 64, 400, [128, 399], [128, 390]),
])
@pytest.mark.parametrize("mode", ["last_query", "accum", "external"])
@pytest.mark.parametrize("fast", [False, True])
def test_whole_step_kernel_equals_the_four_calls(shape, mode, fast):
    """Steps on few units are one launch; the same calls made one after the other on a copy of the state give the same
    cache, lengths, positions, sums and status, and scores to the rounding of the two compilations."""
    B, Hq, Hkv, d, cap, lens, budget, dt = (*shape, torch.bfloat16)[:8]
    g = torch.Generator(device="cpu").manual_seed(cap + d)
    name = "small_step_kernel" if dt == torch.float32 or Hq // Hkv > 8 else "decode_step_kernel"
    mk = lambda: P.EvictionCache(B, Hq, Hkv, d, cap, 1, dt, torch.tensor(budget, dtype=torch.int32), mode, "fill", max_evict=1,
                                 method="fast" if fast else "caote", device=DEV)
    a, b = mk(), mk()
    K0, V0 = (torch.randn((B, Hkv, cap, d), generator=g).to(dt) for _ in range(2))
    base0 = torch.rand((B, Hkv, cap), generator=g) + 0.1
    pos0 = torch.stack([torch.stack([torch.randperm(cap, generator=g) for _ in range(Hkv)]) for _ in range(B)]).to(torch.int32)
    for c in (a, b):
        c.load(K0, V0, torch.tensor(lens, dtype=torch.int32), base=base0, pos=pos0)
        c.n_seen.fill_(cap + 7)
    p = a.params
    for step in range(3):
        q = torch.randn((B, Hq, 1, d), generator=g).to(dt).to(DEV)
        kn, vn = (torch.randn((B, Hkv, 1, d), generator=g).to(dt).to(DEV) for _ in range(2))
        P.caote_trace_enable(True)
        a.step(q, kn, vn)
        torch.cuda.synchronize()
        assert set(P.caote_trace_collect()) == {name}
        P.caote_trace_enable(False)
        P.caote_append(p, b.K, b.V, b.base, b.pos, b.lens, b.n_seen, kn, vn, b.workspace)
        if fast:
            P.caote_vsum(p, b.V, b.lens, b.vsum)
            P.caote_score_fast(p, q, b.K, b.V, b.lens, b.base, b.vsum, b.o, b.scores, b.workspace)
        else:
            P.caote_score(p, q, b.K, b.V, b.lens, b.base, b.o, b.scores, b.workspace)
        P.caote_select_evict(p, b.scores, b.lens, b.budget, b.pos, b.evict_idx, b.n_evict, b.workspace)
        P.caote_compact(p, b.K, b.V, b.base, b.pos, b.lens, b.evict_idx, b.n_evict, "fill", b.workspace)
        torch.cuda.synchronize()
        assert a.status() == b.status()
        assert a.lens.tolist() == b.lens.tolist() and a.n_seen.tolist() == b.n_seen.tolist() and a.n_evict.tolist() == b.n_evict.tolist()
        # (16 heads per group: the four calls run on the tensor cores, P in 16 bits)
        tol = 2e-5 if dt == torch.bfloat16 and Hq // Hkv > 8 else 1e-6
        torch.testing.assert_close(a.o, b.o, rtol=1e-5, atol=tol)
        for s in range(B):
            n = int(a.lens[s])
            if int(a.n_evict[s]):
                assert torch.equal(a.evict_idx[s], b.evict_idx[s])
            assert torch.equal(a.K[s, :, :n], b.K[s, :, :n]) and torch.equal(a.V[s, :, :n], b.V[s, :, :n])
            assert torch.equal(a.pos[s, :, :n], b.pos[s, :, :n])
            torch.testing.assert_close(a.base[s, :, :n], b.base[s, :, :n], rtol=1e-5, atol=1e-6)
            torch.testing.assert_close(a.scores[s, :, :n], b.scores[s, :, :n], rtol=1e-4, atol=1e-6)
        if fast:
            ref = P.EvictionCache(B, Hq, Hkv, d, cap, 1, dt, 1, mode, "fill", method="fast", device=DEV)
            P.caote_vsum(p, a.V, a.lens, ref.vsum)
            # a handful of fp32 additions on sums of up to 2 k normal values (about 45): 1e-5 each
            torch.testing.assert_close(a.vsum, ref.vsum, rtol=1e-5, atol=1e-3)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [
    # B, Hq, Hkv, d, cap, m, budget, dtype
    (3, 14, 2, 128, 400, 1, 390, torch.bfloat16),
    (2, 8, 2, 64, 272, 40, 200, torch.bfloat16),
    (2, 4, 2, 64, 100, 3, 90, torch.float32),
])
@pytest.mark.parametrize("compact", ["fill", "stable"])
@pytest.mark.parametrize("method", ["sum_errors", "post_evict"])
def test_variant_steps_equal_their_separate_calls(shape, compact, method):
    """The whole steps of the two variants launch the kernels of the separate calls (one fused selection aside): the same
    bits everywhere."""
    B, Hq, Hkv, d, cap, m, budget, dt = shape
    g = torch.Generator(device="cpu").manual_seed(cap)
    a, b = (P.EvictionCache(B, Hq, Hkv, d, cap, m, dt, budget, "last_query", compact, method=method, device=DEV) for _ in range(2))
    K0, V0 = (torch.randn((B, Hkv, cap, d), generator=g).to(dt) for _ in range(2))
    for c in (a, b):
        c.load(K0, V0, torch.tensor([budget - 5 * s for s in range(B)], dtype=torch.int32))
    p = a.params
    for _ in range(7):
        q = torch.randn((B, Hq, m, d), generator=g).to(dt).to(DEV)
        kn, vn = (torch.randn((B, Hkv, m, d), generator=g).to(dt).to(DEV) for _ in range(2))
        a.step(q, kn, vn)
        P.caote_append(p, b.K, b.V, b.base, b.pos, b.lens, b.n_seen, kn, vn, b.workspace)
        if method == "sum_errors":
            P.caote_score_sum_errors(p, q, b.K, b.V, b.lens, b.o, b.scores, b.workspace)
        else:
            P.caote_score(p, q, b.K, b.V, b.lens, b.base, b.o, b.scores, b.workspace)
        P.caote_select_evict(p, b.scores, b.lens, b.budget, b.pos, b.evict_idx, b.n_evict, b.workspace)
        if method == "post_evict":
            P.caote_post_evict_output_ws(p, q, b.K, b.V, b.lens, b.evict_idx, b.n_evict, b.o, b.o_post, b.workspace)
        P.caote_compact(p, b.K, b.V, b.base, b.pos, b.lens, b.evict_idx, b.n_evict, compact, b.workspace)
        torch.cuda.synchronize()
        assert a.status() == 0 and b.status() == 0
        for x in ("lens", "n_evict", "n_seen", "o") + (("o_post",) if method == "post_evict" else ()):
            assert torch.equal(getattr(a, x), getattr(b, x)), x
        for s in range(B):
            n = int(a.lens[s])
            assert n <= budget
            for x in ("K", "V", "pos", "scores"):
                assert torch.equal(getattr(a, x)[s, :, :n], getattr(b, x)[s, :, :n]), x
