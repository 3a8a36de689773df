"""GPU parity of greedy multi-token eviction (Appendix B chained) against the oracle's sequence.

The GPU's picks are followed in lock-step: as long as they agree with the oracle's greedy sequence nothing else
is needed; where they differ, the oracle scores the state the GPU was in (the tokens still present, weights
renormalised) and the GPU's pick must lie within the scoring tolerance of the oracle's minimum there; the
comparison then carries on from the GPU's state, so that one tolerated flip cannot cascade."""
import numpy as np
import pytest
import torch

import oracle
import paper_2504_14051_b200 as P

from parity import ATOL, RTOL, f32

pytestmark = pytest.mark.gpu
DEV = "cuda"


def follow(order_gpu, h, V, pos, k):
    """Returns the number of tolerated differences; raises on a pick outside the band."""
    n, d = V.shape
    remaining = list(range(n))
    t, flips = 0, 0
    while t < k:
        hr = h[remaining].astype(np.float64)
        o_order, _, _ = oracle.greedy_evict(hr / hr.sum(), V[remaining], k - t, pos[remaining])
        mapped = [remaining[i] for i in o_order]
        c = 0
        while c < k - t and mapped[c] == order_gpu[t + c]:
            c += 1
        if c == k - t:
            break
        gone = set(mapped[:c])
        rem2 = [j for j in remaining if j not in gone]
        r = oracle.score(np.zeros((1, 1, 1, d), np.float32), np.zeros((1, 1, len(rem2), d), np.float32), V[rem2][None, None],
                         np.array([len(rem2)], np.int32), scale=1.0, base_mode="external",
                         base=h[rem2][None, None].astype(np.float64))
        c_ref = r["scores"][0, 0]
        e = order_gpu[t + c]
        assert e in rem2, f"pick {t + c}: slot {e} was evicted before or is out of range"
        cmin = c_ref.min()
        assert abs(c_ref[rem2.index(e)] - cmin) <= ATOL + RTOL * abs(cmin), (
            f"pick {t + c}: GPU evicts slot {e} (oracle score {c_ref[rem2.index(e)]!r}) but the minimum is {cmin!r}")
        flips += 1
        remaining = [j for j in rem2 if j != e]
        t += c + 1
    return flips


@pytest.mark.parametrize("case", [
    # B, Hkv, d, cap, lens, k, dtype
    (2, 2, 128, 320, [300, 257], 2, torch.bfloat16),
    (2, 2, 128, 320, [300, 257], 8, torch.bfloat16),
    (1, 3, 64, 100, [97], 40, torch.float32),
    (1, 2, 128, 1300, [1280], 128, torch.bfloat16),     # a reduced prompt block: 1152 kept + 128 new, evict 128
    (1, 1, 128, 40, [33], 32, torch.bfloat16),          # down to a single token
    (2, 3, 128, 2104, [2000, 777], 64, torch.bfloat16), # the cluster kernel; the short sequence leaves most CTAs of its clusters without rows
    (1, 2, 128, 6160, [6150], 24, torch.bfloat16),      # the cluster kernel with several hundred rows per CTA
    (1, 2, 128, 13000, [12900], 24, torch.bfloat16),    # more rows than 16 CTAs hold in shared memory: the rest from L2
])
def test_greedy_sequence_follows_the_oracle(case):
    B, Hkv, d, cap, lens, k, dtype = case
    g = torch.Generator(device="cpu").manual_seed(k * 7 + d)
    V = torch.randn((B, Hkv, cap, d), generator=g).to(dtype)
    h = (torch.rand((B, Hkv, cap), generator=g) ** 3 + 1e-3).float()
    pos = torch.stack([torch.stack([torch.randperm(cap, generator=g) for _ in range(Hkv)]) for _ in range(B)]).to(torch.int32)
    lens_t = torch.tensor(lens, dtype=torch.int32)
    budget = lens_t - k
    p = P.make_params(B, Hkv, Hkv, d, cap, 1, dtype, 1.0, "external")
    ws = P.alloc_workspace(p, DEV)
    ev = torch.full((B, Hkv, k), -1, dtype=torch.int32, device=DEV)
    order = torch.full((B, Hkv, k), -1, dtype=torch.int32, device=DEV)
    ne = torch.zeros((B,), dtype=torch.int32, device=DEV)
    P.caote_trace_enable(True)
    P.caote_select_evict_greedy(p, V.to(DEV), h.to(DEV), lens_t.to(DEV), budget.to(DEV), pos.to(DEV), ev, order, ne, ws)
    torch.cuda.synchronize()
    trace = P.caote_trace_collect()
    P.caote_trace_enable(False)
    assert P.caote_read_status(ws) == 0
    assert ne.cpu().tolist() == [k] * B
    if dtype == torch.bfloat16 and d == 128 and cap >= 1300:
        # long units with many picks: the kernel that keeps the value rows in the shared memory of a cluster
        assert "greedy_cluster_kernel" in trace, trace
    Vn, hn, pn = f32(V), h.numpy(), pos.numpy()
    flips = 0
    for b in range(B):
        n = lens[b]
        for hd in range(Hkv):
            og = order[b, hd].cpu().numpy().tolist()
            assert len(set(og)) == k and all(0 <= j < n for j in og)
            assert ev[b, hd].cpu().numpy().tolist() == sorted(og)
            flips += follow(og, hn[b, hd, :n], Vn[b, hd, :n], pn[b, hd, :n], k)
    assert flips <= max(1, (B * Hkv * k) // 20), f"{flips} tolerated differences: too many to be rounding"
    # a second run gives the same sequence
    order2 = torch.full_like(order, -1)
    P.caote_select_evict_greedy(p, V.to(DEV), h.to(DEV), lens_t.to(DEV), budget.to(DEV), pos.to(DEV), ev, order2, ne, ws)
    assert torch.equal(order, order2)


def test_one_greedy_pick_is_the_plain_selection_and_k0_evicts_nothing():
    B, Hkv, d, cap, n = 2, 2, 128, 700, 650
    g = torch.Generator(device="cpu").manual_seed(5)
    q = torch.randn((B, Hkv, 1, d), generator=g).to(torch.bfloat16).to(DEV)
    K = torch.randn((B, Hkv, cap, d), generator=g).to(torch.bfloat16).to(DEV)
    V = torch.randn((B, Hkv, cap, d), generator=g).to(torch.bfloat16).to(DEV)
    h = torch.rand((B, Hkv, cap), generator=g).to(DEV)
    lens = torch.tensor([n, n - 30], dtype=torch.int32, device=DEV)
    p = P.make_params(B, Hkv, Hkv, d, cap, 1, torch.bfloat16, d ** -0.5, "external")
    ws = P.alloc_workspace(p, DEV)
    o = torch.zeros((B, Hkv, 1, d), device=DEV)
    scores = torch.zeros((B, Hkv, cap), device=DEV)
    P.caote_score(p, q, K, V, lens, h, o, scores, ws)
    ev1 = torch.full((B, Hkv, 1), -1, dtype=torch.int32, device=DEV)
    ev2 = torch.full((B, Hkv, 1), -1, dtype=torch.int32, device=DEV)
    ne1 = torch.zeros((B,), dtype=torch.int32, device=DEV)
    ne2 = torch.zeros((B,), dtype=torch.int32, device=DEV)
    budget = lens - 1
    P.caote_select_evict(p, scores, lens, budget, None, ev1, ne1, ws)
    P.caote_select_evict_greedy(p, V, h, lens, budget, None, ev2, None, ne2, ws)
    sc = scores.cpu().numpy()
    for b in range(B):
        for hd in range(Hkv):
            a, c = int(ev1[b, hd, 0]), int(ev2[b, hd, 0])
            assert a == c or abs(sc[b, hd, a] - sc[b, hd, c]) <= ATOL + RTOL * sc[b, hd, a]
    assert ne1.tolist() == ne2.tolist() == [1, 1]
    P.caote_select_evict_greedy(p, V, h, lens, lens.clone(), None, ev2, None, ne2, ws)
    assert ne2.tolist() == [0, 0] and P.caote_read_status(ws) == 0


@pytest.mark.parametrize("case", [
    # n, k, weights: what makes the bounds of the pruned search fail or tie
    (700, 300, "equal"),      # equal weights: every pick moves the output by as much as the scores differ
    (3000, 40, "zeros"),      # most weights zero: their scores tie at 0, the position decides
    (2600, 60, "same_rows"),  # equal weights and equal rows: all scores tie
    (900, 890, "heavy"),      # two tokens hold nearly all the weight, picks go on until little else is left
    (4500, 1600, "tail"),     # more picks than one search of candidates covers
])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.float32, 64)])
def test_greedy_when_bounds_are_loose_or_tie(case, dtype, d):
    n, k, kind = case
    g = torch.Generator(device="cpu").manual_seed(n + k)
    cap = n + 5
    V = torch.randn((1, 1, cap, d), generator=g).to(dtype)
    h = (torch.rand((1, 1, cap), generator=g) + 0.1).float()
    if kind in ("equal", "same_rows"):
        h[:] = 0.5
    if kind == "same_rows":
        V[:] = V[:, :, :1].clone()
    if kind == "zeros":
        h[:, :, torch.randperm(n, generator=g)[:n - 200]] = 0.0
    if kind == "heavy":
        h[:, :, 10], h[:, :, 700] = 3e3, 5e3
    if kind == "tail":
        h = torch.randn((1, 1, cap), generator=g).exp()
    pos = torch.randperm(cap, generator=g).to(torch.int32).view(1, 1, cap)
    p = P.make_params(1, 1, 1, d, cap, 1, dtype, 1.0, "external")
    ws = P.alloc_workspace(p, DEV)
    ev = torch.full((1, 1, k), -1, dtype=torch.int32, device=DEV)
    order, ne = torch.full_like(ev, -1), torch.zeros((1,), dtype=torch.int32, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32)
    P.caote_select_evict_greedy(p, V.to(DEV), h.to(DEV), lens.to(DEV), (lens - k).to(DEV), pos.to(DEV), ev, order, ne, ws)
    assert P.caote_read_status(ws) == 0 and ne.item() == k
    og = order[0, 0].cpu().tolist()
    assert sorted(og) == ev[0, 0].cpu().tolist() and len(set(og)) == k and 0 <= min(og) and max(og) < n
    if kind == "zeros":  # exact ties: smallest position first, no band
        assert og == sorted([j for j in range(n) if h[0, 0, j] == 0], key=lambda j: int(pos[0, 0, j]))[:k]
    if kind in ("zeros", "same_rows"):
        return  # (same rows: every distance is the rounding of X alone, any order is right)
    # the first picks in lock-step with the oracle, in its band (the whole sequence costs minutes on the host)
    follow(og[:24], h[0, 0, :n].numpy(), f32(V)[0, 0, :n], pos[0, 0, :n].numpy(), 24)
    if k > 200:  # ... and picks late in the sequence, from the state the first ones leave
        gone = set(og[:k - 12])
        rem = [j for j in range(n) if j not in gone]
        hr, Vr, pr = h[0, 0, rem].numpy(), f32(V)[0, 0][rem], pos[0, 0, rem].numpy()
        follow([rem.index(j) for j in og[k - 12:]], hr, Vr, pr, 12)


@pytest.mark.parametrize("n,k", [(2, 1), (9, 8), (191, 190), (193, 64), (255, 40), (257, 225), (330, 329)])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128)])
def test_greedy_around_the_length_of_the_list_of_active_tokens(n, k, dtype, d):
    """192 are asked for and 256 fit; a fifth of the weights is 0, tokens without a bound."""
    g = torch.Generator(device="cpu").manual_seed(n * 31 + k)
    cap = n + 3
    V = torch.randn((1, 1, cap, d), generator=g).to(dtype)
    h = torch.randn((1, 1, cap), generator=g).exp()
    none = torch.randperm(n, generator=g)[:n // 5]
    h[:, :, none] = 0.0
    pos = torch.randperm(cap, generator=g).to(torch.int32).view(1, 1, cap)
    p = P.make_params(1, 1, 1, d, cap, 1, dtype, 1.0, "external")
    ws = P.alloc_workspace(p, DEV)
    ev = torch.full((1, 1, k), -1, dtype=torch.int32, device=DEV)
    order, ne = torch.full_like(ev, -1), torch.zeros((1,), dtype=torch.int32, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32)
    P.caote_select_evict_greedy(p, V.to(DEV), h.to(DEV), lens.to(DEV), (lens - k).to(DEV), pos.to(DEV), ev, order, ne, ws)
    assert P.caote_read_status(ws) == 0 and ne.item() == k
    og = order[0, 0].cpu().tolist()
    assert sorted(og) == ev[0, 0].cpu().tolist() and len(set(og)) == k and 0 <= min(og) and max(og) < n
    first = sorted(none.tolist(), key=lambda j: int(pos[0, 0, j]))[:k]
    assert og[:len(first)] == first  # scores of exactly 0: the oldest first
    rem = [j for j in range(n) if j not in set(first)]
    more = [rem.index(j) for j in og[len(first):]][:24]
    if more:
        follow(more, h[0, 0, rem].numpy(), f32(V)[0, 0][rem], pos[0, 0, rem].numpy(), len(more))


@pytest.mark.parametrize("kind,k", [("far_light_token", 1), ("far_light_token", 40), ("nan_light_token", 40), ("infinite_weight", 40),
                                    ("sum_overflows", 40), ("sum_overflows", 300)])
def test_greedy_scores_of_exactly_0_come_first_whatever_the_distance(kind, k):
    """w / (1 - w) of 0 scores 0, also where the distance overflows, is no number or X is none; equal scores: the oldest first."""
    n, d = 600, 128
    g = torch.Generator(device="cpu").manual_seed(k)
    V = torch.randn((1, 1, n, d), generator=g)
    h = torch.rand((1, 1, n), generator=g) + 0.5
    pos = torch.randperm(n, generator=g).to(torch.int32).view(1, 1, n)
    if kind.endswith("light_token"):  # the smallest positive weight over a sum of about 600: 0
        light = [9] if k == 1 else list(range(9, 9 + k))
        V[0, 0, light, 3] = 1e20 if kind == "far_light_token" else float("nan")
        h[0, 0, light] = 1e-45
    elif kind == "infinite_weight":  # (the heavy token itself has the largest score)
        light = [j for j in range(n) if j != 7]
        h[0, 0, 7] = float("inf")
    else:
        light = list(range(n))
        h *= 1e37
    p = P.make_params(1, 1, 1, d, n, 1, torch.float32, 1.0, "external")
    ws = P.alloc_workspace(p, DEV)
    ev = torch.full((1, 1, k), -1, dtype=torch.int32, device=DEV)
    order, ne = torch.full_like(ev, -1), torch.zeros((1,), dtype=torch.int32, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32)
    P.caote_select_evict_greedy(p, V.to(DEV), h.to(DEV), lens.to(DEV), (lens - k).to(DEV), pos.to(DEV), ev, order, ne, ws)
    assert P.caote_read_status(ws) == 0 and ne.item() == k
    og = order[0, 0].cpu().tolist()
    assert og == sorted(light, key=lambda j: int(pos[0, 0, j]))[:k]
    assert ev[0, 0].cpu().tolist() == sorted(og)


def few_rows(n, k, kind, dtype, d, seed, distinct=64):
    """A greedy eviction from n tokens whose value rows are `distinct` different ones; weights equal, log-normal or half of them subnormal."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    which = torch.randint(0, distinct, (n,), generator=g)
    V = torch.randn((distinct, d), generator=g).to(dtype)[which].view(1, 1, n, d).contiguous()
    h = torch.full((1, 1, n), 0.5) if kind == "equal" else torch.randn((1, 1, n), generator=g).exp()
    if kind == "subnormal":
        h = torch.where(torch.rand((1, 1, n), generator=g) < 0.5, (which % 7 + 3).view(1, 1, n) * 1e-42, h)
    pos = torch.randperm(n, generator=g).to(torch.int32).view(1, 1, n)
    p = P.make_params(1, 1, 1, d, n, 1, dtype, 1.0, "external")
    ws = P.alloc_workspace(p, DEV)
    ev = torch.full((1, 1, k), -1, dtype=torch.int32, device=DEV)
    order, ne = torch.full_like(ev, -1), torch.zeros((1,), dtype=torch.int32, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32)
    args = (p, V.to(DEV), h.to(DEV), lens.to(DEV), (lens - k).to(DEV), pos.to(DEV), ev, order, ne, ws)
    return which.tolist(), h[0, 0], f32(V)[0, 0], pos[0, 0], args


@pytest.mark.parametrize("n,k,kind", [(300, 299, "equal"), (4224, 96, "equal"), (700, 400, "subnormal"), (20000, 40, "equal")])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128)])
def test_greedy_when_many_tokens_compete_for_every_pick(n, k, kind, dtype, d):
    """All warps form scores, to the bit those of one warp: tokens of the same row and weight leave in the order of their positions."""
    which, h, V, pos, args = few_rows(n, k, kind, dtype, d, n + d)
    P.caote_select_evict_greedy(*args)
    assert P.caote_read_status(args[-1]) == 0
    og = args[7][0, 0].cpu().tolist()
    assert sorted(og) == args[6][0, 0].cpu().tolist() and len(set(og)) == k and 0 <= min(og) and max(og) < n
    same = {}
    for j in sorted(range(n), key=lambda j: int(pos[j])):
        same.setdefault((which[j], float(h[j])), []).append(j)
    for t, j in enumerate(og):
        oldest = same[which[j], float(h[j])].pop(0)
        assert j == oldest, f"pick {t}: slot {j} leaves before slot {oldest}, an older one of the same row and weight"
    if kind == "equal":
        follow(og[:12], h.numpy(), V, pos.numpy(), 12)


def test_greedy_cost_of_tokens_that_compete():
    """Equal weights and few different rows cost more builds and shared scores, not a walk through the list for every pick: at 4 224
    tokens and 128 picks 7 times the time of log-normal weights and different rows (51 times with the walk)."""
    def device_ms(distinct, kind):
        args = few_rows(4224, 128, kind, torch.bfloat16, 128, 2, distinct)[-1]
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            P.caote_select_evict_greedy(*args)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[2]
    assert device_ms(64, "equal") < 20 * device_ms(4224, "log-normal")
