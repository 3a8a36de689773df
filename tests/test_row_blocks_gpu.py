"""The tensor-core row-block kernels on the shapes between the single-query kernels and long blocks of a prompt: any base
mode, head_dim 64, groups of more than 8, blocks of a few queries."""
import pytest
import torch

import oracle
import paper_2504_14051_b200 as P

from test_gpu_parity import dominant_case, make_case, run_score
from parity import assert_close, check_scores_and_o, f32, oracle_for, sub_problem

pytestmark = pytest.mark.gpu
DEV = "cuda"

# B, Hq, Hkv, d, cap, m, lens: lengths at the edges of key tiles (128) and key-tile pairs (256), of the key splits, and
# of the block itself; counted rows around the 64 below which the complements are kept apart
SHAPES = [
    (2, 16, 1, 128, 300, 1, [128, 129]),        # one query, 16 heads per group
    (3, 4, 1, 64, 1040, 1, [1, 256, 1025]),     # one query, head_dim 64, a single token
    (1, 8, 1, 128, 2064, 1, [2049]),            # one query, 8 heads and (accum, external) carried scores
    (2, 14, 2, 128, 272, 9, [9, 257]),          # 63 rows, a sequence that is nothing but its block
    (1, 8, 1, 64, 1600, 8, [1537]),             # 64 rows
    (1, 2, 1, 128, 4112, 128, [4097]),          # key splits, two row blocks
    (2, 16, 1, 64, 4112, 2, [4096, 130]),       # key splits for one of two sequences
    # one query at head_dim 64: the cluster kernel with many units per cluster, with nine tiles per CTA on its largest
    # cluster, and one tile more than that holds
    (40, 14, 2, 64, 1300, 1, [1300 - 37 * (i % 9) for i in range(40)]),
    (1, 8, 1, 64, 18432, 1, [18432]),
    (1, 4, 1, 64, 18448, 1, [18433]),
]


@pytest.mark.parametrize("mode", ["last_query", "chunk_sum", "accum", "external"])
@pytest.mark.parametrize("shape", SHAPES)
def test_row_block_scores_match_oracle(shape, mode):
    B, Hq, Hkv, d, cap, m, lens = shape
    q, K, V, lens_t = make_case(900 + SHAPES.index(shape), B, Hq, Hkv, d, cap, m, torch.bfloat16, lens)
    base = None
    if mode in ("accum", "external"):
        base = (torch.rand((B, Hkv, cap), generator=torch.Generator().manual_seed(6)) * 2.0).to(DEV)
    base_in = None if base is None else base.clone()
    _, _, o, scores = run_score(q, K, V, lens_t, m, mode, base)
    r = oracle_for(q, K, V, lens_t, scale=d ** -0.5, n_new=m, base_mode=mode, base=base_in)
    check_scores_and_o(r, scores, o, lens_t, f"{shape} {mode}")
    if mode == "accum":
        for b, n in enumerate(lens):
            assert_close(f32(base)[b, :, :n], r["base"][b, :, :n], "accumulated base", rtol=1e-5, atol=1e-6)
            assert torch.equal(base[b, :, n:], base_in[b, :, n:])
    if mode == "external":
        assert torch.equal(base, base_in)


# the any-shape fp32 kernels: rows at the edges of their tiles of 16 and, from 40 on, 64 rows; keys at those of 64
FP32_SHAPES = [
    (2, 3, 1, 128, 208, 13, [193, 13]),     # 39 rows
    (2, 5, 1, 64, 272, 8, [257, 8]),        # 40
    (1, 2, 2, 128, 528, 64, [513]),         # 64
    (2, 5, 1, 128, 400, 13, [320, 64]),     # 65
    (1, 2, 1, 64, 1104, 65, [1089]),        # 130
]


@pytest.mark.parametrize("mode", ["last_query", "chunk_sum", "accum", "external"])
@pytest.mark.parametrize("shape", FP32_SHAPES)
def test_fp32_row_tiles_match_oracle(shape, mode):
    B, Hq, Hkv, d, cap, m, lens = shape
    q, K, V, lens_t = make_case(970 + FP32_SHAPES.index(shape), B, Hq, Hkv, d, cap, m, torch.float32, lens)
    base = None
    if mode in ("accum", "external"):
        base = (torch.rand((B, Hkv, cap), generator=torch.Generator().manual_seed(6)) * 2.0).to(DEV)
    base_in = None if base is None else base.clone()
    _, _, o, scores = run_score(q, K, V, lens_t, m, mode, base)
    r = oracle_for(q, K, V, lens_t, scale=d ** -0.5, n_new=m, base_mode=mode, base=base_in)
    check_scores_and_o(r, scores, o, lens_t, f"{shape} {mode}")


@pytest.mark.parametrize("eps", [1e-1, 1e-2, 1e-3])
@pytest.mark.parametrize("shape", [
    (1, 16, 1, 128, 700, 1, [640], "last_query"),      # one row block
    (1, 8, 2, 64, 5000, 1, [4900], "accum"),           # the planted token in one of several key splits
    (2, 8, 2, 128, 2100, 128, [2048, 700], "last_query"),  # the counted rows of a long block
    (1, 7, 1, 128, 300, 9, [290], "chunk_sum"),        # 63 rows
])
def test_few_rows_that_agree_on_one_token(shape, eps):
    """One token holds all but ~eps of every counted row's weight: the complement is the others' sum, not a difference
    (tolerance as everywhere: at eps 1e-3 a difference of fp32 weights would lose it)."""
    B, Hq, Hkv, d, cap, m, lens, mode = shape
    q, K, V, lens_t = dominant_case(17 + Hq, B, Hq, Hkv, d, cap, m, torch.bfloat16, lens, eps, 77)
    base = None
    if mode == "accum":
        base = (torch.rand((B, Hkv, cap), generator=torch.Generator().manual_seed(3)) * 1e-9).to(DEV)
    base_in = None if base is None else base.clone()
    _, _, o, scores = run_score(q, K, V, lens_t, m, mode, base)
    r = oracle_for(q, K, V, lens_t, scale=d ** -0.5, n_new=m, base_mode=mode, base=base_in)
    assert ((1.0 - r["w"][:, :, 77]) < 8 * eps).all()
    check_scores_and_o(r, scores, o, lens_t, f"{shape} eps {eps}")


@pytest.mark.parametrize("case", [
    # B, Hq, Hkv, d, cap, m, lens, budget, mode: evictions at the edges of a tile of 128 evicted rows, sequences that
    # evict nothing or nearly everything, ragged row blocks
    (2, 8, 2, 128, 500, 64, [500, 300], [372, 300], "last_query"),
    (2, 4, 2, 64, 700, 33, [650, 600], [521, 473], "chunk_sum"),
    (1, 14, 2, 128, 900, 128, [896], [512], "chunk_sum"),
    (1, 6, 2, 64, 300, 100, [270], [13], "last_query"),
])
def test_corrected_output_of_query_blocks(case):
    B, Hq, Hkv, d, cap, m, lens, budget, mode = case
    q, K, V, lens_t = make_case(41 + m, B, Hq, Hkv, d, cap, m, torch.bfloat16, lens)
    p, ws, o, scores = run_score(q, K, V, lens_t, m, mode)
    ev = torch.zeros((B, Hkv, max(n - k for n, k in zip(lens, budget))), dtype=torch.int32, device=DEV)
    ne = torch.zeros((B,), dtype=torch.int32, device=DEV)
    P.caote_select_evict(p, scores, lens_t, torch.tensor(budget, dtype=torch.int32, device=DEV), None, ev, ne, ws)
    o_post = torch.full_like(o, float("nan"))
    P.caote_post_evict_output_ws(p, q, K, V, lens_t, ev, ne, o, o_post, ws)
    assert P.caote_read_status(ws) == 0
    evc, nec = ev.cpu().numpy(), ne.cpu().numpy()
    ref = oracle.post_evict_output(f32(q), f32(K), f32(V), lens, [[evc[b, h, :nec[b]] for h in range(Hkv)] for b in range(B)],
                                   scale=d ** -0.5, n_new=m)
    # o and the evicted share both carry P's 16 bits (8e-6 of the largest value, about 4); what is left over after the
    # subtraction is divided by the retained weight, 0.04 at the least here (13 of 270 tokens kept)
    assert_close(f32(o_post), ref, f"{case}", atol=2e-3 if budget[0] * 4 < lens[0] else 2e-4)


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.float32, 128), (torch.bfloat16, 64)])
@pytest.mark.parametrize("n,first,k", [(4100, 0, 1), (4100, 3000, 2), (3071, 5, 2500), (1025, 1024, 1)])
def test_stable_compaction_over_several_rounds(n, first, k, dtype, d):
    """More slots than a round of the cluster's tiles holds (512 at the least, 2048 at the most), the first evicted slot at
    either end, and more picks than shared memory keeps."""
    g = torch.Generator().manual_seed(n + first)
    B, Hkv, cap = 1, 2, n + 7
    K, V = (torch.randn((B, Hkv, cap, d), generator=g).to(dtype).to(DEV) for _ in range(2))
    base, pos = torch.rand((B, Hkv, cap), generator=g).to(DEV), torch.arange(cap, dtype=torch.int32, device=DEV).expand(B, Hkv, cap).contiguous()
    ev = torch.stack([torch.cat([torch.tensor([first]), first + 1 + torch.randperm(n - first - 1, generator=g)[:k - 1].sort().values])
                      for _ in range(Hkv)]).to(torch.int32).view(B, Hkv, k)
    lens = torch.tensor([n], dtype=torch.int32, device=DEV)
    p = P.make_params(B, Hkv, Hkv, d, cap, 1, dtype, 1.0, "last_query")
    K0, V0, b0 = K.clone(), V.clone(), base.clone()
    P.caote_compact(p, K, V, base, pos, lens, ev.to(DEV), torch.tensor([k], dtype=torch.int32, device=DEV), "stable", P.alloc_workspace(p, DEV))
    assert lens.item() == n - k
    for h in range(Hkv):
        keep = torch.ones(n, dtype=torch.bool)
        keep[ev[0, h].long()] = False
        idx = keep.nonzero().flatten().to(DEV)
        assert torch.equal(pos[0, h, :n - k].long(), idx)
        assert torch.equal(K[0, h, :n - k], K0[0, h, idx]) and torch.equal(V[0, h, :n - k], V0[0, h, idx])
        assert torch.equal(base[0, h, :n - k], b0[0, h, idx])
        assert torch.equal(K[0, h, n:], K0[0, h, n:]) and torch.equal(V[0, h, n:], V0[0, h, n:])


@pytest.mark.parametrize("mode", ["fill", "stable"])
@pytest.mark.parametrize("Hkv", [1, 3, 8, 9])
def test_compaction_leaves_its_workspace_alone(Hkv, mode):
    """caote_compact takes any 256 bytes: not zeroed ones, and ones that a call on another stream is using."""
    B, d, cap, n, k = 3, 64, 300, 290, 2
    p = P.make_params(B, Hkv, Hkv, d, cap, 1, torch.bfloat16, 1.0, "last_query")
    ws = torch.full((256,), 0xA5, dtype=torch.uint8, device=DEV)
    ev = torch.tensor([3, 77], dtype=torch.int32, device=DEV).expand(B, Hkv, k).contiguous()
    ne = torch.tensor([2, 0, 1], dtype=torch.int32, device=DEV)
    caches, streams = [], [torch.cuda.Stream() for _ in range(2)]
    for _ in streams:
        K, V = (torch.randn((B, Hkv, cap, d), device=DEV).to(torch.bfloat16) for _ in range(2))
        pos = torch.arange(cap, dtype=torch.int32, device=DEV).expand(B, Hkv, cap).contiguous()
        caches.append((K, V, pos, torch.full((B,), n, dtype=torch.int32, device=DEV)))
    torch.cuda.synchronize()
    for turn in range(2):
        for (K, V, pos, lens), st in zip(caches, streams):
            P.caote_compact(p, K, V, None, pos, lens, ev, ne, mode, ws, stream=st)
    torch.cuda.synchronize()
    for _, _, pos, lens in caches:
        assert lens.tolist() == [n - 4, n, n - 2]
        for h in range(Hkv):
            for b, gone in ((0, {3, 77}), (1, set()), (2, {3})):
                left = pos[b, h, :lens[b]].tolist()
                assert len(set(left)) == len(left) and set(left) <= set(range(n)) - gone
    assert (ws == 0xA5).all()


@pytest.mark.parametrize("eps", [3e-1, 1e-2, 1e-3, 1e-4])  # (above and below the share from which the kernel for them scores it)
@pytest.mark.parametrize("case", [
    # B, Hq, Hkv, d, cap, m, lens, mode, carried scores
    (1, 8, 2, 128, 700, 64, [640], "accum", "zero"),         # one key split
    (2, 4, 2, 128, 2100, 128, [2048, 300], "accum", "sink"),  # the same token holds nearly all of the carried scores
    (1, 4, 2, 64, 2100, 128, [2048], "accum", "spread"),
    (1, 8, 2, 64, 700, 64, [640], "chunk_sum", None),
    (1, 8, 2, 128, 700, 128, [640], "chunk_sum", None),
    (1, 8, 2, 128, 700, 128, [640], "last_query", None),     # few counted rows
    (1, 16, 1, 128, 300, 1, [290], "accum", "sink"),         # one query
])
def test_token_that_holds_most_of_the_weight(case, eps):
    """One token holds all but ~eps of the weight of every row: neither 1 - w nor || X - v || may be a difference of nearly equal
    numbers (tolerance as everywhere; X from the tensor cores is 1e-6 off, 1e-2 of a distance of 1e-4)."""
    B, Hq, Hkv, d, cap, m, lens, mode, carried = case
    q, K, V, lens_t = dominant_case(31 + d + m, B, Hq, Hkv, d, cap, m, torch.bfloat16, lens, eps, 77)
    base = None
    if carried:
        base = torch.rand((B, Hkv, cap), generator=torch.Generator().manual_seed(3)) * (eps / cap if carried == "sink" else 1.0)
        if carried == "zero":
            base.zero_()
        if carried == "sink":
            base[:, :, 77] = 1.0
        base = (base * (m * Hq // Hkv if carried == "sink" else 1e-9)).to(DEV)
    base_in = None if base is None else base.clone()
    _, _, o, scores = run_score(q, K, V, lens_t, m, mode, base)
    r = oracle_for(q, K, V, lens_t, scale=d ** -0.5, n_new=m, base_mode=mode, base=base_in)
    assert ((1.0 - r["w"][:, :, 77]) < 8 * eps).all()
    check_scores_and_o(r, scores, o, lens_t, f"{case} eps {eps}")


def test_token_that_holds_most_of_the_weight_with_fast_scores():
    B, Hq, Hkv, d, cap, m, lens, eps = 1, 8, 2, 128, 700, 64, [640], 1e-4
    q, K, V, lens_t = dominant_case(8, B, Hq, Hkv, d, cap, m, torch.bfloat16, lens, eps, 77)
    p = P.make_params(B, Hq, Hkv, d, cap, m, torch.bfloat16, d ** -0.5, "chunk_sum")
    ws, vsum = P.alloc_workspace(p, DEV), torch.zeros((B, Hkv, d), device=DEV)
    o, scores = torch.zeros(q.shape, device=DEV), torch.zeros((B, Hkv, cap), device=DEV)
    P.caote_vsum(p, V, lens_t, vsum)
    P.caote_score_fast(p, q, K, V, lens_t, None, vsum, o, scores, ws)
    r = oracle_for(q, K, V, lens_t, scale=d ** -0.5, n_new=m, base_mode="chunk_sum")
    for h in range(Hkv):
        assert_close(f32(scores)[0, h, :lens[0]], oracle.fast_scores(r["w"][0, h, :lens[0]], f32(V)[0, h, :lens[0]]), f"[{h}]")


@pytest.mark.parametrize("d", [128, 64])
def test_carried_sums_beside_the_attention_pass(d):
    """Steps with accumulated scores whose launches overlap give the bits of steps whose launches are kept apart (by the
    events that tracing records between them): the sum over the carried scores starts before the attention pass is over."""
    B, Hq, Hkv, m, budget, steps = 2, 8, 4, 64, 4000, 5
    def run(apart):
        g = torch.Generator(device=DEV).manual_seed(4)
        rn = lambda *s: torch.randn(s, generator=g, device=DEV).to(torch.bfloat16)
        cache = P.EvictionCache(B, Hq, Hkv, d, budget + m, m, torch.bfloat16, budget, base_mode="accum")
        lens = torch.tensor([budget, budget - 30], dtype=torch.int32, device=DEV)
        cache.load(rn(B, Hkv, budget + m, d), rn(B, Hkv, budget + m, d), lens, base=torch.rand((B, Hkv, budget + m), generator=g, device=DEV))
        P.caote_trace_enable(apart)
        try:
            outs = [cache.step(rn(B, Hq, m, d), rn(B, Hkv, m, d), rn(B, Hkv, m, d)).clone() for _ in range(steps)]
            torch.cuda.synchronize()
        finally:
            P.caote_trace_enable(False)
            traced = P.caote_trace_collect()
        assert cache.status() == 0 and (not apart or traced["prefill_carried_sum_kernel"][0] == steps)
        return outs + [cache.base, cache.scores, cache.K, cache.V, cache.pos, cache.lens]
    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("mode", ["last_query", "chunk_sum", "accum"])
@pytest.mark.parametrize("case", [
    # B, Hq, Hkv, d, cap, m, n, key tiles per CTA
    (1, 1, 1, 128, 18448, 128, 18433, 19),  # 145 tiles in 8 splits; one counted row under last_query
    (1, 8, 1, 64, 18448, 16, 18433, 19),
    (1, 16, 1, 128, 18448, 1, 18433, 19),   # one query, 16 heads per group: few counted rows in every mode
    (38, 2, 2, 128, 2440, 128, 2400, 19),   # enough row blocks that none is split
    (38, 2, 2, 64, 2440, 128, 2400, 19),
])
def test_row_blocks_with_logits_that_grow_along_the_keys(case, mode):
    """Keys far above all that came before them in tiles 3, 8, 11, 16 and the last one of a CTA's share: the softmax reference
    moves before a share of the output is closed, on the tile that closes it, and with earlier shares set aside; for one row of
    a warp, for several, and for the counted rows. Two runs give the same bits."""
    B, Hq, Hkv, d, cap, m, n, tiles = case
    G = Hq // Hkv
    q, K, V, lens_t = make_case(60 + d + m, B, Hq, Hkv, d, cap, m, torch.bfloat16, [n] * B)
    units = [(0, 0)] if B == 1 else [(0, 1), (37, 0)]
    rows = [(0, 0), (G // 2, m // 2), (G - 1, m - 1)]  # head of the group, query: the last one is counted in every mode
    for b, h in units:
        for first in range(0, (n + 127) // 128, 3 * tiles):  # the first CTA's share, and every third
            for i, t in enumerate((3, 8, 11, 16, 18)):  # log2 of the weights: about 22 more from one to the next
                for g, r in (rows if i % 2 else rows[2:]):
                    j = (first + t) * 128 + 5 + 7 * g
                    if j < n - m:
                        K[b, h, j] = (q[b, h * G + g, r].float() * (1.3 * (i + 1) * (128 / d) ** 0.5)).to(K.dtype)
    base = None
    if mode == "accum":
        base = (torch.rand((B, Hkv, cap), generator=torch.Generator().manual_seed(6)) * 2.0).to(DEV)
    base_in = None if base is None else base.clone()
    _, _, o, scores = run_score(q, K, V, lens_t, m, mode, base)
    qs, Ks, Vs, ls, bs = sub_problem(q, K, V, lens_t, base_in, units, Hkv, G)
    r = oracle_for(qs, Ks, Vs, ls, scale=d ** -0.5, n_new=m, base_mode=mode, base=bs)
    check_scores_and_o(r, torch.stack([scores[b, h:h + 1] for b, h in units]), torch.stack([o[b, h * G:(h + 1) * G] for b, h in units]),
                       ls, f"{case} {mode}")
    base2 = None if base_in is None else base_in.clone()
    _, _, o2, scores2 = run_score(q, K, V, lens_t, m, mode, base2)
    assert torch.equal(o, o2) and torch.equal(scores[:, :, :n], scores2[:, :, :n])


@pytest.mark.parametrize("mode,d", [("chunk_sum", 64), ("accum", 64), ("chunk_sum", 128)])
def test_scores_of_many_equal_calls_have_the_same_bits(mode, d):
    """Value tiles are handed back to the copies only when every row has been read: 2 500 calls of eight items per CTA each."""
    B, Hq, Hkv, m, n = 7, 28, 4, 128, 10444
    g = torch.Generator(device=DEV).manual_seed(1)
    q, K, V = (torch.randn(s, generator=g, device=DEV).to(torch.bfloat16) for s in ((B, Hq, m, d), (B, Hkv, n, d), (B, Hkv, n, d)))
    base = torch.rand((B, Hkv, n), generator=g, device=DEV)
    lens = torch.full((B,), n, dtype=torch.int32, device=DEV)
    p = P.make_params(B, Hq, Hkv, d, n, m, torch.bfloat16, d ** -0.5, mode)
    ws = P.alloc_workspace(p, DEV)
    o, scores = torch.zeros(q.shape, device=DEV), torch.zeros((B, Hkv, n), device=DEV)
    first, differ, carried = None, torch.zeros((), dtype=torch.int64, device=DEV), torch.empty_like(base)
    for _ in range(2500 if (mode, d) == ("chunk_sum", 64) else 500):
        carried.copy_(base)
        P.caote_score(p, q, K, V, lens, carried if mode == "accum" else None, o, scores, ws)
        if first is None:
            first = scores.clone()
        differ += (scores != first).sum()
    assert differ.item() == 0 and P.caote_read_status(ws) == 0
