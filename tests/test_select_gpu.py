"""Selection of several tokens per unit at the sizes where the kernel changes its ways: scores in registers (up to 8 or 24 per
thread of 1024) or read again in every pass, thresholds that fall into ties, score ranges of one bit to all bits."""
import numpy as np
import pytest
import torch

import oracle
import paper_2504_14051_b200 as P

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("kind", ["narrow", "wide", "ties", "few_ties", "equal"])
@pytest.mark.parametrize("n,k", [(3, 2), (1024, 1023), (8192, 37), (8193, 512), (24576, 2), (24577, 300)])
def test_several_smallest_are_bit_exact(n, k, kind):
    g = torch.Generator().manual_seed(n + k)
    if kind == "narrow":  # one binade: the leading bits are the same everywhere
        s = 1.0 + torch.rand((1, 2, n), generator=g) * 1e-3
    elif kind == "wide":  # zeros, denormals, infinities
        s = torch.exp(torch.randn((1, 2, n), generator=g) * 30)
        s[0, 0, ::7], s[0, 1, ::5] = 0.0, float("inf")
    elif kind == "ties":  # thousands of each value
        s = torch.randint(0, 6, (1, 2, n), generator=g).float()
    elif kind == "few_ties":  # up to a few hundred of each
        s = torch.randint(0, max(n // 60, 2), (1, 2, n), generator=g).float()
    else:
        s = torch.full((1, 2, n), 0.25)
    pos = torch.stack([torch.randperm(n, generator=g) for _ in range(2)]).view(1, 2, n).to(torch.int32)
    p = P.make_params(1, 2, 2, 64, n, 1, torch.float32, 1.0, "last_query")
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32)
    for use_pos in (True, False):
        ev, ne = torch.full((1, 2, k), -1, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
        P.caote_select_evict(p, s.to(DEV), lens.to(DEV), (lens - k).to(DEV), pos.to(DEV) if use_pos else None, ev, ne, ws)
        ref, _ = oracle.select_evict(s.numpy(), [n], [n - k], pos.numpy() if use_pos else None)
        assert ne.item() == k
        for h in range(2):
            assert ev[0, h].cpu().tolist() == ref[0][h].tolist()


@pytest.mark.parametrize("kind", ["any_bits", "mostly_all_ones", "any_positions"])
@pytest.mark.parametrize("n,k", [(200, 150), (3000, 2500), (9000, 100), (25000, 24000)])
def test_order_is_that_of_the_bits(n, k, kind):
    """A caller's own scores and positions may have any bits (signs, NaNs, all ones): the order is that of the unsigned 64-bit
    keys (score bits, position)."""
    g = np.random.default_rng(n)
    bits, pos = g.integers(0, 2 ** 32, n, dtype=np.uint32), g.permutation(n).astype(np.uint32)
    if kind == "mostly_all_ones":
        bits[g.random(n) < 0.75] = 0xFFFFFFFF
    if kind == "any_positions":
        bits[:] = 0x3F800000
        pos = np.unique(g.integers(0, 2 ** 32, 2 * n, dtype=np.uint32))[-n:]  # (the largest, 0xffffffff among them)
        pos[-1] = 0xFFFFFFFF
        g.shuffle(pos)
    want = np.sort(np.argsort((bits.astype(np.uint64) << np.uint64(32)) | pos.astype(np.uint64))[:k])
    p = P.make_params(1, 1, 1, 64, n, 1, torch.float32, 1.0, "last_query")
    ev, ne = torch.full((1, 1, k), -1, dtype=torch.int32, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    lens = torch.tensor([n], dtype=torch.int32, device=DEV)
    P.caote_select_evict(p, torch.from_numpy(bits.view(np.float32)).to(DEV).view(1, 1, n), lens, lens - k,
                         torch.from_numpy(pos.view(np.int32)).to(DEV).view(1, 1, n), ev, ne, torch.zeros(256, dtype=torch.uint8, device=DEV))
    assert ne.item() == k and ev[0, 0].tolist() == want.tolist()
