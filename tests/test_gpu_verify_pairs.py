"""The verifier's two pairs to a word, against the oracle: lengths that differ
within a word and end at every column of eight, odd counts, thresholds up to its
limit and just above it, refused pairs beside valid ones, and a large grouped
batch whose chunks mix both widths."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_sliced import ragged

pytestmark = pytest.mark.gpu
LENS = [0, 1, 7, 8, 9, 15, 16, 17, 24, 31, 32, 33, 63, 64, 65, 100, 127, 128, 150]


@pytest.fixture(scope="module")
def pf():
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as m
    return m


def packed(pf, ctx, P):
    reads, refs = (torch.from_numpy(np.append(x, np.uint8(65))).cuda() for x in (P.reads, P.refs))
    return pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off)


@pytest.mark.parametrize("n", [1, 31, 33, 63, 65, 700])
@pytest.mark.parametrize("E_max", [0, 1, 3, 6, 7, 8])
def test_small_bands(pf, n, E_max):
    rng = np.random.default_rng(100 * n + E_max)
    lens = rng.choice(LENS, size=n)
    ctx = pf.pf_create(0)
    try:
        for E in (np.full(n, E_max), rng.integers(0, E_max + 1, size=n)):
            P = ragged(n + E_max, lens, E)
            pairs, want = packed(pf, ctx, P), oracle.verify_batch(P)
            ld, Ed = torch.from_numpy(P.lens).cuda(), torch.from_numpy(P.E).cuda()
            d = torch.full((n,), 77, dtype=torch.int32, device="cuda")
            one = bool((E == E_max).all())
            pf.pf_verify(ctx, pairs, ld, None if one else Ed, E_max, None, None, d)
            pf.pf_sync(ctx)
            assert np.array_equal(d.cpu().numpy(), want)
            # an index list in reverse, every other pair
            idx = torch.arange(n - 1, -1, -2, device="cuda")
            cnt = torch.tensor([len(idx)], device="cuda")
            d.fill_(77)
            pf.pf_verify(ctx, pairs, ld, Ed, E_max, idx, cnt, d)
            pf.pf_sync(ctx)
            sel = idx.cpu().numpy()
            exp = np.full(n, 77)
            exp[sel] = want[sel]
            assert np.array_equal(d.cpu().numpy(), exp)
            # refused pairs leave the other half of their word alone
            at = np.arange(0, n, 5)
            Ed[torch.from_numpy(at).cuda()] = E_max + 1
            ld[n // 2] = -3
            pf.pf_verify(ctx, pairs, ld, Ed, E_max, None, None, d)
            with pytest.raises(pf.PFError):
                pf.pf_sync(ctx)
            exp = want.copy()
            exp[at] = -1
            exp[n // 2] = -1
            assert np.array_equal(d.cpu().numpy(), exp)
    finally:
        pf.pf_destroy(ctx)


@pytest.mark.parametrize("E_max", [12, 25])
def test_large_grouped_batch(pf, E_max):
    """Enough pairs to verify that the warps take 64 at a time, thresholds on
    both sides of the limit."""
    m, n = 4000, 3_000_000
    rng = np.random.default_rng(E_max)
    E = rng.choice([0, 3, 7, 8, E_max], size=m, p=[0.1, 0.3, 0.4, 0.1, 0.1])
    P = ragged(E_max, rng.choice([16, 33, 64, 100], size=m), E, kmax=6)
    ctx = pf.pf_create(0)
    try:
        pairs, want = packed(pf, ctx, P), oracle.verify_batch(P)
        oa, _ = oracle.filter_batch(P)
        rep = np.arange(n) % m
        rd = torch.from_numpy(rep).cuda()
        pairs.read.word_off = pairs.ref.word_off = pairs.read.word_off[rd].contiguous()
        ld, Ed = torch.from_numpy(P.lens).cuda()[rd], torch.from_numpy(P.E).cuda()[rd]
        pf.pf_set_resolve_by_bounds(ctx, False)
        acc = torch.empty(n, dtype=torch.uint8, device="cuda")
        cnt = torch.empty(n, dtype=torch.int16, device="cuda")
        dist = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        pf.pf_filter_verify(ctx, pf.PF_SNEAKYSNAKE, pairs, ld, Ed, E_max, acc, cnt, dist, n)
        pf.pf_sync(ctx)
        assert int(acc.sum()) >= 64 * 8 * 3 * 152   # what the wide chunks ask for
        exp = np.where(oa[0], want, P.E + 1)[rep]
        assert np.array_equal(dist.cpu().numpy(), exp)
    finally:
        pf.pf_destroy(ctx)
