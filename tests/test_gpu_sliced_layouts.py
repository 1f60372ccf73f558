"""Bit-sliced kernels where the two sides of the pairs lie differently: one side
in strided rows, the other ragged with gaps, repeated or reversed, at sizes that
end inside a tile, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_sliced import ctx, pf, ragged  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
M, W = 150, 5
BASE = 1501          # different pairs


def offsets(kind, n):
    """First words of n sequences of W words; repeated: pairs p and p + BASE
    (the same sequences) share theirs."""
    p = np.arange(n, dtype=np.int64)
    if kind == "gaps":
        return np.cumsum(W + p % 3) - W
    if kind == "repeated":
        return (p % BASE) * W
    return (n - 1 - p) * W


def moved(pf, seqs, n, kind):
    """The strided rows of BASE sequences as n sequences, over and over, at
    offsets(kind), or as strided rows."""
    row = torch.arange(n, device=DEV) % BASE
    rows = [x.view(BASE, W)[row] for x in (seqs.lo, seqs.hi, seqs.nmask)]
    if kind == "strided":
        return pf.Seqs(*[x.reshape(-1).contiguous() for x in rows], stride_words=W)
    off = torch.from_numpy(offsets(kind, n)).to(DEV)
    at = (off[:, None] + torch.arange(W, device=DEV)).reshape(-1)
    out = []
    for x in rows:
        plane = torch.full((int(off.max()) + W,), -1, dtype=x.dtype, device=DEV)
        plane[at] = x.reshape(-1)
        out.append(plane)
    return pf.Seqs(*out, word_off=off)


def batch(pf, c, seed, n, E):
    """BASE pairs of M bases (threshold E), then n pairs repeating them."""
    P = ragged(seed, np.full(BASE, M), np.full(BASE, E))
    pairs = pf.pack_pairs(c, torch.from_numpy(P.reads).to(DEV), torch.from_numpy(P.refs).to(DEV),
                          length=M)
    return P, pairs, np.arange(n) % BASE


KINDS = [("strided", "gaps"), ("gaps", "strided"), ("strided", "repeated"),
         ("reversed", "strided"), ("gaps", "reversed")]


def run(pf, c, P, pairs, rep, E, per_pair):
    n = len(rep)
    oa, oc = oracle.filter_batch(P)
    want = np.where(oa[0] == 1, oracle.verify_batch(P), E + 1)
    wantg = np.where(oa[1] == 1, oracle.verify_batch(P), E + 1)
    lens = torch.full((n,), M, dtype=torch.int32, device=DEV)
    Ed = torch.full((n,), E, dtype=torch.int16, device=DEV) if per_pair else None
    for dec in (1, 2, 3):
        slots, rows = (2, [0, 1]) if dec == 3 else (1, [dec - 1])
        acc = torch.full((slots * n,), 9, dtype=torch.uint8, device=DEV)
        cnt = torch.full((slots * n,), 99, dtype=torch.int16, device=DEV)
        dist = torch.full((n,), -7, dtype=torch.int32, device=DEV)
        pf.pf_filter_verify(c, dec, pairs, lens, Ed, E, acc, cnt, dist, n)
        pf.pf_sync(c)
        assert np.array_equal(cnt.cpu().numpy().reshape(slots, n), oc[rows][:, rep])
        assert np.array_equal(acc.cpu().numpy().reshape(slots, n), oa[rows][:, rep])
        assert np.array_equal(dist.cpu().numpy(), (wantg if dec == 2 else want)[rep])


@pytest.mark.parametrize("sides", KINDS)
@pytest.mark.parametrize("per_pair", [False, True])
def test_scheduler(pf, ctx, sides, per_pair):  # noqa: F811
    """Every batch through the scheduler, four and eight lanes per group; with
    per-pair thresholds all pairs fall in one bin."""
    for E, n in ((6, 700), (16, 1501), (30, 257), (11, 1)):
        P, pairs, rep = batch(pf, ctx, E, n, E)
        moved_pairs = pf.Pairs(moved(pf, pairs.read, n, sides[0]), moved(pf, pairs.ref, n, sides[1]))
        run(pf, ctx, P, moved_pairs, rep, E, per_pair)


@pytest.mark.parametrize("sides", KINDS)
@pytest.mark.parametrize("n,E,per_pair", [(60011, 13, False), (100031, 16, False),
                                          (100031, 16, True), (1048700, 16, False)])
def test_default_routes(pf, sides, n, E, per_pair):  # noqa: F811
    """16 lanes, 8 lanes, 16 lanes grouped, and the scheduler's default."""
    c = pf.pf_create(0)
    try:
        P, pairs, rep = batch(pf, c, n, n, E)
        run(pf, c, P, pf.Pairs(moved(pf, pairs.read, n, sides[0]), moved(pf, pairs.ref, n, sides[1])),
            rep, E, per_pair)
    finally:
        pf.pf_destroy(c)


@pytest.mark.parametrize("sides", KINDS)
@pytest.mark.parametrize("n", [300, 200003])
def test_submatrices(pf, sides, n):  # noqa: F811
    c = pf.pf_create(0)
    try:
        for E in (9, 28):
            P, pairs, rep = batch(pf, c, E, n, E)
            want = oracle.int_batch("ss_partitioned", P, p0=8, p1=2)[rep]
            moved_pairs = pf.Pairs(moved(pf, pairs.read, n, sides[0]),
                                   moved(pf, pairs.ref, n, sides[1]))
            lens = torch.full((n,), M, dtype=torch.int32, device=DEV)
            acc = torch.full((n,), 9, dtype=torch.uint8, device=DEV)
            cnt = torch.full((n,), 99, dtype=torch.int16, device=DEV)
            pf.pf_filter_partitioned(c, moved_pairs, lens, None, E, 8, 2, acc, cnt, n)
            pf.pf_sync(c)
            assert np.array_equal(cnt.cpu().numpy(), want)
            assert np.array_equal(acc.cpu().numpy(), (want <= E).astype(np.uint8))
    finally:
        pf.pf_destroy(c)


@pytest.mark.parametrize("n", [300, 200003])
@pytest.mark.parametrize("both", [False, True])
def test_submatrices_over_rows_that_run_backwards(pf, n, both):  # noqa: F811
    """pf_filter_partitioned takes a negative stride; the rows lie in reverse
    behind the planes' first one."""
    c = pf.pf_create(0)
    try:
        E = 9
        P, pairs, rep = batch(pf, c, 77, n, E)
        want = oracle.int_batch("ss_partitioned", P, p0=8, p1=2)[rep]

        def backwards(seqs):
            fwd = moved(pf, seqs, n, "strided")
            planes = [x.view(n, W).flip(0).reshape(-1) for x in (fwd.lo, fwd.hi, fwd.nmask)]
            return pf.Seqs(*[x[(n - 1) * W:] for x in planes], stride_words=-W)

        read = backwards(pairs.read)
        ref = backwards(pairs.ref) if both else moved(pf, pairs.ref, n, "strided")
        lens = torch.full((n,), M, dtype=torch.int32, device=DEV)
        acc = torch.full((n,), 9, dtype=torch.uint8, device=DEV)
        cnt = torch.full((n,), 99, dtype=torch.int16, device=DEV)
        pf.pf_filter_partitioned(c, pf.Pairs(read, ref), lens, None, E, 8, 2, acc, cnt, n)
        pf.pf_sync(c)
        assert np.array_equal(cnt.cpu().numpy(), want)
        assert np.array_equal(acc.cpu().numpy(), (want <= E).astype(np.uint8))
    finally:
        pf.pf_destroy(c)
