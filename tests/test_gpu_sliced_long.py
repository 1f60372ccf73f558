"""Long pairs and the bit-sliced kernels: tiles leave them to the word-per-pair
kernels, in every route, with the same answers; and a call with long pairs takes
about as long as by those kernels alone."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_dev
from test_gpu_sliced import check, ctx, pf, ragged  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# around the first long lengths of E < 10, E < 16 and E >= 16
EDGES = [351, 352, 353, 479, 480, 481, 640, 641, 1000]


def submat(pf, c, pairs, lens, E, n):  # noqa: F811
    acc = torch.full((n,), 9, dtype=torch.uint8, device=DEV)
    cnt = torch.full((n,), 99, dtype=torch.int16, device=DEV)
    pf.pf_filter_partitioned(c, pairs, lens, None, E, 8, 2, acc, cnt, n)
    pf.pf_sync(c)
    return cnt.cpu().numpy()


@pytest.mark.parametrize("E", [8, 13, 20, 29])
@pytest.mark.parametrize("share", [0.005, 0.3, 1.0])
def test_lengths_around_the_line(pf, ctx, E, share):  # noqa: F811
    """A few, a third or all of the pairs long, in tiles of one threshold, and
    some pairs refused."""
    rng = np.random.default_rng(E)
    n = 1200
    lens = np.where(rng.random(n) < share, rng.choice(EDGES, size=n), rng.integers(0, 300, size=n))
    P = ragged(E, lens, np.full(n, E))
    pairs = pf.pack_pairs(ctx, to_dev(P.reads), to_dev(P.refs), byte_off=P.read_off)
    check(pf, ctx, P, pairs, None, E)
    Eb = P.E.copy()
    bad = [0, 300, n - 1]
    Eb[bad] = [-1, 32, E + 1]
    check(pf, ctx, P, pairs, Eb, E, bad)
    assert np.array_equal(submat(pf, ctx, pairs, to_dev(P.lens), E, n),
                          oracle.int_batch("ss_partitioned", P, p0=8, p1=2))


@pytest.mark.parametrize("n,E", [(50_001, 13), (300_003, 9), (200_001, 20), (1_100_000, 10)])
@pytest.mark.parametrize("long", [0.01, 0.5])
def test_default_routes(pf, n, E, long):  # noqa: F811
    """The routes at their default settings, over repeated pairs."""
    rng = np.random.default_rng(n)
    m = 1500
    lens = np.where(rng.random(m) < long, rng.choice(EDGES, size=m), rng.choice([33, 100], size=m))
    P = ragged(E, lens, np.full(m, E))
    c = pf.pf_create(0)
    try:
        pairs = pf.pack_pairs(c, to_dev(P.reads), to_dev(P.refs), byte_off=P.read_off)
        rep = np.arange(n) % m
        rd = to_dev(rep)
        pairs.read.word_off = pairs.ref.word_off = pairs.read.word_off[rd].contiguous()
        ld = to_dev(P.lens)[rd]
        oa, oc = oracle.filter_batch(P)
        od = np.where(oa[0] == 1, oracle.verify_batch(P), E + 1)
        for dec in (1, 3):
            slots = 2 if dec == 3 else 1
            acc = torch.full((slots * n,), 9, dtype=torch.uint8, device=DEV)
            cnt = torch.full((slots * n,), 99, dtype=torch.int16, device=DEV)
            dist = torch.full((n,), -7, dtype=torch.int32, device=DEV)
            pf.pf_filter_verify(c, dec, pairs, ld, None, E, acc, cnt, dist, n)
            pf.pf_sync(c)
            assert np.array_equal(cnt.cpu().numpy().reshape(slots, n), oc[:slots][:, rep])
            assert np.array_equal(acc.cpu().numpy().reshape(slots, n), oa[:slots][:, rep])
            assert np.array_equal(dist.cpu().numpy(), od[rep])
        assert np.array_equal(submat(pf, c, pairs, ld, E, n),
                              oracle.int_batch("ss_partitioned", P, p0=8, p1=2)[rep])
    finally:
        pf.pf_destroy(c)


@pytest.mark.parametrize("n,E", [(30_011, 13), (1_100_000, 8), (200_001, 21)])
def test_long_rows(pf, n, E):  # noqa: F811
    """Strided rows whose length says that every pair is long."""
    m, base = 700, 500
    P = ragged(n, np.full(base, m), np.full(base, E))
    c = pf.pf_create(0)
    try:
        one = pf.pack_pairs(c, to_dev(P.reads), to_dev(P.refs), length=m)
        row = torch.arange(n, device=DEV) % base
        W = one.read.stride_words
        wide = [pf.Seqs(*[x.view(base, W)[row].reshape(-1) for x in (s.lo, s.hi, s.nmask)],
                        stride_words=W) for s in (one.read, one.ref)]
        pairs = pf.Pairs(*wide)
        rep = np.arange(n) % base
        ld = torch.full((n,), m, dtype=torch.int32, device=DEV)
        _, oc = oracle.filter_batch(P)
        acc = torch.full((2 * n,), 9, dtype=torch.uint8, device=DEV)
        cnt = torch.full((2 * n,), 99, dtype=torch.int16, device=DEV)
        pf.pf_filter(c, 3, pairs, ld, None, E, acc, cnt, n)
        pf.pf_sync(c)
        assert np.array_equal(cnt.cpu().numpy().reshape(2, n), oc[:, rep])
        assert np.array_equal(submat(pf, c, pairs, ld, E, n),
                              oracle.int_batch("ss_partitioned", P, p0=8, p1=2)[rep])
    finally:
        pf.pf_destroy(c)


def best_ms(f, reps=7):
    best = 1e9
    for _ in range(reps):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("spikes", [True, False])
def test_long_pairs_take_no_longer_than_by_the_word_kernels(pf, spikes):  # noqa: F811
    """SneakySnake at E = 8 over equal pairs: one of a thousand has 4,000 bases
    and the others 150, or all have 1,000.  The tiles took six and five times as
    long as the word-per-pair configuration of that threshold."""
    n, E = (1_100_000, 8)
    lens = torch.full((n,), 150 if spikes else 1000, dtype=torch.int32, device=DEV)
    if spikes:
        lens[::1000] = 4000
    words = (lens.to(torch.int64) + 31) // 32
    off = (torch.cumsum(words, 0) - words).contiguous()
    total = int(words.sum())
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    lo, hi = (torch.randint(-2**31, 2**31 - 1, (total,), generator=g, device=DEV).to(torch.int32)
              for _ in range(2))
    side = lambda: pf.Seqs(lo, hi, torch.zeros_like(lo), word_off=off)
    pairs = pf.Pairs(side(), side())
    acc = torch.zeros(n, dtype=torch.uint8, device=DEV)
    cnt = torch.zeros(n, dtype=torch.int16, device=DEV)
    c = pf.pf_create(0)
    try:
        call = lambda: pf.pf_filter(c, pf.PF_SNEAKYSNAKE, pairs, lens, None, E, acc, cnt, n)
        own = best_ms(call)
        words_cfg = [i for i, x in enumerate(pf.pf_kernel_configs()) if x[3] == E and x[0] == 1][0]
        pf.pf_tune_set(c, 1, E, words_cfg, 256)
        assert own < 1.5 * best_ms(call)
        assert int(cnt.abs().sum()) == 0 and bool((acc == 1).all())
    finally:
        pf.pf_destroy(c)


def test_lengths_near_the_largest_int(pf):  # noqa: F811
    """Unrelated pairs of up to 2^31 - 1 bases (all share one read and one
    reference): column counts past the length do not fit an int."""
    top, n, E = 2**31 - 1, 100_010, 20
    g = torch.Generator(device=DEV)
    g.manual_seed(2)
    word = lambda: torch.randint(-2**31, 2**31 - 1, (1 << 26,), generator=g,
                                 device=DEV).to(torch.int32)
    nm = torch.zeros(1 << 26, dtype=torch.int32, device=DEV)
    off = torch.zeros(n, dtype=torch.int64, device=DEV)
    pairs = pf.Pairs(pf.Seqs(word(), word(), nm, word_off=off), pf.Seqs(word(), word(), nm, word_off=off))
    lens = (top - torch.arange(n, device=DEV) % 40).to(torch.int32)
    lens[5::64] = 100
    Ed = torch.full((n,), E, dtype=torch.int16, device=DEV)
    Ed[::3] = 17
    new = lambda: (torch.full((2 * n,), 9, dtype=torch.uint8, device=DEV),
                   torch.full((2 * n,), 99, dtype=torch.int16, device=DEV))
    c = pf.pf_create(0)
    try:
        for e in (None, Ed):
            for dec in (1, 2, 3):
                got, want = new(), new()
                pf.pf_filter(c, dec, pairs, lens, e, E, *got, n)
                pf.pf_filter_plain(c, dec, pairs, lens, e, E, *want, n)
                pf.pf_sync(c)
                assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
                assert not got[0][:n][lens > 100].any()
        dist = torch.full((n,), -7, dtype=torch.int32, device=DEV)
        pf.pf_verify(c, pairs, lens, None, 6, None, None, dist, n)   # two pairs to a word
        pf.pf_sync(c)
        assert bool((dist == 7).all())
    finally:
        pf.pf_destroy(c)
