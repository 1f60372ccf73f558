"""The bit-sliced kernels at the edges of their tiles, against the oracle:
ragged pairs of mixed lengths in one tile, lengths around word and segment
boundaries, bins of fewer pairs than a tile, words in any order, planes of
different layouts on the two sides, and invalid per-pair thresholds."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as m
    return m


@pytest.fixture()
def ctx(pf):
    c = pf.pf_create(0)
    pf.pf_set_small_batch(c, 0)
    # every threshold that a bit-sliced configuration serves
    cfgs = pf.pf_kernel_configs()
    for e in range(32):
        own = [i for i, x in enumerate(cfgs) if x[3] == e and x[0] > 1]
        for dec in (1, 2, 3):
            if own:
                pf.pf_tune_set(c, dec, e, own[0], 64)
    yield c
    pf.pf_destroy(c)


def ragged(seed, lens, E, kmax=40):
    """Pairs of the given lengths and thresholds with N's, random edits and
    some reads that match nowhere."""
    rng = np.random.default_rng(seed)
    off = np.zeros(len(lens) + 1, dtype=np.int64)
    np.cumsum(lens, out=off[1:])
    letters = np.frombuffer(b"ACGTN", np.uint8)
    prob = [0.295, 0.205, 0.205, 0.29, 0.005]
    refs = rng.choice(letters, size=max(int(off[-1]), 1), p=prob)
    reads = refs.copy()
    for p, m in enumerate(lens):
        r = list(refs[off[p]:off[p] + m])
        for _ in range(int(rng.integers(0, min(kmax, 2 * E[p] + 3)))):
            at = int(rng.integers(0, m)) if m else 0
            kind = rng.integers(0, 3)
            if not m:
                break
            if kind == 0:
                r[at] = rng.choice(letters)
            elif kind == 1:
                r.insert(at, rng.choice(letters))
            else:
                del r[at]
                r.append(rng.choice(letters))
        reads[off[p]:off[p] + m] = np.array(r[:m], np.uint8)
    return synth.Pairs(reads[:off[-1]], refs[:off[-1]], off, off,
                       np.asarray(lens, np.int32), np.asarray(E, np.int16))


def check(pf, ctx, P, pairs, E, E_max, bad=()):
    dev = "cuda:0"
    n = P.n
    oa, oc = oracle.filter_batch(P)
    od = oracle.verify_batch(P)
    ok = np.ones(n, bool)
    ok[list(bad)] = False
    lens = torch.from_numpy(P.lens).to(dev)
    Ed = None if E is None else torch.from_numpy(np.asarray(E, np.int16)).to(dev)
    for dec in (1, 2, 3):
        slots = 2 if dec == 3 else 1
        rows = [0, 1] if dec == 3 else [dec - 1]
        acc = torch.full((slots * n,), 9, dtype=torch.uint8, device=dev)
        cnt = torch.full((slots * n,), 99, dtype=torch.int16, device=dev)
        dist = torch.full((n,), -7, dtype=torch.int32, device=dev)
        pf.pf_filter_verify(ctx, dec, pairs, lens, Ed, E_max, acc, cnt, dist, n)
        if len(bad):
            with pytest.raises(pf.PFError):
                pf.pf_sync(ctx)
        else:
            pf.pf_sync(ctx)
        c = cnt.cpu().numpy().reshape(slots, n)
        a = acc.cpu().numpy().reshape(slots, n)
        assert np.array_equal(c[:, ok], oc[rows][:, ok])
        assert np.array_equal(a[:, ok], oa[rows][:, ok])
        want = np.where(oa[rows[0]] == 1, od, P.E.astype(np.int32) + 1)
        assert np.array_equal(dist.cpu().numpy()[ok], want[ok])
        assert (c[:, ~ok] == -1).all() and (a[:, ~ok] == 0).all()
        assert (dist.cpu().numpy()[~ok] == -1).all()


@pytest.mark.parametrize("E", [5, 7, 11, 16, 27, 28, 31])
@pytest.mark.parametrize("n", [1, 255, 257, 700])
def test_lengths_around_words_in_one_tile(pf, ctx, E, n):
    """One threshold, lengths 0..330 mixed in every tile (pair order: one
    bin), so that a tile's pairs end in different words and segments."""
    rng = np.random.default_rng(1000 * E + n)
    lens = rng.choice([0, 1, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 150, 160, 161, 192, 250,
                       256, 257, 288, 330], size=n)
    P = ragged(E + n, lens, np.full(n, E))
    dev = "cuda:0"
    reads, refs = (torch.from_numpy(np.ascontiguousarray(x if x.size else np.zeros(1, np.uint8))).to(dev)
                   for x in (P.reads, P.refs))
    check(pf, ctx, P, pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off), None, E)


@pytest.mark.parametrize("m", [1, 32, 150, 160, 250, 256, 300])
def test_one_length_in_a_strided_layout(pf, ctx, m):
    """The strided layout (rows of one stride), a last tile of few pairs."""
    for E in (6, 13, 30):
        n = 256 * 3 + 41
        P = ragged(m + E, np.full(n, m), np.full(n, E))
        dev = "cuda:0"
        pairs = pf.pack_pairs(ctx, torch.from_numpy(P.reads).to(dev),
                              torch.from_numpy(P.refs).to(dev), length=m)
        check(pf, ctx, P, pairs, None, E)


@pytest.mark.parametrize("group", [False, True])
def test_thresholds_and_invalid_pairs_mixed(pf, ctx, group):
    """Per-pair thresholds 0..31 in bins of some tens of pairs, in both
    ragged layouts; thresholds above E_max and below 0 are refused pair by
    pair."""
    rng = np.random.default_rng(77)
    n = 3000
    lens = rng.choice([40, 100, 150, 250], size=n)
    E = rng.integers(0, 32, size=n)
    P = ragged(5, lens, E)
    dev = "cuda:0"
    reads, refs = torch.from_numpy(P.reads).to(dev), torch.from_numpy(P.refs).to(dev)
    pairs = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off, group_E=E if group else None)
    check(pf, ctx, P, pairs, E, 31)
    bad = [0, 255, 256, 1700, n - 1]
    Eb = E.copy()
    Eb[bad] = [-1, 33, 400, -32768, 32]
    check(pf, ctx, P, pairs, Eb, 31, bad)


def test_sides_in_different_layouts(pf, ctx):
    """Reads in pair order, references in the grouped layout."""
    rng = np.random.default_rng(8)
    n = 900
    lens = rng.choice([100, 150, 250], size=n)
    E = rng.integers(5, 26, size=n)
    P = ragged(6, lens, E)
    dev = "cuda:0"
    reads, refs = torch.from_numpy(P.reads).to(dev), torch.from_numpy(P.refs).to(dev)
    a = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off)
    b = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off, group_E=E)
    check(pf, ctx, P, pf.Pairs(a.read, b.ref), E, 25)


@pytest.mark.parametrize("n,m,E,E_max", [
    (700, 0, None, 31),        # one warp per pair
    (9000, 0, None, 12),
    (45001, 0, None, 31),      # grouped by threshold, 16 lanes per group
    (76000, 0, None, 15),
    (2500, 90, 20, 20),        # one threshold: one warp per pair,
    (30011, 64, 13, 13),       # 16 lanes,
    (100031, 40, 25, 25),      # 8 lanes,
    (100031, 33, 9, 9),
    (450100, 33, 9, 9),        # the scheduler
])
def test_small_batch_routes(pf, n, m, E, E_max):
    """Each way a batch below the small-batch size can run, at the default
    setting, on both sides of the lines between them."""
    if m:
        P = synth.generate(synth.SKEWED, 31 * n + m, n, m=m, E=E, kmax=40)
    else:
        P = synth.generate(synth.SERVE, 17 * n, n, kmax=60)
        P.E = np.minimum(P.E, E_max).astype(np.int16)
        if E_max > 25:
            P.E[::97] = np.arange(len(P.E[::97])) % 32
    ctx = pf.pf_create(0)
    try:
        dev = "cuda:0"
        reads, refs = torch.from_numpy(P.reads).to(dev), torch.from_numpy(P.refs).to(dev)
        pairs = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off)
        check(pf, ctx, P, pairs, None if m else P.E, E_max)
    finally:
        pf.pf_destroy(ctx)


@pytest.mark.parametrize("t,y", [(8, 2), (8, 8), (5, 3), (32, 32), (1, 1), (13, 4), (32, 1), (32, 31)])
@pytest.mark.parametrize("n", [300, 200003])
def test_submatrices_at_one_threshold(pf, t, y, n):
    """Both forms of the bit-sliced sub-matrix kernel (16 and 4 lanes per
    group) and what small thresholds take beside them, each count of replication
    bits, every class of thresholds, lengths mixed in a tile."""
    dev = "cuda:0"
    few = n > 1000
    for E in (0, 4, 7, 11, 15, 20, 25, 31) if not few else (0, 2, 5, 6, 9, 13, 20, 28):
        rng = np.random.default_rng(E * 100 + t)
        m = 3000 if few else n
        lens = rng.choice([0, 1, 31, 33, 64, 65, 100, 127, 150, 161], size=m)
        P = ragged(E + t, lens, np.full(m, E))
        ctx = pf.pf_create(0)
        try:
            reads, refs = torch.from_numpy(P.reads).to(dev), torch.from_numpy(P.refs).to(dev)
            pairs = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off)
            want = oracle.int_batch("ss_partitioned", P, p0=t, p1=y).copy()
            if few:   # the same pairs over and over
                rep = np.arange(n) % m
                off = pairs.read.word_off[torch.from_numpy(rep).to(dev)].contiguous()
                pairs.read.word_off = pairs.ref.word_off = off
                lens, want = P.lens[rep], want[rep]
            ld = torch.from_numpy(np.ascontiguousarray(lens, dtype=np.int32)).to(dev)
            acc = torch.full((n,), 9, dtype=torch.uint8, device=dev)
            cnt = torch.full((n,), 99, dtype=torch.int16, device=dev)
            pf.pf_filter_partitioned(ctx, pairs, ld, None, E, t, y, acc, cnt, n)
            pf.pf_sync(ctx)
            c = cnt.cpu().numpy()
            assert np.array_equal(c, want), (E, np.nonzero(c != want)[0][:5])
            assert np.array_equal(acc.cpu().numpy(), (want <= E).astype(np.uint8))
            if not few:   # a negative length is refused, its neighbours are not
                ld[5] = -1
                pf.pf_filter_partitioned(ctx, pairs, ld, None, E, t, y, acc, cnt, n)
                with pytest.raises(pf.PFError):
                    pf.pf_sync(ctx)
                c = cnt.cpu().numpy()
                assert c[5] == -1 and acc[5].item() == 0
                assert np.array_equal(np.delete(c, 5), np.delete(want, 5))
        finally:
            pf.pf_destroy(ctx)
