"""Bit-sliced tiles end where every pair is decided: counts that pass the
threshold around the segments' ends, and pairs whose columns are worth skipping."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import to_dev
from test_gpu_sliced import check, ctx, pf  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def prefix_pairs(seed, lens, E, upto):
    """Pair p's first upto[p] bases are unrelated, the others equal."""
    rng = np.random.default_rng(seed)
    off = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    letters = np.frombuffer(b"ACGT", np.uint8)
    refs = rng.choice(letters, size=int(off[-1]))
    reads = refs.copy()
    for p, m in enumerate(lens):
        k = min(int(upto[p]), int(m))
        reads[off[p]:off[p] + k] = rng.choice(letters, size=k)
    return synth.Pairs(reads, refs, off, off, np.asarray(lens, np.int32),
                       np.full(len(lens), E, np.int16))


@pytest.mark.parametrize("E", [5, 8, 15, 21, 29])
@pytest.mark.parametrize("same", [True, False])
def test_counts_that_pass_the_threshold_near_a_segment_end(pf, ctx, E, same):  # noqa: F811
    """Tiles of one length and of mixed ones, some pairs absent; the unrelated
    part ends around the columns where the obstacles (about one in four to
    seven columns) and the edits pass E, so that tiles are decided or just not."""
    rng = np.random.default_rng(E)
    n = 256 * 12 + 37
    lens = np.full(n, 300) if same else rng.choice([31, 64, 65, 200, 290, 300], size=n)
    # a tile's pairs agree on the range: few tiles have a pair far off it
    mid = np.repeat(rng.integers(2 * E, 16 * E, size=(n + 63) // 64), 64)[:n]
    P = prefix_pairs(E, lens, E, mid + rng.integers(-3, 4, size=n))
    pairs = pf.pack_pairs(ctx, to_dev(P.reads), to_dev(P.refs), byte_off=P.read_off)
    check(pf, ctx, P, pairs, None, E)
    want = oracle.int_batch("ss_partitioned", P, p0=8, p1=2)
    lens_d = to_dev(P.lens)
    acc = torch.full((n,), 9, dtype=torch.uint8, device=DEV)
    cnt = torch.full((n,), 99, dtype=torch.int16, device=DEV)
    pf.pf_filter_partitioned(ctx, pairs, lens_d, None, E, 8, 2, acc, cnt, n)
    pf.pf_sync(ctx)
    assert np.array_equal(cnt.cpu().numpy(), want)


@pytest.mark.parametrize("dec", [1, 2, 3])
def test_decided_tiles_cost_no_more_columns(pf, dec):  # noqa: F811
    """Unrelated pairs of 50,000 bases are decided in their first few hundred:
    a call may not take several times as long as on pairs of 500."""
    n, m, base, E = 110_000, 50_000, 64, 25
    rng = np.random.default_rng(dec)
    c = pf.pf_create(0)
    try:
        letters = np.frombuffer(b"ACGT", np.uint8)
        reads, refs = (to_dev(rng.choice(letters, size=base * m)) for _ in range(2))
        pairs = pf.pack_pairs(c, reads, refs, byte_off=np.arange(base + 1, dtype=np.int64) * m)
        rep = torch.arange(n, device=DEV) % base
        pairs.read.word_off = pairs.ref.word_off = pairs.read.word_off[rep].contiguous()
        Ed = to_dev(rng.integers(16, E + 1, size=n).astype(np.int16))
        acc = torch.zeros(2 * n, dtype=torch.uint8, device=DEV)
        cnt = torch.zeros(2 * n, dtype=torch.int16, device=DEV)

        def ms(length):
            lens = torch.full((n,), length, dtype=torch.int32, device=DEV)
            best = 1e9
            for _ in range(5):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                pf.pf_filter(c, dec, pairs, lens, Ed, E, acc, cnt, n)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best

        assert ms(m) < 3 * ms(500)
    finally:
        pf.pf_destroy(c)
