"""Four- and eight-lane tiles over a real order: large batches with per-pair
thresholds, grouped in the planes, against the oracle on the pairs that they
repeat.  With few thresholds every bin has its own launch, with many a launch
takes the bins of a class; bins end inside a tile, one is empty, some pairs are
refused and some are long."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_dev
from test_gpu_sliced import pf, ragged  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def grouped_batch(pf, c, seed, thresholds, n, kinds):  # noqa: F811
    """About n pairs in the order of their threshold and words, which repeat
    `kinds` pairs of each threshold; returns the pairs, their lengths and
    thresholds and the repeated pair of each."""
    rng = np.random.default_rng(seed)
    E = np.repeat(thresholds, kinds)
    lens = rng.choice([1, 31, 33, 64, 90, 100, 127, 150], size=len(E))
    lens[rng.random(len(E)) < 0.01] = 700
    P = ragged(seed, lens, E)
    words = (P.lens.astype(np.int64) + 31) // 32
    share = n // len(thresholds)
    rep = []
    for e in thresholds:
        own = np.nonzero(E == e)[0]
        some = rng.choice(own, size=share + int(rng.integers(1, 250)))
        rep.append(some[np.argsort(words[some], kind="stable")])
    rep = np.concatenate(rep)
    base = pf.pack_pairs(c, to_dev(P.reads), to_dev(P.refs), byte_off=P.read_off)
    rd, wd = to_dev(rep), to_dev(words[rep])
    off = torch.cumsum(wd, 0) - wd
    # word k of the batch: its pair's first word there, plus how far on it is
    src = torch.repeat_interleave(base.read.word_off[rd] - off, wd)
    src += torch.arange(len(src), device=DEV)
    side = lambda s: pf.Seqs(s.lo[src], s.hi[src], s.nmask[src], word_off=off)
    return P, pf.Pairs(side(base.read), side(base.ref)), rep, rd


@pytest.mark.parametrize("dec", [1, 2, 3])
@pytest.mark.parametrize("thresholds,n", [
    ([0, 5, 6, 7, 8, 10, 11, 13, 15, 16, 19, 21, 22, 24, 25, 26, 27, 28, 30, 31], 1_700_000),
    ([3, 5, 7, 8], 4_300_000)])
def test_large_grouped_batches(pf, dec, thresholds, n):  # noqa: F811
    E_max = max(thresholds)
    c = pf.pf_create(0)
    try:
        cfgs = pf.pf_kernel_configs()
        for i, x in enumerate(cfgs):   # the bit-sliced configuration of every threshold
            if x[3] >= 0 and x[0] > 1:
                pf.pf_tune_set(c, dec, x[3], i, 64)
        P, pairs, rep, rd = grouped_batch(pf, c, dec + n, np.array(thresholds), n, 180)
        n = len(rep)
        lens, E = to_dev(P.lens)[rd], to_dev(P.E)[rd]
        bad = torch.arange(77, n, n // 50, device=DEV)
        E[bad[::3]] = E_max + 1
        E[bad[1::3]] = -5
        lens[bad[2::3]] = -1
        slots, rows = (2, [0, 1]) if dec == 3 else (1, [dec - 1])
        acc = torch.full((slots * n,), 9, dtype=torch.uint8, device=DEV)
        cnt = torch.full((slots * n,), 99, dtype=torch.int16, device=DEV)
        dist = torch.full((n,), -7, dtype=torch.int32, device=DEV)
        pf.pf_filter_verify(c, dec, pairs, lens, E, E_max, acc, cnt, dist, n)
        with pytest.raises(pf.PFError):
            pf.pf_sync(c)
        oa, oc = oracle.filter_batch(P)
        od = np.where(oa[rows[0]] == 1, oracle.verify_batch(P), P.E.astype(np.int32) + 1)
        want_c, want_a, want_d = to_dev(oc[rows])[:, rd], to_dev(oa[rows])[:, rd], to_dev(od)[rd]
        want_c[:, bad], want_a[:, bad], want_d[bad] = -1, 0, -1
        assert torch.equal(cnt.view(slots, n), want_c.to(torch.int16))
        assert torch.equal(acc.view(slots, n), want_a.to(torch.uint8))
        assert torch.equal(dist, want_d.to(torch.int32))
    finally:
        pf.pf_destroy(c)
