"""Batches below the small-batch size: every route on both sides of the lines
between them gives the plain kernel's answers, and takes no longer than it."""
import numpy as np
import pytest
import torch

from gpu_util import to_dev
from test_gpu_sliced import pf  # noqa: F401

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def pairs_of(pf, n, m, seed):  # noqa: F811
    """n strided pairs of m bases: a quarter equal but for a few bases, the
    others unrelated."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    W = (m + 31) // 32
    word = lambda: torch.randint(-2**31, 2**31 - 1, (n, W), generator=g, device=DEV).to(torch.int32)
    lo, hi = word(), word()
    near = (torch.arange(n, device=DEV) % 4 == 0)[:, None]
    few = word() & word() & word() & word() & word()
    rlo, rhi = torch.where(near, lo ^ few, word()), torch.where(near, hi, word())
    nm = torch.zeros((n, W), dtype=torch.int32, device=DEV)
    side = lambda a, b: pf.Seqs(a.reshape(-1), b.reshape(-1), nm.reshape(-1), stride_words=W)
    return pf.Pairs(side(rlo, rhi), side(lo, hi)), torch.full((n,), m, dtype=torch.int32, device=DEV)


LINES = [(12, 3, 39_999), (12, 3, 40_000), (15, 1, 99_999), (15, 1, 100_000), (11, 1, 49_999),
         (10, 1, 50_000), (10, 3, 119_999), (11, 3, 120_000), (8, 1, 249_999), (9, 1, 250_000),
         (9, 3, 449_999), (9, 3, 450_000), (8, 3, 649_999), (8, 3, 650_000), (8, 1, 600_000),
         (7, 1, 599_999), (7, 1, 600_000), (7, 3, 650_000), (9, 3, 550_000), (20, 2, 7_999),
         (20, 2, 8_000), (17, 2, 549_999), (17, 2, 550_000)]


@pytest.mark.parametrize("E,dec,n", LINES)
def test_one_threshold(pf, E, dec, n):  # noqa: F811
    pairs, lens = pairs_of(pf, n, 100, E)
    compare(pf, dec, pairs, lens, None, E, n)


@pytest.mark.parametrize("E,dec,n", [(8, 1, 174_999), (14, 1, 175_000), (15, 1, 99_999), (15, 1, 100_000), (12, 3, 99_999),
                                     (12, 3, 100_000), (25, 2, 174_999), (25, 2, 175_000),
                                     (15, 3, 10_000), (15, 3, 10_001), (25, 1, 40_000),
                                     (25, 1, 40_001)])
def test_thresholds_per_pair(pf, E, dec, n):  # noqa: F811
    pairs, lens = pairs_of(pf, n, 100, E)
    compare(pf, dec, pairs, lens,
            to_dev(np.random.default_rng(n).integers(0, E + 1, size=n).astype(np.int16)), E, n)


def compare(pf, dec, pairs, lens, Ed, E, n):  # noqa: F811
    slots = 2 if dec == 3 else 1
    out = [(torch.full((slots * n,), 9, dtype=torch.uint8, device=DEV),
            torch.full((slots * n,), 99, dtype=torch.int16, device=DEV)) for _ in range(2)]
    c = pf.pf_create(0)
    try:
        pf.pf_filter(c, dec, pairs, lens, Ed, E, *out[0], n)
        pf.pf_filter_plain(c, dec, pairs, lens, Ed, E, *out[1], n)
        pf.pf_sync(c)
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert 0 < int(out[0][0].sum()) < slots * n
    finally:
        pf.pf_destroy(c)


@pytest.mark.parametrize("E,dec,n", [(12, 3, 30_000), (8, 1, 80_000), (10, 3, 60_000),
                                     (7, 3, 460_000), (8, 3, 460_000)])
def test_no_slower_than_the_plain_kernel(pf, E, dec, n):  # noqa: F811
    """250 bp, where the other routes once began too early (20 to 40 % slower)."""
    pairs, lens = pairs_of(pf, n, 250, E)
    acc = torch.zeros(2 * n, dtype=torch.uint8, device=DEV)
    cnt = torch.zeros(2 * n, dtype=torch.int16, device=DEV)
    c = pf.pf_create(0)

    def us(call):
        best = 1e9
        for _ in range(15):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(8):
                call()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 125)
        return best

    try:
        own = us(lambda: pf.pf_filter(c, dec, pairs, lens, None, E, acc, cnt, n))
        plain = us(lambda: pf.pf_filter_plain_exact(c, dec, pairs, lens, E, acc, cnt, n))
        assert own < 1.12 * plain
    finally:
        pf.pf_destroy(c)
