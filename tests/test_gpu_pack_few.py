"""The ragged packers on both sides of the line between 64 and 256 sequences a
block, consecutive words and words at given starts, against a packing in
numpy."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def planes(seqs, off, n, W):
    """lo, hi, N words (n, W) of the sequences, N behind their ends."""
    cols = np.arange(32 * W)
    lens = np.diff(off)
    at = np.minimum(off[:-1, None] + cols, max(len(seqs) - 1, 0))
    c = np.where(cols < lens[:, None], seqs[at], ord("N"))
    code = np.full(256, 4, np.uint8)
    code[list(b"ACGT")] = range(4)
    c = code[c]
    bits = [(c == 1) | (c == 3), (c == 2) | (c == 3), c == 4]
    return [np.packbits(b, axis=1, bitorder="little").view("<u4").reshape(n, W) for b in bits]


@pytest.mark.parametrize("n", [1, 63, 64, 65, 129, 49999, 50000, 50257])
def test_ragged_words(n):
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as pf
    rng = np.random.default_rng(n)
    lens = rng.choice([0, 1, 31, 32, 33, 64, 65, 100], size=n)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    seqs = rng.choice(np.frombuffer(b"ACGTN", np.uint8), size=int(off[-1]) + 1)
    lo, hi, nm = planes(seqs, off, n, 4)
    ctx = pf.pf_create(0)
    try:
        dev = torch.from_numpy(seqs).cuda()
        for group in (None, rng.integers(0, 9, size=n).astype(np.int16)):
            pairs = pf.pack_pairs(ctx, dev, dev, byte_off=off, group_E=group)
            pf.pf_sync(ctx)
            start = pairs.read.word_off.cpu().numpy()[:n]
            got = [x.cpu().numpy().view(np.uint32) for x in (pairs.read.lo, pairs.read.hi,
                                                             pairs.read.nmask)]
            for w in range(4):
                has = lens > 32 * w
                for g, want in zip(got, (lo, hi, nm)):
                    assert np.array_equal(g[start[has] + w], want[has, w])
    finally:
        pf.pf_destroy(ctx)
