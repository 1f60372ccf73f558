"""The verifier's two pairs to a word end when both are over."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_verify_pairs import packed, pf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("partner", ["short", "absent", "refused"])
def test_a_partner_that_is_over_does_not_hold_a_long_pair(pf, partner):  # noqa: F811
    """Two to a word: an unrelated pair of a million bases beside a short equal
    one, nothing or a refused pair is over after its first few hundred columns."""
    m, E = 1_000_000, 6
    n = 100_000 + (32 if partner == "absent" else 0)   # the last 32 have no partners
    rng = np.random.default_rng(9)
    letters = np.frombuffer(b"ACGT", np.uint8)
    refs = rng.choice(letters, size=m)
    reads = rng.choice(letters, size=m)
    P = synth.Pairs(np.concatenate([reads, refs[:100]]), np.concatenate([refs, refs[:100]]),
                    np.array([0, m, m + 100]), np.array([0, m, m + 100]),
                    np.array([m, 100], np.int32), np.array([E, E], np.int16))
    ctx = pf.pf_create(0)
    try:
        pairs = packed(pf, ctx, P)
        t = torch.arange(n, device="cuda")
        # position t and t + 32 of a chunk of 64 share a word
        other = t % 64 >= 32 if partner != "absent" else torch.zeros_like(t, dtype=torch.bool)
        kind = (other & (partner == "short")).to(torch.int64)
        pairs.read.word_off = pairs.ref.word_off = pairs.read.word_off[kind].contiguous()
        lens = torch.where(kind == 1, 100, m).to(torch.int32)
        if partner == "refused":
            lens[other] = -1
        dist = torch.full((n,), 77, dtype=torch.int32, device="cuda")

        def ms(e):
            best = 1e9
            for _ in range(3):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                pf.pf_verify(ctx, pairs, lens, None, e, None, None, dist, n)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best

        one = ms(15)
        assert ms(E) < 3 * one        # (one pair a thread at E = 15)
        if partner == "refused":
            with pytest.raises(pf.PFError):
                pf.pf_sync(ctx)
        d = dist.cpu().numpy()
        o = other.cpu().numpy()
        assert (d[~o] == E + 1).all()
        assert (d[o] == (0 if partner == "short" else -1)).all()
    finally:
        pf.pf_destroy(ctx)
