"""Shouji's table of steps and its rows at constant shifts, against the oracle:
every class of kernels, thresholds that move rows across a read word, lengths
that end at every column of eight, per-pair thresholds."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_sliced import ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [0, 1, 6, 7, 8, 15, 16, 24, 31])
def test_shouji_edges(E):
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as pf
    rng = np.random.default_rng(E)
    n = 600
    lens = np.concatenate([np.arange(0, 70), rng.choice([95, 96, 97, 128, 150, 161, 250],
                                                        size=n - 70)])
    ctx = pf.pf_create(0)
    try:
        for Es in (np.full(n, E), rng.integers(0, E + 1, size=n)):
            P = ragged(E + 7, lens, Es)
            reads, refs = torch.from_numpy(P.reads).cuda(), torch.from_numpy(P.refs).cuda()
            pairs = pf.pack_pairs(ctx, reads, refs, byte_off=P.read_off)
            want = oracle.int_batch("shouji", P)
            one = bool((Es == E).all())
            acc = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
            cnt = torch.full((n,), 99, dtype=torch.int16, device="cuda")
            pf.pf_filter_shouji(ctx, pairs, torch.from_numpy(P.lens).cuda(),
                                None if one else torch.from_numpy(P.E).cuda(), E, acc, cnt, n)
            pf.pf_sync(ctx)
            assert np.array_equal(cnt.cpu().numpy(), want)
            assert np.array_equal(acc.cpu().numpy(), (want <= P.E).astype(np.uint8))
    finally:
        pf.pf_destroy(ctx)
