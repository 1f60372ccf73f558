"""pf_run_host calls of one context share its slots: chunk counts around the
line from enqueued to replayed chunks, calls that grow and shrink, lengths and
layouts that change between calls, memory that is given back."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


def test_calls_of_different_shapes():
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as pf
    fixed = [synth.generate(synth.SKEWED, 31, 1601, m=150, E=6),
             synth.generate(synth.SKEWED, 32, 1601, m=100, E=4)]
    mixed = synth.generate(synth.MIXED, 33, 1601)
    want = {}
    for P in fixed + [mixed]:
        acc, cnt = oracle.filter_batch(P)
        want[id(P)] = acc, cnt, np.where(acc[0] == 1, oracle.verify_batch(P),
                                         P.E.astype(np.int32) + 1)
    ctx = pf.pf_create(0)
    try:
        free0 = torch.cuda.mem_get_info()[0]
        for chunk in (0, 801, 800, 229, 200, 178, 1601, 100):
            for P, m, E in ((fixed[0], 150, 6), (mixed, 0, 0), (fixed[1], 100, 4)):
                if m:
                    got = pf.pf_run_host(ctx, 3, P.reads, P.refs, E, length=m, chunk_pairs=chunk)
                else:
                    got = pf.pf_run_host(ctx, 3, P.reads, P.refs, int(P.E.max()),
                                         byte_off=P.read_off, E=P.E, chunk_pairs=chunk)
                for a, b in zip(got, want[id(P)]):
                    assert np.array_equal(a, b), (chunk, m)
        # a slot of more than a gigabyte is not kept
        n = 2500 * 1024
        rep = lambda x: np.tile(x[:150 * 1024], n // 1024)
        P = fixed[0]
        acc, cnt, dist = pf.pf_run_host(ctx, 1, rep(P.reads), rep(P.refs), 6, length=150,
                                        chunk_pairs=3 << 20)
        assert np.array_equal(dist, np.tile(want[id(P)][2][:1024], n // 1024))
        assert free0 - torch.cuda.mem_get_info()[0] < 1 << 30
    finally:
        pf.pf_destroy(ctx)
