"""pf_run_host at the limit of device memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def pf():
    from paper_1910_03936_gb300 import build
    build.build()
    import paper_1910_03936_gb300 as m
    return m


def leave_free(nbytes):
    """Hold all of the device's memory but nbytes (in pieces, so that the call
    under test meets an ordinary refusal)."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    piece = 1 << 34
    while piece >= 1 << 24:
        if torch.cuda.mem_get_info()[0] - piece < nbytes:
            piece >>= 1
            continue
        held.append(torch.empty(piece, dtype=torch.uint8, device=DEV))
    return held


def pair_bytes(n, m):
    one = np.frombuffer(b"ACGT" * (m // 4), np.uint8)
    return np.tile(one, n)


def test_a_call_without_room_for_both_slots_writes_nothing(pf):
    """Two chunks, room for one slot (1.2 GB each) and a half."""
    m, chunk = 10_000, 40_000
    reads = pair_bytes(2 * chunk, m)
    out = (np.full(2 * chunk, 9, np.uint8), np.full(2 * chunk, 99, np.int16),
           np.full(2 * chunk, -7, np.int32))
    c = pf.pf_create(0)
    try:
        pf.pf_run_host(c, 1, reads[:8 * m], reads[:8 * m], 2, length=m)   # kernels loaded
        held = leave_free(1_800_000_000)
        try:
            with pytest.raises(pf.PFError) as e:
                pf.pf_run_host(c, 1, reads, reads, 2, length=m, chunk_pairs=chunk, out=out)
            assert e.value.status == 2   # PF_ENOMEM
            assert (out[0] == 9).all() and (out[1] == 99).all() and (out[2] == -7).all()
        finally:
            held.clear()
            torch.cuda.empty_cache()
        pf.pf_last_error(c)
        pf.pf_run_host(c, 1, reads, reads, 2, length=m, chunk_pairs=chunk, out=out)
        assert (out[0] == 1).all() and not out[1].any() and not out[2].any()
    finally:
        pf.pf_destroy(c)


@pytest.mark.parametrize("what", ["filter", "tune", "serve", "serve loop"])
def test_kept_slots_make_room_for_other_calls(pf, what):
    """What pf_run_host keeps (two slots of 0.9 GB) is given back where another
    call of the context needs the memory."""
    m, chunk = 8_000, 37_000
    reads = pair_bytes(2 * chunk, m)
    n = {"filter": 45_000_000, "tune": 60_000_000}.get(what, 1)
    lens = torch.full((n,), 32, dtype=torch.int32, device=DEV)
    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    pairs = pf.Pairs(pf.Seqs(word, word, word), pf.Seqs(word, word, word))   # all the same
    acc = torch.zeros(n if what == "filter" else 1, dtype=torch.uint8, device=DEV)
    cnt = torch.zeros(n if what == "filter" else 1, dtype=torch.int16, device=DEV)
    c = pf.pf_create(0)
    try:
        if what == "tune":   # scratch for n pairs is there, the tuner's outputs are not
            a, k = (torch.zeros(n, dtype=t, device=DEV) for t in (torch.uint8, torch.int16))
            pf.pf_filter(c, 1, pairs, lens, None, 0, a, k, n)
            pf.pf_sync(c)
            del a, k
        pf.pf_run_host(c, 1, reads, reads, 2, length=m, chunk_pairs=chunk)
        room = 130_000_000 if what == "tune" else 600_000_000
        held = leave_free(room)
        try:
            assert torch.cuda.mem_get_info()[0] < room + 40_000_000
            if what == "filter":
                pf.pf_filter(c, 1, pairs, lens, None, 0, acc, cnt, n)
                pf.pf_sync(c)
                assert bool((acc == 1).all()) and not bool(cnt.any())
            elif what == "tune":
                pf.pf_tune(c, 1, pairs, lens, 0, reps=1)
            else:
                mode = {"mode": 1} if what == "serve loop" else {}
                pf.pf_serve_start(c, hbm_budget=900_000_000, **mode)
                pf.pf_serve_stop(c)
        finally:
            held.clear()
            torch.cuda.empty_cache()
    finally:
        pf.pf_destroy(c)
