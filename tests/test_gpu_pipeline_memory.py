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
