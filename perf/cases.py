"""Performance cases of the pre-alignment filter: the calls a read mapper makes.

Every case is a batch of read / reference-segment pairs taken through the
public calls of ``paper_1910_03936_gb300``.  The kinds:

  step     ASCII on the device -> pf_pack* x 2 -> pf_filter_verify: the whole
           path of a mapper that keeps its candidates on the GPU
  snake    ASCII on the device -> pf_pack* x 2 -> pf_filter: a mapper that
           aligns elsewhere and wants accept flags and counts only
  filter   pf_filter on planes packed once (a threshold tried on them)
  verify   pf_verify of every pair, no filter before it
  submat   pf_filter_partitioned (SneakySnake on t-column sub-matrices)
  shouji   pf_filter_shouji
  host     pf_run_host: page-locked host ASCII in, results in host memory
  serve    pf_submit of several requests, pf_wait for each

Lengths are 100, 150 and 250 bases (the configurations of the benchmark) and
odd ones near them; thresholds are 0 to 10 % of the length.  Bases are 0.1 % N
and 41 % GC, edits are substitutions, insertions and deletions 0.6/0.2/0.2,
and most candidate locations are wrong ones: a fifth of the pairs is within
its threshold, the rest has up to 60 edits (``mix``), or the number of edits is
uniform (``uniform``).
"""
import math

import numpy as np
import torch

import paper_1910_03936_gb300 as pf

DEV = "cuda:0"
BOTH = pf.PF_SNEAKYSNAKE | pf.PF_GATEKEEPER
GEN_CHUNK = 1 << 20     # pairs generated, and checked, at a time


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # The smallest device call: the candidates of a handful of reads, mixed
        # lengths and thresholds, too few to fill the GPU; launches and latency.
        dict(name="step_mixed_1k", kind="step", n=1_000, length=0, lengths="serving", E=-1,
             deciders=BOTH, edits="mix", tuned=False),
        # Benchmark configuration 1: 100k pairs of 100 bp, one threshold.
        dict(name="snake_100bp_E5_100k", kind="snake", n=100_000, length=100, lengths="fixed", E=5,
             deciders=pf.PF_SNEAKYSNAKE, edits="uniform", tuned=False),
        # A batch of serving requests as it stands on the device: 100/150/250 bp,
        # every pair its own threshold, below the scheduler's small-batch size.
        dict(name="step_mixed_100k", kind="step", n=100_000, length=0, lengths="serving", E=-1,
             deciders=BOTH, edits="mix", tuned=False),
        # The headline workload (150 bp, E = 6, both deciders) at half its
        # benchmark size, tuned once as the benchmark does.
        dict(name="step_150bp_E6_10M", kind="step", n=10_000_000, length=150, lengths="fixed", E=6,
             deciders=BOTH, edits="mix", tuned=True),
        # One threshold of the 150 bp sweep, untuned, SneakySnake alone, on
        # planes that are packed already: the filter by itself.
        dict(name="filter_150bp_E3_4M", kind="filter", n=4_000_000, length=150, lengths="fixed",
             E=3, deciders=pf.PF_SNEAKYSNAKE, edits="mix", tuned=False),
        # An odd read length and a middle threshold, both deciders, untuned.
        dict(name="step_127bp_E10_1500k", kind="step", n=1_500_001, length=127, lengths="fixed",
             E=10, deciders=BOTH, edits="mix", tuned=False),
        # Benchmark configuration 3: 100/150/250 bp, thresholds of 2/5/8 % of
        # the length per pair, the grouped layout, tuned on the batch.
        dict(name="step_mixed_3M", kind="step", n=3_000_000, length=0, lengths="mixed", E=-1,
             deciders=BOTH, edits="mix", tuned=True),
        # Benchmark configuration 4: long reads at the largest threshold in use.
        dict(name="step_250bp_E25_1200k", kind="step", n=1_200_000, length=250, lengths="fixed",
             E=25, deciders=BOTH, edits="uniform", tuned=False),
        # Verification of every pair: what a user without a filter runs.
        dict(name="verify_150bp_E6_2M", kind="verify", n=2_000_000, length=150, lengths="fixed",
             E=6, deciders=0, edits="mix", tuned=False),
        # The thesis's FPGA setting of SneakySnake on sub-matrices.
        dict(name="submat_150bp_E6_2M", kind="submat", n=2_000_000, length=150, lengths="fixed",
             E=6, deciders=0, edits="mix", tuned=False, t=8, y=2),
        # Shouji on the same batch, for the comparison of the deciders.
        dict(name="shouji_150bp_E6_2M", kind="shouji", n=2_000_000, length=150, lengths="fixed",
             E=6, deciders=0, edits="mix", tuned=False),
        # Host buffers in, host buffers out, more than one chunk.
        dict(name="host_150bp_E6_1500k", kind="host", n=1_500_000, length=150, lengths="fixed",
             E=6, deciders=BOTH, edits="mix", tuned=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges, without a name."""
    kind = rng.choice(["step"] * 5 + ["snake", "filter", "filter", "verify", "submat", "shouji",
                                      "host", "serve"])
    c = dict(kind=kind, deciders=0, tuned=False, edits=rng.choice(["mix", "mix", "uniform"]))
    if kind in ("step", "snake", "filter", "host"):
        c["deciders"] = rng.choice([BOTH, BOTH, pf.PF_SNEAKYSNAKE, pf.PF_GATEKEEPER])
    if kind == "serve":
        c.update(lengths="serving", length=0, E=-1, deciders=BOTH, requests=rng.randint(1, 6),
                 n=_log_int(rng, 1_000, 60_000))
        return c
    if kind in ("step", "filter", "host") and rng.random() < 0.4:
        c.update(lengths=rng.choice(["mixed", "serving"]), length=0, E=-1)
        c["n"] = _log_int(rng, 1_000, 2_000_000)
        c["tuned"] = kind == "step" and c["n"] > (1 << 20) and rng.random() < 0.5
        return c
    length = rng.choice([100, 150, 250, rng.randint(60, 260), rng.randint(60, 260)])
    c.update(lengths="fixed", length=length, E=rng.randint(0, length // 10))
    # bounded so that no drawn case costs more than the largest listed one
    top = min(4_000_000, int(6.0e8 / (length * (2 + c["E"]))) * 4)
    c["n"] = _log_int(rng, 1_000, top)
    if kind == "submat":
        c["t"] = rng.choice([4, 8, 16, 32])
        c["y"] = rng.choice([1, 2, c["t"]])
    return c


# ---------------------------------------------------------------------------
# inputs

def _bases(g, shape):
    """ASCII bases: 0.1 % N, 41 % GC."""
    u = torch.rand(shape, generator=g, device=DEV)
    b = torch.full(shape, ord("T"), dtype=torch.uint8, device=DEV)
    b[u < 0.704] = ord("A")
    b[u < 0.409] = ord("G")
    b[u < 0.205] = ord("C")
    b[u < 0.001] = ord("N")
    return b


def _shapes(case, g, n):
    """Per-pair lengths and thresholds."""
    if case["lengths"] == "fixed":
        return (torch.full((n,), case["length"], dtype=torch.int32, device=DEV),
                torch.full((n,), case["E"], dtype=torch.int16, device=DEV))
    u = torch.rand(n, generator=g, device=DEV)
    v = torch.rand(n, generator=g, device=DEV)
    if case["lengths"] == "mixed":  # .4/.4/.2, 2/5/8 %
        m = torch.where(u < 0.4, 100, torch.where(u < 0.8, 150, 250))
        r = torch.where(v < 1 / 3, 2, torch.where(v < 2 / 3, 5, 8))
        e = (m * r + 50) // 100
    else:                           # uniform over the lengths and over 0..10 %
        m = torch.where(u < 1 / 3, 100, torch.where(u < 2 / 3, 150, 250))
        e = torch.floor(v * 0.10 * m + 0.5)
    return m.to(torch.int32), e.to(torch.int16)


def _ascii(case, g, lens, E):
    """Reads and references of these pairs, back to back."""
    n = lens.numel()
    M = int(lens.max())
    within = torch.rand(n, generator=g, device=DEV)
    u = torch.rand(n, generator=g, device=DEV)
    e = E.to(torch.float32)
    if case["edits"] == "uniform":
        k = torch.floor(u * (4 * e + 1))
    else:
        k = torch.where(within < 0.2, torch.floor(u * (e + 1)), e + 1 + torch.floor(u * (60 - e)))
    src = _bases(g, (n, M + 64))
    p = torch.rand((n, M), generator=g, device=DEV) * (lens.to(torch.float32) / k.clamp(min=1))[:, None]
    p[k == 0] = 9.0
    sub, ins, dele = p < 0.6, (p >= 0.6) & (p < 0.8), (p >= 0.8) & (p < 1.0)
    shift = torch.cumsum(dele.to(torch.int32) - ins.to(torch.int32), 1)
    at = (torch.arange(M, device=DEV) + shift).clamp_(0, M + 63)
    read = torch.gather(src, 1, at)
    read = torch.where(sub | ins, _bases(g, (n, M)), read)
    ref = src[:, :M]
    if case["lengths"] == "fixed":
        return read.reshape(-1), ref.reshape(-1)
    keep = torch.arange(M, device=DEV) < lens[:, None]
    return read[keep], ref[keep]


def _inputs(case, seed, n):
    """Reads, references, lengths and thresholds of n pairs, on the device."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    lens, E = _shapes(case, g, n)
    parts = [_ascii(case, g, lens[a:a + GEN_CHUNK], E[a:a + GEN_CHUNK])
             for a in range(0, n, GEN_CHUNK)]
    reads = torch.cat([x[0] for x in parts])
    refs = torch.cat([x[1] for x in parts])
    return reads, refs, lens, E


def _offsets(lens):
    off = np.zeros(lens.numel() + 1, dtype=np.int64)
    np.cumsum(lens.cpu().numpy(), out=off[1:])
    return off


# ---------------------------------------------------------------------------
# prepare, run

class _State:
    pass


def _pack(s):
    if s.length:
        pf.pf_pack_fixed(s.ctx, s.reads, s.n, s.length, s.pairs.read)
        pf.pf_pack_fixed(s.ctx, s.refs, s.n, s.length, s.pairs.ref)
    elif s.grouped:
        pf.pf_pack_starts(s.ctx, s.reads, s.byte_off, s.words, s.pairs.read)
        pf.pf_pack_starts(s.ctx, s.refs, s.byte_off, s.words, s.pairs.ref)
    else:
        pf.pf_pack(s.ctx, s.reads, s.byte_off, s.words, s.pairs.read)
        pf.pf_pack(s.ctx, s.refs, s.byte_off, s.words, s.pairs.ref)


def _prepare_host(s, case, seed):
    """Page-locked host buffers, as pf_host_alloc gives them."""
    def host(t):
        a = t.cpu().numpy()
        h = pf.host_empty(a.size, a.dtype)
        h[:] = a.reshape(-1)
        return h
    reads, refs, lens, E = _inputs(case, seed, s.n)
    s.reads, s.refs = host(reads), host(refs)
    s.byte_off = s.E = None
    s.length, s.E_max = case["length"], case["E"]
    if case["lengths"] != "fixed":
        s.length, s.E, s.E_max = 0, host(E), int(E.max())
        s.byte_off = pf.host_empty(s.n + 1, np.int64)
        s.byte_off[:] = _offsets(lens)
    slots = bin(case["deciders"]).count("1")
    s.out = (pf.host_empty(slots * s.n, np.uint8), pf.host_empty(slots * s.n, np.int16),
             pf.host_empty(s.n, np.int32))
    s.ctx = pf.pf_create(0)


def _serve_sizes(case):
    """Requests of one, two thirds, one third... of n pairs."""
    return [max(1, case["n"] * (case["requests"] - i) // case["requests"])
            for i in range(case["requests"])]


def _prepare_serve(s, case, seed):
    s.ctx = pf.pf_create(0)
    s.requests = []
    for i, n in enumerate(_serve_sizes(case)):
        reads, refs, lens, E = _inputs(case, seed * 64 + i, n)
        s.requests.append(pf.Request(case["deciders"], reads.cpu().numpy(), refs.cpu().numpy(),
                                     _offsets(lens), E.cpu().numpy(), pinned=True))
    pf.pf_serve_start(s.ctx, hbm_budget=1 << 31)


def prepare(case, seed):
    s = _State()
    s.case, s.n, s.kind, s.deciders = case, case["n"], case["kind"], case["deciders"]
    if s.kind == "host":
        _prepare_host(s, case, seed)
        return s
    if s.kind == "serve":
        _prepare_serve(s, case, seed)
        return s
    n = s.n
    s.reads, s.refs, s.lens, s.E = _inputs(case, seed, n)
    s.ctx = pf.pf_create(0)
    s.length, s.grouped = case["length"], False
    if case["lengths"] == "fixed":
        # one threshold for the batch goes in as a scalar
        s.E, s.E_max = None, case["E"]
        s.pairs = pf.pack_pairs(s.ctx, s.reads, s.refs, length=s.length)
    else:
        s.E_max = int(s.E.max())
        off = _offsets(s.lens)
        # the grouped layout is the one for large batches of mixed thresholds
        s.grouped = n > (1 << 20)
        s.byte_off = torch.from_numpy(off).to(DEV)
        s.pairs = pf.pack_pairs(s.ctx, s.reads, s.refs, byte_off=off,
                                group_E=s.E.cpu().numpy() if s.grouped else None)
        s.words = s.pairs.read.word_off
    slots = max(1, bin(s.deciders).count("1"))
    s.accept = torch.zeros(slots * n, dtype=torch.uint8, device=DEV)
    s.count = torch.zeros(slots * n, dtype=torch.int16, device=DEV)
    s.dist = torch.zeros(n, dtype=torch.int32, device=DEV)
    if case["tuned"]:
        if s.E is None:
            pf.pf_tune(s.ctx, s.deciders, s.pairs, s.lens, s.E_max, n=min(n, 2_000_000))
        else:
            pf.pf_tune_batch(s.ctx, s.deciders, s.pairs, s.lens, s.E, s.E_max)
    if s.kind in ("filter", "verify", "submat", "shouji"):
        s.reads = s.refs = None      # the planes are the input
    return s


def run(s):
    k = s.kind
    if k == "host":
        acc, cnt, dist = pf.pf_run_host(s.ctx, s.deciders, s.reads, s.refs, s.E_max,
                                        byte_off=s.byte_off, length=s.length, E=s.E, out=s.out)
        return {"accept": acc, "count": cnt, "dist": dist}
    if k == "serve":
        for r in s.requests:
            pf.pf_submit(s.ctx, r)
        for r in s.requests:
            status, _ = pf.pf_wait(s.ctx, r.ticket)
            if status != 0:
                raise pf.PFError(status, "request failed")
        return [{"accept": r.accept, "count": r.count, "dist": r.dist} for r in s.requests]
    if k in ("step", "snake"):
        _pack(s)
    if k == "step":
        pf.pf_filter_verify(s.ctx, s.deciders, s.pairs, s.lens, s.E, s.E_max, s.accept, s.count,
                            s.dist, s.n)
        return {"accept": s.accept, "count": s.count, "dist": s.dist}
    if k == "verify":
        pf.pf_verify(s.ctx, s.pairs, s.lens, s.E, s.E_max, None, None, s.dist, s.n)
        return {"dist": s.dist}
    if k == "submat":
        pf.pf_filter_partitioned(s.ctx, s.pairs, s.lens, s.E, s.E_max, s.case["t"], s.case["y"],
                                 s.accept, s.count, s.n)
    elif k == "shouji":
        pf.pf_filter_shouji(s.ctx, s.pairs, s.lens, s.E, s.E_max, s.accept, s.count, s.n)
    else:
        pf.pf_filter(s.ctx, s.deciders, s.pairs, s.lens, s.E, s.E_max, s.accept, s.count, s.n)
    return {"accept": s.accept, "count": s.count}


# ---------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    """Bytes of one pass.  A base is one byte of ASCII and 3/8 byte of planes;
    a call that packs writes the planes and the next one reads them.  The
    path has no floating-point operations (its work is 32-bit logic)."""
    n = sum(_serve_sizes(case)) if case["kind"] == "serve" else case["n"]
    m = case["length"] if case["lengths"] == "fixed" else \
        (0.4 * 100 + 0.4 * 150 + 0.2 * 250 if case["lengths"] == "mixed" else 500 / 3)
    slots = max(1, bin(case["deciders"]).count("1"))
    per_pair = 0.0 if case["lengths"] == "fixed" else 2.0         # threshold
    if case["kind"] in ("step", "snake", "host", "serve"):
        per_pair += 2 * m + 2 * 0.75 * m
        per_pair += 0.0 if case["lengths"] == "fixed" else 8.0    # offset
    else:
        per_pair += 0.75 * m
    if case["kind"] not in ("host", "serve"):
        per_pair += 4                                             # length
    if case["kind"] != "verify":
        per_pair += 3 * slots
    if case["kind"] in ("step", "verify", "host", "serve"):
        per_pair += 4                                             # distance
    return {"bytes": int(n * per_pair), "flops": 0}


# ---------------------------------------------------------------------------
# the same outputs from plain torch, cell by cell

def _columns(flat, lens, n_as, pad, E):
    """(M + 2E, n) symbols: N as `n_as`, cells outside a sequence `pad`."""
    n, M = lens.numel(), int(lens.max())
    keep = torch.arange(M, device=DEV) < lens[:, None]
    x = torch.full((n, M), pad, dtype=torch.uint8, device=DEV)
    x[keep] = flat
    x[x == ord("N")] = n_as
    out = torch.full((M + 2 * E, n), pad, dtype=torch.uint8, device=DEV)
    out[E:E + M] = x.t()
    return out


def _exact_chunk(case, reads, refs, lens, E):
    """Accept flags and counts per decider and distances of some pairs."""
    kind = case["kind"]
    n, M, e = lens.numel(), int(lens.max()), int(E.max())
    D = 2 * e + 1
    dev = dict(device=DEV)
    # N and vacant cells never match: other symbols on the two sides
    read = _columns(reads, lens, 1, 2, e)
    ref = _columns(refs, lens, 3, 4, 0)
    off = torch.arange(-e, e + 1, **dev)
    live = off.abs()[:, None] <= E[None, :].to(torch.int64)        # (D, n)
    Ei = E.to(torch.int32)
    col = lambda i: read[i:i + D] != ref[i]                        # mismatch cells of column i
    sat = lambda c: torch.minimum(c, Ei + 1)
    zeros = lambda: torch.zeros(n, dtype=torch.int32, **dev)
    out = {}

    def snake(t=0, y=0):
        alive, total, part = live.clone(), zeros(), zeros()
        for i in range(M):
            if t and i % t == 0:
                alive, total, part = live.clone(), total + part, zeros()
            alive &= ~col(i)
            blocked = ~alive.any(0) & (lens > i)
            part += blocked
            if t:
                part.clamp_(max=y)
            alive |= blocked & live
        return total + part

    def gatekeeper():
        h, fc = zeros(), zeros()
        none = torch.zeros((D, n), dtype=torch.bool, **dev)
        mask = lambda i: (col(i) & (lens > i)) if i < M else none
        l2, l1, mid, r1 = none, none, mask(0), mask(1)
        for i in range(M):
            r2 = mask(i + 2)
            h += mid[e]
            amended = mid | (l1 & (r1 | r2)) | (l2 & r1)
            fc += (amended | ~live).all(0) & (lens > i)
            l2, l1, mid, r1 = l1, mid, r1, r2
        return torch.where(h <= Ei, h, fc)

    def shouji():
        ones = zeros()
        order = torch.arange(D, dtype=torch.int16, **dev)[:, None]
        full = torch.ones((D, n), dtype=torch.bool, **dev)
        cells = lambda i: (col(i) | (lens <= i)) if i < M else full
        b = [cells(0), cells(1), cells(2)]
        state = torch.full((n,), 7, dtype=torch.int16, **dev)      # bits c, c+1, c+2
        pop = torch.tensor([bin(v).count("1") for v in range(16)], dtype=torch.int16, **dev)
        for i in range(M):
            b.append(cells(i + 3))
            v = sum(x.to(torch.int16) << j for j, x in enumerate(b))
            cost = (2 * pop[v.long()] + b[0]) * 64 + order
            cost = torch.where(live, cost, 32000)
            best = (cost.min(0).values % 64).long()
            v = v.gather(0, best[None])[0]
            cur = state | 8
            nxt = torch.where(pop[v.long()] < pop[cur.long()], v, cur)
            ones += (nxt & 1) * (lens > i)
            state = nxt >> 1
            b.pop(0)
        return ones

    def distance():
        # band cells k: row j - e + k of column j; rows above the first
        # are |row| away as the boundary is, none of them matches
        k = torch.arange(D, dtype=torch.int32, **dev)[:, None]
        cur = (k - e).abs().expand(D, n).contiguous()
        cur = torch.where(live, cur, 10000)
        dist = cur[e].clone()
        for j in range(M):
            diag = cur + col(j)
            up = torch.cat([cur[1:] + 1, torch.full((1, n), 20000, dtype=torch.int32, **dev)])
            new = torch.minimum(diag, up)
            new = torch.where(live, new, 10000)
            new = torch.cummin(new - k, 0).values + k
            cur = torch.where(live, new, 10000)
            dist = torch.where(lens > j, cur[e], dist)
        return sat(dist)

    counts = []
    if kind == "submat":
        counts.append(sat(snake(case["t"], case["y"])))
    elif kind == "shouji":
        counts.append(sat(shouji()))
    elif kind != "verify":
        if case["deciders"] & pf.PF_SNEAKYSNAKE:
            counts.append(sat(snake()))
        if case["deciders"] & pf.PF_GATEKEEPER:
            counts.append(sat(gatekeeper()))
    if counts:
        out["accept"] = [(c <= Ei).to(torch.uint8) for c in counts]
        out["count"] = [c.to(torch.int16) for c in counts]
    if kind in ("step", "verify", "host", "serve"):
        dist = distance()
        if counts:   # a pair that the first decider rejects is not verified
            dist = torch.where(counts[0] <= Ei, dist, Ei + 1)
        out["dist"] = [dist.to(torch.int32)]
    return out


def _exact_batch(case, seed, n):
    reads, refs, lens, E = _inputs(case, seed, n)
    off = _offsets(lens)
    step = 1 << 18
    parts = [_exact_chunk(case, reads[off[a]:off[min(n, a + step)]],
                          refs[off[a]:off[min(n, a + step)]], lens[a:a + step], E[a:a + step])
             for a in range(0, n, step)]
    # slot after slot, each over the whole batch
    return {key: torch.cat([torch.cat([p[key][s] for p in parts])
                            for s in range(len(parts[0][key]))]) for key in parts[0]}


def exact(case, seed):
    if case["kind"] == "serve":
        return [{k: v.cpu().numpy() for k, v in _exact_batch(case, seed * 64 + i, n).items()}
                for i, n in enumerate(_serve_sizes(case))]
    # every column and diagonal of every pair: some seconds at this many cells
    m = case["length"] if case["lengths"] == "fixed" else 250
    e = case["E"] if case["lengths"] == "fixed" else 25
    if case["n"] * m * (2 * e + 1) > 6e10:
        return None
    out = _exact_batch(case, seed, case["n"])
    if case["kind"] == "host":
        out = {k: v.cpu().numpy() for k, v in out.items()}
        slots = bin(case["deciders"]).count("1")
        out["accept"] = out["accept"].reshape(slots, -1)
        out["count"] = out["count"].reshape(slots, -1)
    return out
