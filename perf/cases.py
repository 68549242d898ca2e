"""The calls whose time is measured: X-drop seed-and-extend through the library's entry points.

The listed cases are the workloads that the library is built for (single
small calls, the 29x genome overlaps at three thresholds, heavy-tailed
lengths, host buffers, resident reads, serving, seed discovery, the
allocation-free call); draw() gives more of the same ranges.  Inputs are
drawn on the GPU with the generators' error model and length laws
(paper_2309_07270_gb300/workloads.py), vectorised so that a preparation
takes a fraction of a second.
"""
import math

import numpy as np
import torch

from paper_2309_07270_gb300 import xdrop as X

SEED_LEN = 17            # planted seed, bases
ERROR = 0.12             # substitutions, deletions and insertions, a third each
TAIL_WORDS = 64          # zero words after the packed reads
DEV = "cuda:0"

# call:   device (align_device), host (align), resident (submit_pairs over
#         resident reads), serve (concurrent requests to a serving context),
#         static (align_static), seeds (find_candidates)
# reads:  template (two noisy copies of one template per pair), genome (all
#         overlaps >= 2 kb of the reads of one genome), uneven (Pareto
#         lengths, a fifth of the pairs unrelated)
BASE = dict(call="device", reads="template", pairs=0, len_lo=2000, len_hi=4000, genome=0,
            coverage=29.0, rc=0.0, requests=0, match=1, mismatch=-1, gap=-1, x=50, accept=False,
            k=31, lo=20, hi=50, error=ERROR)


def listed():
    return [
        # a handful of short reads: the latency of one call
        _case("tiny64_x20", pairs=64, len_lo=0, len_hi=200, x=20),
        # one small batch of long reads: the latency of its longest extension
        _case("template200_x50", pairs=200),
        # all overlaps of a 4.6 Mb genome at 29x (E. coli): the assembly batch
        _case("genome29x_x50", reads="genome", genome=4_600_000),
        # the same at a generous threshold: wide bands
        _case("genome29x_x100", reads="genome", genome=4_600_000, x=100),
        # the same at a tight threshold: narrow bands
        _case("genome29x_x15", reads="genome", genome=4_600_000, x=15),
        # a million pairs of very uneven lengths, then the acceptance test and the best seed
        _case("uneven1m_x50", reads="uneven", pairs=1_000_000, accept=True),
        # end to end from host buffers, half of the pairs on the reverse strand
        _case("host_genome29x_rc_x50", call="host", reads="genome", genome=2_000_000, rc=0.5),
        # a batch of 10,000 pairs against resident reads
        _case("resident10k_x50", call="resident", reads="genome", genome=1_000_000, pairs=10_000,
              rc=0.5),
        # 25 producers with 3 requests each of 1,000 to 20,000 pairs, served together
        _case("serve75_x50", call="serve", reads="genome", genome=1_000_000, requests=75),
        # candidate pairs of a 1 Mb genome's reads at 29x, 1% errors
        _case("seeds_genome1m_k31", call="seeds", reads="genome", genome=1_000_000, error=0.01),
        # a scoring in which a mismatch costs more than two gaps
        _case("template500_2_3_1_x30", pairs=500, match=2, mismatch=-3, gap=-1, x=30),
        # the allocation-free call on a small batch
        _case("static64_x50", call="static", pairs=64),
    ]


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["device", "device", "device", "device", "host", "resident", "serve",
                       "static", "seeds"])
    x = _log_int(rng, 10, 120)
    if call == "seeds":
        err = rng.choice([0.01, 0.03])
        return _case(call="seeds", reads="genome", genome=_log_int(rng, 30_000, 900_000),
                     coverage=float(rng.randint(20, 35)), error=err, k=rng.choice([17, 21, 31]),
                     lo=rng.randint(2, 20), hi=rng.randint(30, 50))
    if call == "static":
        lo = _log_int(rng, 20, 1500)
        return _case(call="static", pairs=_log_int(rng, 1, 200), len_lo=lo,
                     len_hi=lo + _log_int(rng, 1, 1500), x=x)
    if call == "serve":
        return _case(call="serve", reads="genome", genome=_log_int(rng, 200_000, 1_000_000),
                     requests=rng.randint(15, 60), x=x)
    if call in ("host", "resident"):
        return _case(call=call, reads="genome", genome=_log_int(rng, 100_000, 1_500_000),
                     pairs=_log_int(rng, 1_000, 50_000), coverage=float(rng.randint(10, 35)),
                     rc=rng.choice([0.0, 0.3, 0.5]), x=x)
    reads = rng.choice(["template", "template", "genome", "uneven"])
    m, mm, g = rng.choice([(1, -1, -1)] * 4 + [(2, -3, -2), (5, -4, -3), (1, -2, -1),
                                                (2, -3, -1), (1, 0, -1)])
    if reads == "genome":
        return _case(reads="genome", genome=_log_int(rng, 100_000, 3_000_000),
                     coverage=float(rng.randint(10, 35)), x=x)
    if reads == "uneven":
        return _case(reads="uneven", pairs=_log_int(rng, 1_001, 500_000), x=x,
                     accept=rng.random() < 0.5)
    lo = _log_int(rng, 1, 5_000)
    return _case(pairs=_log_int(rng, 1, 3_000), len_lo=lo, len_hi=lo + _log_int(rng, 1, 5_000),
                 match=m, mismatch=mm, gap=g, x=x * m)


# ---------------------------------------------------------------- inputs


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _segments(lens):
    """Owner and offset inside it of every element of consecutive segments."""
    owner = torch.repeat_interleave(torch.arange(len(lens), device=DEV), lens)
    start = torch.cumsum(lens, 0) - lens
    return owner, torch.arange(int(lens.sum()), device=DEV) - start[owner], start


def _copies(g, pool, start, lens, noisy, protect, error, flip=None):
    """Noisy copies of the pool's segments [start, start + lens), packed.

    protect: the first of SEED_LEN error-free template bases per read, or
    None.  Returns the packed words, read offsets and lengths (tensors), the
    read position of every template base, the template bases copied exactly
    with no insertion before them (clean), and each read's first template
    base in those arrays."""
    owner, off, first = _segments(lens)
    base = pool[start[owner] + off]
    u = torch.rand(off.numel(), generator=g, device=DEV)
    e = error / 3
    free = ~noisy[owner]
    if protect is not None:
        p = protect[owner]
        free |= (off >= p) & (off < p + SEED_LEN)
    u[free] = 1.0
    sub, dele, ins = u < e, (u >= e) & (u < 2 * e), (u >= 2 * e) & (u < 3 * e)
    shift = torch.randint(1, 4, (off.numel(),), generator=g, device=DEV, dtype=torch.uint8)
    base = torch.where(sub, (base + shift) & 3, base)
    count = 1 - dele.to(torch.int64) + ins.to(torch.int64)
    end = torch.cumsum(count, 0)
    total = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), end])
    head = total[first]
    rlen = total[first + lens] - head
    pos = end - 1 - head[owner]
    roff = (rlen + 15) // 16 * 16
    roff = torch.cumsum(roff, 0) - roff
    words = int((roff[-1] + rlen[-1] + 15) // 16) + TAIL_WORDS

    def place(at, read):  # buffer position of read base `at`
        if flip is not None:
            at = torch.where(flip[read], rlen[read] - 1 - at, at)
        return roff[read] + at

    buf = torch.zeros(words * 16, dtype=torch.uint8, device=DEV)
    kept = ~dele
    value = base if flip is None else torch.where(flip[owner], 3 - base, base)
    buf[place(pos[kept], owner[kept])] = value[kept]
    extra = torch.randint(0, 4, (int(ins.sum()),), generator=g, device=DEV, dtype=torch.uint8)
    buf[place(pos[ins] - 1, owner[ins])] = extra
    packed = torch.zeros(words, dtype=torch.int64, device=DEV)
    for q in range(16):
        packed |= buf[q::16].to(torch.int64) << (2 * q)
    clean = ~(sub | dele)
    return packed, roff, rlen, pos, clean, ins, first


def _to_host(packed, roff, rlen):
    return (packed.cpu().numpy().astype(np.uint32), roff.cpu().numpy().astype(np.uint64),
            rlen.cpu().numpy().astype(np.uint32))


def _pairs(a, b, sa, sb):
    out = np.zeros(len(a), X.PAIR_DTYPE)
    for name, v in (("a", a), ("b", b), ("seed_a", sa), ("seed_b", sb)):
        out[name] = v.cpu().numpy() if isinstance(v, torch.Tensor) else v
    out["seed_len"] = SEED_LEN
    return out


def _pareto(rng, n, xm=100.0, alpha=1.5, cap=50_000):
    u = rng.random(n) * (1.0 - (xm / cap) ** alpha)
    return np.maximum((xm * (1.0 - u) ** (-1.0 / alpha)).astype(np.int64), SEED_LEN)


def _planted(case, seed):
    """template and uneven: reads 2p and 2p + 1 share one planted seed."""
    rng, g, n = np.random.default_rng(seed), _generator(seed), case["pairs"]
    true = np.ones(n, bool)
    if case["reads"] == "uneven":
        true = rng.random(n) < 0.8
        la = _pareto(rng, n)
        lb = np.where(true, la, _pareto(rng, n))
    else:
        la = lb = rng.integers(case["len_lo"], case["len_hi"] + 1, n) + (
            SEED_LEN if case["len_lo"] < SEED_LEN else 0)
    pa = (rng.random(n) * (la - SEED_LEN + 1)).astype(np.int64)
    pb = np.where(true, pa, (rng.random(n) * (lb - SEED_LEN + 1)).astype(np.int64))
    # a true pair's reads copy one template; an unrelated pair's have one each
    tl = np.stack([la, np.where(true, 0, lb)], 1).reshape(-1)
    ts = np.cumsum(tl) - tl
    start = np.stack([ts[0::2], np.where(true, ts[0::2], ts[1::2])], 1).reshape(-1)
    lens = np.stack([la, lb], 1).reshape(-1)
    prot = np.stack([pa, pb], 1).reshape(-1)
    t = [torch.from_numpy(v).to(DEV) for v in (start, lens, prot, np.repeat(true, 2))]
    pool = torch.randint(0, 4, (int(tl.sum()),), generator=g, device=DEV, dtype=torch.uint8)
    kmer = torch.randint(0, 4, (n, SEED_LEN), generator=g, device=DEV, dtype=torch.uint8)
    at = (t[0] + t[2]).reshape(n, 2)
    step = torch.arange(SEED_LEN, device=DEV)
    for side in (0, 1):  # the same bases twice for a true pair
        pool[at[:, side, None] + step] = kmer
    packed, roff, rlen, pos, _, _, first = _copies(g, pool, t[0], t[1], t[3], t[2], case["error"])
    seed_at = pos[first + t[2]]
    ids = np.arange(n)
    return (*_to_host(packed, roff, rlen), _pairs(2 * ids, 2 * ids + 1, seed_at[0::2], seed_at[1::2]))


def _read_layout(rng, case):
    """Lognormal lengths (mean 10 kb, sd 6 kb, at least 1 kb), uniform starts."""
    G = case["genome"]
    n = max(int(math.ceil(case["coverage"] * G / 10_000)), 2)
    s2 = math.log(1.0 + 0.36)
    lens = rng.lognormal(math.log(10_000) - s2 / 2, math.sqrt(s2), n)
    while (lens < 1000).any():
        bad = lens < 1000
        lens[bad] = rng.lognormal(math.log(10_000) - s2 / 2, math.sqrt(s2), int(bad.sum()))
    lens = np.minimum(lens.astype(np.int64), G)
    return rng.integers(0, G - lens + 1), lens


def _overlaps(start, lens, least=2000):
    order = np.argsort(start, kind="stable")
    s, end = start[order], (start + lens)[order]
    hi = np.searchsorted(s, end - least, side="right")
    cnt = np.maximum(hi - np.arange(len(s)) - 1, 0)
    ra = np.repeat(np.arange(len(s)), cnt)
    rb = ra + 1 + np.arange(len(ra)) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    keep = np.minimum(end[ra], end[rb]) - s[rb] >= least
    return order[ra[keep]], order[rb[keep]]


def _pair_count(case):
    """Pairs of a genome case: the number asked for, or 0.97 of the overlaps
    that such a layout has on average (both reads stored flipped: left out)."""
    return case["pairs"] or int(0.97 * _overlap_count(case) * (1 - case["rc"] ** 2))


def _overlap_count(case):
    # overlaps of >= 2 kb hold about 0.505 coverage bases per read base, 6,230 on average
    return case["coverage"] ** 2 * case["genome"] * 0.505 / 6_230


def _genome_reads(case, seed, flip_frac=0.0):
    rng, g = np.random.default_rng(seed), _generator(seed)
    start, lens = _read_layout(rng, case)
    pool = torch.randint(0, 4, (case["genome"],), generator=g, device=DEV, dtype=torch.uint8)
    flip = torch.from_numpy(rng.random(len(lens)) < flip_frac).to(DEV) if flip_frac else None
    noisy = torch.ones(len(lens), dtype=torch.bool, device=DEV)
    made = _copies(g, pool, torch.from_numpy(start).to(DEV), torch.from_numpy(lens).to(DEV), noisy,
                   None, case["error"], flip)
    return rng, start, lens, flip, made


def _genome_pairs(case, seed):
    """Every overlapping pair, seeded by the clean window nearest its middle;
    with rc, that fraction of the reads is stored reverse-complemented and
    the pairs of two strands carry the reverse-strand flag."""
    rng, start, lens, flip, made = _genome_reads(case, seed, case["rc"])
    packed, roff, rlen, pos, clean, ins, first = made
    a, b = _overlaps(start, lens)
    if flip is not None:  # read a as stored: pairs whose a is flipped swap ends
        fl = flip.cpu().numpy()
        swap = fl[a] & ~fl[b]
        a, b = np.where(swap, b, a), np.where(swap, a, b)
        both = fl[a] & fl[b]
        a, b = a[~both], b[~both]
    ce = torch.cat([torch.zeros(1, dtype=torch.int32, device=DEV),
                    torch.cumsum(~clean, 0, dtype=torch.int32)])
    ci = torch.cat([torch.zeros(1, dtype=torch.int32, device=DEV),
                    torch.cumsum(ins, 0, dtype=torch.int32)])
    ok = torch.zeros(clean.numel(), dtype=torch.bool, device=DEV)
    n = clean.numel() - SEED_LEN + 1
    ok[:n] = ((ce[SEED_LEN:] - ce[:n]) == 0) & ((ci[SEED_LEN:] - ci[1:n + 1]) == 0)
    A, B = torch.from_numpy(a).to(DEV), torch.from_numpy(b).to(DEV)
    st, ln = torch.from_numpy(start).to(DEV), torch.from_numpy(lens).to(DEV)
    lo = torch.maximum(st[A], st[B])
    hi = torch.minimum(st[A] + ln[A], st[B] + ln[B]) - SEED_LEN
    mid = (lo + hi) // 2
    seed_t = torch.full_like(mid, -1)
    for c0 in range(0, 1000, 125):  # nearest first
        todo = torch.nonzero(seed_t < 0).squeeze(1)
        if todo.numel() == 0:
            break
        d = torch.arange(c0, c0 + 125, device=DEV)
        t = mid[todo, None] + torch.stack([d, -d], 1).reshape(1, -1)
        t = torch.minimum(torch.maximum(t, lo[todo, None]), hi[todo, None])
        wa = first[A[todo], None] + t - st[A[todo], None]
        wb = first[B[todo], None] + t - st[B[todo], None]
        hit = ok[wa] & ok[wb]
        k = hit.to(torch.int8).argmax(1)
        got = hit.gather(1, k[:, None]).squeeze(1)
        seed_t[todo[got]] = t[torch.arange(todo.numel(), device=DEV), k][got]
    # the rare pair without a clean window is left out; the count is the case's
    keep = torch.nonzero(seed_t >= 0).squeeze(1).cpu().numpy()
    if case["pairs"]:
        keep = rng.permutation(keep)
    keep = torch.from_numpy(np.resize(keep, _pair_count(case))).to(DEV)
    A, B, t = A[keep], B[keep], seed_t[keep]
    sa, sb = pos[first[A] + t - st[A]], pos[first[B] + t - st[B]]
    bid = B.clone()
    if flip is not None:  # positions of a flipped b are those of its reverse complement
        bid[flip[B]] |= X.XDROP_PAIR_RC
    return (*_to_host(packed, roff, rlen), _pairs(A, bid, sa, sb))


class _State:
    """Inputs and the context of one case; the context ends with the state."""

    def __init__(self, case):
        self.case = case
        self.sc = X.scoring(case["match"], case["mismatch"], case["gap"], case["x"])
        self.al = None

    def __del__(self):
        if self.al is not None:
            self.al.close()


_server = {}  # the one serving context: a server keeps its read set, requests differ


def _serving(case):
    key = (case["genome"], case["coverage"], case["error"])
    if _server.get("key") != key:
        if _server:
            _server["al"].close()
            _server.clear()
        packed, roff, rlen, pairs = _genome_pairs(case, 7)
        al = X.Aligner(device=0, mode=X.XDROP_MODE_SERVE)
        X.xdrop_load_reads(al.ctx, packed, roff, rlen)
        _server.update(key=key, al=al, pool=pairs)
    return _server["al"], _server["pool"]


def _request_sizes(case):
    return [int(k) for k in np.random.default_rng(25).integers(1_000, 20_001, case["requests"])]


def prepare(case, seed):
    s = _State(case)
    if case["call"] == "seeds":
        s.reads = _to_host(*_genome_reads(case, seed, 0.5)[4][:3])
        s.al = X.Aligner(device=0)
        return s
    if case["call"] == "serve":
        al, pool = _serving(case)
        s.ctx = al.ctx
        rng, size = np.random.default_rng(seed), _request_sizes(case)
        s.requests = [np.ascontiguousarray(pool[rng.integers(0, len(pool), k)]) for k in size]
        return s
    s.reads = _genome_pairs(case, seed) if case["reads"] == "genome" else _planted(case, seed)
    if case["call"] in ("device", "static"):
        s.dev = X.DeviceInputs(*s.reads, device=DEV)
        s.longest = int(s.reads[2].max())
    if case["call"] != "static":
        s.al = X.Aligner(device=0)
    if case["call"] == "resident":
        X.xdrop_load_reads(s.al.ctx, *s.reads[:3])
    torch.cuda.synchronize()
    return s


def run(s):
    case, sc = s.case, s.sc
    if case["call"] == "device":
        out = s.al.align_device(s.dev, sc)
        if not case["accept"]:
            return out
        return [out, s.al.accept_device(s.dev, sc), s.al.best_seeds_device(s.dev, sc.match)]
    if case["call"] == "host":
        return s.al.align(*s.reads, sc).view(np.int32)
    if case["call"] == "resident":
        out = np.zeros(len(s.reads[3]), X.RESULT_DTYPE)
        X.xdrop_sync(s.al.ctx, X.xdrop_submit_pairs(s.al.ctx, s.reads[3], sc, out))
        return out.view(np.int32)
    if case["call"] == "serve":
        out = np.zeros(sum(map(len, s.requests)), X.RESULT_DTYPE)
        parts = np.split(out, np.cumsum([len(p) for p in s.requests])[:-1])
        tickets = [X.xdrop_submit_pairs(s.ctx, p, sc, o) for p, o in zip(s.requests, parts)]
        for t in tickets:
            X.xdrop_sync(s.ctx, t)
        return out.view(np.int32)
    if case["call"] == "static":
        d = s.dev
        X.xdrop_align_static(d.packed.data_ptr(), d.packed.numel(), d.read_off.data_ptr(),
                             d.read_len.data_ptr(), d.read_len.numel(), d.pairs.data_ptr(),
                             d.n_pairs, sc, s.longest, d.out.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        return d.out
    pairs, shared = s.al.find_candidates(*s.reads, k=case["k"], lo=case["lo"], hi=case["hi"])
    # the number of candidates depends on the reads: records in arrays of one size
    rec = np.zeros(2 * int(_overlap_count(case)) + 4096, X.PAIR_DTYPE)
    cnt = np.zeros(len(rec), np.uint32)
    n = min(len(pairs), len(rec))
    rec[:n], cnt[:n] = pairs[:n], shared[:n]
    return [rec.view(np.int32), cnt.view(np.int32), len(pairs)]


# ---------------------------------------------------------------- work


def work(case):
    """Bytes: packed bases, pair records and results, each once.  Operations:
    8 integer operations per cell; a related pair's band holds about 0.85 x /
    max(1, match) cells on each of its (len_a + len_b) anti-diagonals."""
    bases_per_byte = 4.0
    if case["reads"] == "genome":
        total = case["coverage"] * case["genome"]
        pairs = float(sum(_request_sizes(case)) if case["call"] == "serve" else _pair_count(case))
        diagonals = 2 * 6_230 * pairs
        if case["call"] == "seeds":
            # codes written and read once, the nonzeros of A likewise, the candidates out
            return {"bytes": total / bases_per_byte + 16 * total + 8 * total + 24 * pairs,
                    "flops": 20 * total}
    else:
        pairs = float(case["pairs"])
        mean = 290.0 * 0.8 if case["reads"] == "uneven" else (case["len_lo"] + case["len_hi"]) / 2
        diagonals, total = 2 * mean * pairs, 2 * mean * pairs
    band = 0.85 * case["x"] / max(1, case["match"]) + 1
    return {"bytes": total / bases_per_byte + 48 * pairs, "flops": 8 * band * diagonals}


# ---------------------------------------------------------------- exact


def _unpack(words, off, n):
    w = words[off // 16:(off + n + 15) // 16 + 1].astype(np.int64)
    c = (w[:, None] >> (2 * np.arange(16))[None, :]) & 3
    return c.reshape(-1)[:n]


def _extend(seqs, sc):
    """Score and end of every extension (a, b), in 64-bit integers, all
    extensions together, one anti-diagonal a step, cells indexed by i."""
    none = -(1 << 40)
    m = torch.tensor([len(a) for a, _ in seqs], device=DEV)[:, None]
    n = torch.tensor([len(b) for _, b in seqs], device=DEV)[:, None]
    M, N = int(m.max()), int(n.max())

    def table(k, width):
        t = np.full((len(seqs), width + 1), 4 + k, np.int64)
        for row, s in zip(t, seqs):
            row[1:len(s[k]) + 1] = s[k]
        return torch.from_numpy(t).to(DEV)
    a, b = table(0, M), table(1, N)
    i = torch.arange(M + 1, device=DEV)[None, :]
    h1 = torch.full((len(seqs), M + 1), none, dtype=torch.int64, device=DEV)
    h1[:, 0] = 0
    h2 = torch.full_like(h1, none)
    best = torch.zeros(len(seqs), 1, dtype=torch.int64, device=DEV)
    bi, bd = torch.zeros_like(best), torch.zeros_like(best)
    running = torch.ones_like(best, dtype=torch.bool)
    was_dead = torch.zeros_like(running)
    edge = torch.full((len(seqs), 1), none, dtype=torch.int64, device=DEV)
    for d in range(1, M + N + 1):
        j = d - i
        inside = (j >= 0) & (j <= n) & (i <= m) & running
        s = torch.where(a == torch.gather(b, 1, j.clamp(0, N).expand_as(a)), sc[0], sc[1])
        up = torch.cat([edge, h1[:, :-1]], 1)
        diag = torch.cat([edge, h2[:, :-1]], 1) + s
        r = torch.maximum(torch.maximum(up, h1) + sc[2], diag)
        r = torch.where(inside & (r >= best - sc[3]), r, none)
        top = r.max(1, keepdim=True).values
        better = top > best
        if bool(better.any()):
            at = torch.where(r == top, i, M + 1).min(1, keepdim=True).values
            bi, bd = torch.where(better, at, bi), torch.where(better, d, bd)
            best = torch.where(better, top, best)
        dead = top == none
        running &= ~(dead & was_dead)
        was_dead = dead
        if d % 64 == 0 and not bool(running.any()):
            break
        h2, h1 = h1, r
    return torch.cat([best, bi, bd - bi], 1).cpu().numpy()


def exact(case, seed):
    if case["reads"] != "template" or case["call"] not in ("device", "static"):
        return None
    longest = case["len_hi"] + SEED_LEN
    if 4.0 * case["pairs"] * longest * longest > 4e10:
        return None
    words, off, lens, pairs = _planted(case, seed)
    seqs = []
    for p in pairs:
        a, b = (_unpack(words, int(off[r]), int(lens[r])) for r in (p["a"], p["b"]))
        sa, sb, k = int(p["seed_a"]), int(p["seed_b"]), int(p["seed_len"])
        seqs += [(a[:sa][::-1], b[:sb][::-1]), (a[sa + k:], b[sb + k:])]
    e = _extend(seqs, (case["match"], case["mismatch"], case["gap"], case["x"]))
    left, right = e[0::2], e[1::2]
    out = np.zeros((len(pairs), 7), np.int32)
    out[:, 0], out[:, 3] = left[:, 0], right[:, 0]
    for c, name in ((1, "seed_a"), (2, "seed_b")):
        out[:, c] = pairs[name].astype(np.int64) - left[:, c]
        out[:, 3 + c] = pairs[name].astype(np.int64) + SEED_LEN + right[:, c]
    return torch.from_numpy(out.reshape(-1))
