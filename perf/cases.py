"""Performance cases: the calls a program makes of this library, with the
sizes, input shapes and options they are made with in earnest.

Inputs are drawn on the GPU from the seed alone: per pair a text of uniform
bases and a pattern that is the text after a number of edit events
(substitution, insertion or deletion, 1/3 each, at uniform positions), the
shape of the read sets the library is for.  A case's fields:

  call       device: Aligner.align_device; graph: the same with graph=True
             (batches repeated in the same buffers); host: the C call on
             page-locked host arrays; serve: requests through a Server
  n          pairs (serve: requests, of batch_lo .. batch_hi pairs each,
             log-uniform)
  len_lo/hi  text length, log-uniform
  rate_lo/hi edit events per base, uniform per pair
  flank      > 0: reads in windows: the pattern is the text's read, and the
             text gets U{0..flank} uniform bases on either side; text ends free
  repeats    share of texts that carry a tandem repeat (a 50-mer, 2-6 times)
  x, o, e    penalties
  offsets    whether the program passes its offset arrays
  score_only scores without CIGARs
  arena_gib  the context's scratch arena (0: the default)
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2204_02085_gb300 as pkg

DEV = "cuda:0"
BASE = dict(call="device", n=0, len_lo=100, len_hi=100, rate_lo=0.04, rate_hi=0.04, flank=0, repeats=0.0, x=4, o=6,
            e=2, offsets=False, score_only=False, arena_gib=0, batch_lo=1, batch_hi=1)


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)

    return [
        # a handful of reads, as an interactive tool or a filter inside
        # another pipeline aligns them: latency only
        case("few_reads", n=37),
        # the paper's workload, 5 million 100 bp pairs at E = 2 % and 4 %:
        # batch after batch through the same device buffers
        case("reads_e2", call="graph", n=5_000_000, rate_lo=0.02, rate_hi=0.02),
        case("reads_e4", call="graph", n=5_000_000),
        # quality-trimmed reads of uneven length, one call per batch, with
        # the offsets of the caller's own layout
        case("reads_trimmed", n=400_001, len_lo=60, len_hi=120, offsets=True),
        # 150 bp sequencer reads, some trimmed
        case("reads_150", n=1_000_000, len_lo=120, len_hi=150, rate_lo=0.01, rate_hi=0.03),
        # edit distance of 100 bp reads (clustering, deduplication)
        case("reads_edit_distance", n=2_000_000, x=1, o=0, e=1),
        # reads placed in the reference windows a seeding step proposed:
        # semi-global (text ends free)
        case("reads_in_windows", n=200_000, rate_lo=0.03, rate_hi=0.03, flank=100, arena_gib=8),
        # reads of very uneven length and divergence
        case("mixed_lengths", call="graph", n=200_000, len_lo=100, len_hi=2000, rate_lo=0.0, rate_hi=0.10, repeats=0.05,
             arena_gib=16),
        # 10 kbp long reads: overlap scores, and full alignments
        case("long_score", n=4_000, len_lo=10_000, len_hi=10_000, rate_lo=0.01, rate_hi=0.05, score_only=True,
             arena_gib=16),
        case("long_cigar", n=2_000, len_lo=10_000, len_hi=10_000, rate_lo=0.01, rate_hi=0.05, arena_gib=16),
        # a file's reads from page-locked host memory and back
        case("host_reads", call="host", n=2_200_000),
        # a service: a burst of requests of uneven size and read length
        case("serving", call="serve", n=48, len_lo=100, len_hi=5000, rate_lo=0.02, rate_hi=0.08, batch_lo=1,
             batch_hi=512, arena_gib=8),
    ]


def draw(rng):
    def logu(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["reads", "reads", "reads", "windows", "mixed", "long", "host", "serve"])
    c = dict(BASE)
    if kind in ("reads", "host"):
        lo = int(logu(30, 250))
        hi = min(255, int(lo * rng.uniform(1.0, 1.4)))
        rate = max(logu(0.005, 0.06), 1.0 / lo)
        c.update(call="host" if kind == "host" else rng.choice(["device", "graph"]), len_lo=min(lo, hi), len_hi=hi,
                 rate_lo=rate * rng.choice([0.0, 1.0]), rate_hi=rate, offsets=rng.random() < 0.5,
                 score_only=rng.random() < 0.2)
        c["x"], c["o"], c["e"] = rng.choice([(4, 6, 2)] * 4 + [(2, 3, 1), (1, 0, 1), (3, 0, 2), (5, 8, 3)])
        # the cost of a pair grows with the square of its edits
        cap = min(2_500_000 if kind == "reads" else 2_200_000, 4e7 / (hi * (1 + (0.4 * hi * rate) ** 2)))
        c["n"] = int(logu(16 if kind == "reads" else 1000, max(2000, cap)))
    elif kind == "windows":
        lo = int(logu(50, 150))
        c.update(n=int(logu(100, 150_000)), len_lo=lo, len_hi=lo, rate_lo=0.0, rate_hi=rng.uniform(0.01, 0.04),
                 flank=rng.randint(20, 100), arena_gib=8, score_only=rng.random() < 0.2)
    elif kind == "mixed":
        c.update(call=rng.choice(["device", "graph"]), n=int(logu(200, 150_000)), len_lo=rng.randint(80, 200),
                 len_hi=rng.randint(500, 2000), rate_lo=0.0, rate_hi=rng.uniform(0.02, 0.10),
                 repeats=rng.choice([0.0, 0.05]), arena_gib=16, score_only=rng.random() < 0.2)
    elif kind == "long":
        lo = int(logu(2_200, 20_000))
        hi = int(lo * rng.uniform(1.0, 1.5))
        rate = rng.uniform(0.01, 0.05)
        cap = min(3_000, 4e8 / (hi * rate) ** 2)
        c.update(n=int(logu(8, max(16, cap))), len_lo=lo, len_hi=hi, rate_lo=0.01, rate_hi=rate, arena_gib=16,
                 score_only=rng.random() < 0.5)
    else:
        c.update(call="serve", n=rng.randint(8, 48), len_lo=100, len_hi=int(logu(300, 5000)), rate_lo=0.02,
                 rate_hi=rng.uniform(0.03, 0.08), batch_hi=int(logu(16, 512)), arena_gib=8)
    return c


# ----------------------------------------------------------------- inputs


def _sizes(c):
    """Pairs of each request (serve; the same for every seed), else the one
    batch."""
    if c["call"] != "serve":
        return [c["n"]]
    rng = np.random.Generator(np.random.PCG64(c["n"]))
    return [int(v) for v in np.exp(rng.uniform(math.log(c["batch_lo"]), math.log(c["batch_hi"] + 1), size=c["n"]))]


def _starts(lengths):
    return torch.cumsum(lengths, 0) - lengths


def _expand(starts, lengths, total):
    """For each element of back-to-back rows: its row and its place in it."""
    row = torch.repeat_interleave(torch.arange(len(lengths), device=DEV), lengths, output_size=total)
    return row, torch.arange(total, device=DEV) - starts[row]


def _inputs(c, seed):
    """Pattern bytes, pattern lengths, text bytes and text lengths (torch,
    GPU), all from the seed."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    n = sum(_sizes(c))

    def ints(hi, size):
        return torch.randint(0, hi, (int(size),), generator=g, device=DEV, dtype=torch.uint8)

    def uni(size):
        return torch.rand(int(size), generator=g, device=DEV, dtype=torch.float64)

    lo, hi = math.log(c["len_lo"]), math.log(c["len_hi"])
    tlen = torch.exp(lo + (hi - lo) * uni(n)).round().to(torch.int64)
    k = ((c["rate_lo"] + (c["rate_hi"] - c["rate_lo"]) * uni(n)) * tlen).round().to(torch.int64)
    total, events = int(tlen.sum()), int(k.sum())
    tstart = _starts(tlen)
    text = ints(4, total)
    if c["repeats"] > 0:
        pick = torch.nonzero(uni(n) < c["repeats"]).flatten()
        unit = ints(4, 50 * len(pick))
        first = (uni(len(pick)) * tlen[pick]).to(torch.int64)
        span = torch.minimum(50 * (2 + ints(5, len(pick)).to(torch.int64)), tlen[pick] - first)
        row, j = _expand(_starts(span), span, int(span.sum()))
        text[tstart[pick][row] + first[row] + j] = unit[50 * row + j % 50]
    # the edit events: base they act on, and kind
    erow = torch.repeat_interleave(torch.arange(n, device=DEV), k, output_size=events)
    at = tstart[erow] + (uni(events) * tlen[erow]).to(torch.int64)
    kind = ints(3, events)
    delta = 1 + ints(3, events)
    edited = text.clone()
    edited.index_add_(0, at[kind == 0], delta[kind == 0])
    edited &= 3
    out = torch.ones(total, dtype=torch.int32, device=DEV)  # bases of the pattern each text base becomes
    keep = torch.ones(total, dtype=torch.bool, device=DEV)
    keep[at[kind == 1]] = False
    out -= (~keep).to(torch.int32)
    ins = at[kind == 2]
    out.index_add_(0, ins, torch.ones(len(ins), dtype=torch.int32, device=DEV))
    ends = torch.cumsum(out, 0, dtype=torch.int64)
    pattern = ints(4, int(ends[-1]))  # inserted bases; the kept ones follow
    pattern[ends[keep] - 1] = edited[keep]
    pend = ends[tstart + tlen - 1]
    plen = pend.clone()
    plen[1:] -= pend[:-1]
    del out, keep, ends, edited, at, kind, delta
    if c["flank"] > 0:
        # the unedited read is the pattern; the text is its edited copy
        # between two flanks
        text, tlen, pattern, plen = pattern, plen, text, tlen
        left = (uni(n) * (c["flank"] + 1)).to(torch.int64)
        right = (uni(n) * (c["flank"] + 1)).to(torch.int64)
        wide = left + tlen + right
        window = ints(4, int(wide.sum()))
        row, j = _expand(_starts(tlen), tlen, int(tlen.sum()))
        window[(_starts(wide) + left)[row] + j] = text
        text, tlen = window, wide
    acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)

    def letters(codes):
        return acgt[codes.to(torch.int32)] if len(codes) < 1 << 26 else torch.cat(
            [acgt[p.to(torch.int32)] for p in codes.split(1 << 26)])

    return letters(pattern), plen.to(torch.int32), letters(text), tlen.to(torch.int32)


def _free(c):
    return 4 * (c["len_hi"] + 2 * c["flank"]) if c["flank"] > 0 else 0


def _runs(c):
    """CIGAR words a pair may take: its score is at most max(x, o + e) an
    edit event, and every two runs cost min(x, o + e)."""
    edits = int(c["rate_hi"] * c["len_hi"] + 1)
    lo, hi = min(c["x"], c["o"] + c["e"]), max(c["x"], c["o"] + c["e"])
    return 2 * (edits * hi // lo) + 1 + (2 if c["flank"] > 0 else 0)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


class State:
    """What the program keeps: inputs, output buffers and the handle."""

    def close(self):
        if getattr(self, "handle", None) is not None:
            self.handle.close()
            self.handle = None

    def __del__(self):
        self.close()


def prepare(case, seed):
    c = dict(BASE, **case)
    s = State()
    s.c = c
    s.pen = pkg.Penalties(c["x"], c["o"], c["e"])
    pat, plen, txt, tlen = _inputs(c, seed)
    n = len(plen)
    poff, toff = _starts(plen.to(torch.int64)), _starts(tlen.to(torch.int64))
    if c["call"] == "serve":
        s.handle = pkg.Server(0, workers=2, memory_budget_bytes=c["arena_gib"] << 30)
        hp, ht, hpl, htl, hpo, hto = (_pinned(t).numpy() for t in (pat, txt, plen, tlen, poff, toff))
        s.batches, i = [], 0
        for size in _sizes(c):
            one = slice(i, i + size)
            s.batches.append(pkg.synth.Batch(hp, hpo[one], hpl[one], ht, hto[one], htl[one]))
            i += size
        s.words = [len(b.pattern_lengths) * _runs(c) for b in s.batches]
        s.cigars = np.zeros(sum(s.words), dtype=np.uint32)
        torch.cuda.synchronize()
        return s
    s.handle = pkg.Aligner(0, scratch_bytes=c["arena_gib"] << 30)
    if c["flank"] > 0:
        s.handle.set_ends_free(text_begin=_free(c), text_end=_free(c))
    cap = 1 if c["score_only"] else max(1, n * _runs(c))
    where = dict(device="cpu", pin_memory=True) if c["call"] == "host" else dict(device=DEV)
    s.out = {"scores": torch.zeros(n, dtype=torch.int32, **where), "status": torch.zeros(n, dtype=torch.int8, **where)}
    s.cigars = s.cigar_offsets = None
    if not c["score_only"]:
        s.out["cigars"] = s.cigars = torch.zeros(cap, dtype=torch.int32, **where)
        s.out["cigar_offsets"] = s.cigar_offsets = torch.zeros(n + 1, dtype=torch.int64, **where)
    s.inputs = [pat, poff if c["offsets"] else None, plen, txt, toff if c["offsets"] else None, tlen]
    if c["call"] == "host":
        s.inputs = [None if t is None else _pinned(t) for t in s.inputs]
    torch.cuda.synchronize()
    return s


def run(s):
    c = s.c
    if c["call"] == "serve":
        ids = [s.handle.submit(b, s.pen, cigar_capacity=w) for b, w in zip(s.batches, s.words)]
        got, at = [s.handle.wait(i)[0] for i in ids], 0
        for g in got:  # the requests' CIGARs one after another
            s.cigars[at:at + len(g[2])] = g[2]
            at += len(g[2])
        return {"scores": np.concatenate([g[0] for g in got]), "status": np.concatenate([g[1] for g in got]),
                "cigars": s.cigars.view(np.int32), "cigar_offsets": np.concatenate([g[3] for g in got])}
    if c["call"] == "host":
        flags = pkg.WFA_GPU_SCORE_ONLY if c["score_only"] else 0
        at = [None if t is None else t.data_ptr() for t in s.inputs]
        rc = pkg.wfa_gpu_align_batch(
            s.handle.ctx, len(s.inputs[2]), *at, s.pen, 0, flags, s.out["scores"].data_ptr(),
            s.out["status"].data_ptr(), None if s.cigars is None else s.cigars.data_ptr(),
            0 if s.cigars is None else s.cigars.numel(),
            None if s.cigar_offsets is None else s.cigar_offsets.data_ptr())
    else:
        rc = s.handle.align_device(*s.inputs, s.out["scores"], s.out["status"], s.cigars, s.cigar_offsets, pen=s.pen,
                                   score_only=c["score_only"], graph=c["call"] == "graph")
    if rc != pkg.WFA_GPU_OK:
        raise RuntimeError(pkg.wfa_gpu_strerror(rc))
    return s.out


def work(case):
    """Bytes of one pass: bases, lengths (and offsets) in; scores, statuses,
    CIGAR offsets and runs out.  The arithmetic is integer work, no flops."""
    c = dict(BASE, **case)

    def log_mean(lo, hi):
        return (hi - lo) / math.log(hi / lo) if hi > lo else float(lo)

    n = c["n"] * (log_mean(c["batch_lo"], c["batch_hi"]) if c["call"] == "serve" else 1)
    length = log_mean(c["len_lo"], c["len_hi"])
    per = 2 * length + c["flank"] + 8 + (16 if c["offsets"] or c["call"] == "serve" else 0) + 5
    if not c["score_only"]:
        per += 8 + 4 * (1 + 2 * length * (c["rate_lo"] + c["rate_hi"]) / 2 + (2 if c["flank"] > 0 else 0))
    return {"bytes": float(n * per), "flops": 0.0}


# ------------------------------------------------------------------ exact


def exact(case, seed):
    """The scores by the textbook dynamic program (row by row, the gap along
    the text as a running minimum), 64-bit integers; the CIGARs have none
    (which of the equally good alignments is this library's own rule)."""
    c = dict(BASE, **case)
    longest = c["len_hi"] * (1 + c["rate_hi"]) + 2 * c["flank"]
    if work(c)["bytes"] * longest > 2e10:
        return None
    pat, plen, txt, tlen = _inputs(c, seed)
    poff, toff = _starts(plen.to(torch.int64)), _starts(tlen.to(torch.int64))
    scores = torch.empty(len(plen), dtype=torch.int64, device=DEV)
    step = max(1, int(5e7 / longest))
    for i in range(0, len(plen), step):
        scores[i:i + step] = _gotoh(c, pat, poff[i:i + step], plen[i:i + step].to(torch.int64), txt, toff[i:i + step],
                                    tlen[i:i + step].to(torch.int64))
    return {"scores": scores, "status": None, "cigars": None, "cigar_offsets": None}


def _gotoh(c, pat, poff, plen, txt, toff, tlen):
    n, m = int(plen.max()), int(tlen.max())
    col = torch.arange(m + 1, device=DEV)
    text = txt[torch.minimum(toff[:, None] + col[None, :m], torch.tensor(len(txt) - 1, device=DEV))]
    first = torch.zeros_like(col) if c["flank"] > 0 else torch.where(col > 0, c["o"] + c["e"] * col, 0)
    h = first.expand(len(plen), m + 1).clone()
    d = torch.full_like(h, 1 << 40)
    got = torch.zeros(len(plen), dtype=torch.int64, device=DEV)

    def take(i):
        last = h.gather(1, tlen[:, None])[:, 0]
        if c["flank"] > 0:
            last = torch.where(col[None, :] <= tlen[:, None], h, 1 << 40).amin(1)
        got[plen == i] = last[plen == i]

    take(0)
    for i in range(1, n + 1):
        d = torch.minimum(d + c["e"], h + (c["o"] + c["e"]))
        letter = pat[torch.clamp(poff + i - 1, max=len(pat) - 1)]
        t = d.clone()
        t[:, 1:] = torch.minimum(t[:, 1:], h[:, :-1] + c["x"] * (text != letter[:, None]))
        best = torch.cummin(t - c["e"] * col, 1).values
        h = t
        h[:, 1:] = torch.minimum(h[:, 1:], best[:, :-1] + c["o"] + c["e"] * col[1:])
        take(i)
    return got
