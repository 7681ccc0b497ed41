"""The band kernels where their forms and limits lie: parity with the oracle
bit for bit (integer results)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2204_02085_gb300 as p

    p.load()
    return p


def _check(got, want):
    for i in (0, 1, 3, 2):
        np.testing.assert_array_equal(got[i], want[i])


def _windows(count, length, flank, rate, seed):
    """Reads in windows: the text is the edited read between two flanks."""
    from paper_2204_02085_gb300 import synth

    core = synth.random_pairs(count, length, length, seed=seed, edit_rate=rate)
    rng = np.random.Generator(np.random.PCG64(seed))

    def seq(n):
        return rng.choice(list(b"ACGT"), size=int(n)).astype(np.uint8).tobytes()

    return synth.from_pairs([(core.pair(i)[0], seq(rng.integers(flank // 2, flank)) + core.pair(i)[1] +
                              seq(rng.integers(flank // 2, flank))) for i in range(core.n)])


@pytest.mark.parametrize("count,length,flank", [(600, 300, 700), (40, 2100, 700)])
def test_free_ends_on_teams(pkg, oracle_mod, count, length, flank):
    """Rows over more free start diagonals than a warp takes: teams of four
    warps, and of eight where few pairs are long."""
    b = _windows(count, length, flank, 0.04, count)
    ends = (0, 0, 2 * flank + length, 2 * flank + length)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8, ends=ends)
    with pkg.Aligner(0, 1 << 30) as al:
        al.set_ends_free(*ends)
        for _ in range(3):
            s, st, _, _ = al.align(b, (4, 6, 2), score_only=True)
            np.testing.assert_array_equal(s, want[0])
            np.testing.assert_array_equal(st, want[1])
        _check(al.align(b, (4, 6, 2)), want)


@pytest.mark.parametrize("store", ["lane_l191_t12", "lane_l255_t12_i16", "lane_l255_t16_i16"])
def test_forced_store_of_a_longer_class(pkg, oracle_mod, monkeypatch, store):
    """Forced onto a call of shorter reads, whose planes it has no room for, a
    store of a longer class is left out."""
    from paper_2204_02085_gb300 import synth

    b = synth.uniform_reads(5000, 100, 3, seed=9)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        index = next(i for i in range(64) if al.variant_name(i) == store)
    monkeypatch.setenv("WFA_GPU_SHORT_VARIANT", str(index))
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, (4, 6, 2)), want)
        assert al.variant_name(al.timing()["short_variant"]).startswith("lane_")
        assert al.timing()["short_variant"] != index


def test_chunked_call_grows_the_cigar_pool(pkg, oracle_mod, monkeypatch):
    """A host call in chunks whose first chunk's CIGARs outgrow the pool: the
    chunks after it use the one that replaced it.  (300 unrelated bases take
    some 300 words of the pool, which starts with room for 6.3 million.)"""
    import torch

    from paper_2204_02085_gb300 import synth

    chunk, n = 1 << 15, 1 << 21
    monkeypatch.setenv("WFA_GPU_PIPE_CHUNK", str(chunk))
    rng = np.random.Generator(np.random.PCG64(21))
    plen = np.ones(n, np.int32)
    for c in (0, 1, 5):
        plen[c * chunk:c * chunk + 24_000] = 300
    total = int(plen.sum())

    def pinned(a):
        t = torch.empty(a.shape, dtype=torch.from_numpy(a[:0]).dtype, pin_memory=True)
        t.numpy()[...] = a
        return t.numpy()

    letters = np.frombuffer(b"ACGT", np.uint8)
    pat, txt = (pinned(letters[rng.integers(0, 4, size=total)]) for _ in range(2))
    plen = pinned(plen)
    offs = np.cumsum(plen, dtype=np.int64) - plen
    want = oracle_mod.wfa_batch(synth.Batch(pat, offs, plen, txt, offs, plen), (1, 0, 1), nthreads=16)
    cap = int(want[3][-1])
    s, st, off, w = (pinned(np.zeros(k, t)) for k, t in ((n, np.int32), (n, np.int8), (n + 1, np.int64),
                                                         (cap, np.int32)))
    with pkg.Aligner(0, 4 << 30) as al:
        rc = pkg.wfa_gpu_align_batch(al.ctx, n, pat.ctypes.data, None, plen.ctypes.data, txt.ctypes.data, None,
                                     plen.ctypes.data, pkg.Penalties(1, 0, 1), 0, 0, s.ctypes.data, st.ctypes.data,
                                     w.ctypes.data, cap, off.ctypes.data)
    assert rc == pkg.WFA_GPU_OK
    _check((s, st, w.view(np.uint32), off), want)


def test_small_arena_retries_on_the_whole_arena(pkg, oracle_mod):
    """Pairs that outgrow their slices of an arena too small for two one-CTA
    teams get the whole of it before the call gives up."""
    from paper_2204_02085_gb300 import synth

    b = synth.random_pairs(16, 2400, 2400, seed=31, edit_rate=0.06)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
    with pkg.Aligner(0, 4 << 20) as al:
        _check(al.align(b, (4, 6, 2)), want)


@pytest.mark.parametrize("pen,holds", [((4, 6, 1), 20), ((16, 6, 2), 16), ((5, 8, 3), 30)])
def test_store_chosen_holds_the_scores(pkg, oracle_mod, pen, holds):
    """Batches with one pair in twelve above the middle stores and none above
    the largest (its last score, scaled, in `holds`): the store chosen from the
    sample holds every pair."""
    from math import gcd

    from paper_2204_02085_gb300 import synth

    g = gcd(gcd(pen[0], pen[1]), pen[2])
    pool = synth.uniform_reads(60_000, 100, 1, seed=3), synth.uniform_reads(30_000, 100, 2, seed=4)
    score = [oracle_mod.wfa_batch(b, pen, nthreads=16, want_cigar=False)[0] // g for b in pool]
    easy = np.nonzero(score[0] <= 12)[0][:22_000]
    hard = np.nonzero((score[1] > 12) & (score[1] <= holds))[0][:2_000]
    pairs = [pool[0].pair(int(i)) for i in easy] + [pool[1].pair(int(i)) for i in hard]
    order = np.random.default_rng(5).permutation(len(pairs))
    b = synth.from_pairs([pairs[i] for i in order])
    want = oracle_mod.wfa_batch(b, pen, nthreads=16)
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, pen), want)
        assert al.timing()["deferred_pairs"] == 0


def _tiled(b, want, times):
    """The batch repeated, and its results."""
    from paper_2204_02085_gb300 import synth

    pairs = [b.pair(i) for i in range(b.n)] * times
    words = want[3][-1] * np.arange(times, dtype=np.int64)
    off = np.concatenate([(want[3][:-1] + words[:, None]).ravel(), [want[3][-1] * times]])
    return synth.from_pairs(pairs), (np.tile(want[0], times), np.tile(want[1], times), np.tile(want[2], times), off)


def _class_pairs(longest, count, seed, gap=14):
    """Pairs of up to `longest` bases, most with up to two edits: lengths at
    word borders of the bit planes, gaps of up to `gap`, some empty,
    unrelated or with other bytes."""
    rng = np.random.Generator(np.random.PCG64(seed))

    def seq(n):
        return rng.choice(list(b"ACGT"), size=int(n)).astype(np.uint8).tobytes()

    out = [(b"", b""), (b"", seq(5)), (seq(9), b""), (seq(longest), seq(longest)), (seq(longest), seq(longest - 20)),
           (seq(40).lower(), seq(41)), (seq(60) + b"-", seq(61))]
    lens = [128, 129, 159, 160, 161, longest - 32, longest - 31, longest - 1, longest]
    while len(out) < count:
        t = bytearray(seq(rng.choice(lens) if rng.random() < 0.4 else rng.integers(60, longest + 1)))
        p = bytes(t)
        for _ in range(int(rng.integers(0, 3)) if rng.random() < 0.97 else 6):
            i, kind = int(rng.integers(0, len(t))), int(rng.integers(0, 3))
            if kind == 0:
                t[i] = int(rng.choice(list(b"ACGT")))
            elif kind == 1:
                t[i:i] = seq(rng.choice([1, 1, 1, 2, gap]))
            else:
                del t[i:i + int(rng.choice([1, 1, 1, 2, gap]))]
        out.append((p, bytes(t[:longest])))
    return out


@pytest.mark.parametrize("pen,gap", [((4, 6, 2), 14), ((5, 8, 3), 14), ((1, 1, 1), 14), ((1, 0, 1), 14), ((3, 0, 2), 14),
                                     ((1, 0, 1), 3), ((3, 0, 2), 3)])
@pytest.mark.parametrize("longest", [191, 255])
def test_ordered_classes_above_127_bases(pkg, oracle_mod, longest, pen, gap):
    """The ordered kernel's classes of up to 191 and 255 bases, in batches from
    the size on that they take, and in call order below it.  (Under the
    gap-linear model the kernel in call order stores the higher scores: it
    keeps a batch with wide gaps.)"""
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_class_pairs(longest, 5000, longest + sum(pen), gap))
    want = oracle_mod.wfa_batch(b, pen, nthreads=16)
    big, big_want = _tiled(b, want, 106 if pen[1] == 0 else 14)
    with pkg.Aligner(0, 1 << 30) as al:
        _check(al.align(b, pen), want)
        assert al.variant_name(al.timing()["short_variant"]).startswith("g")
        _check(al.align(big, pen), big_want)
        if pen[1] > 0 or gap < 14:
            assert al.variant_name(al.timing()["short_variant"]).startswith("lane_l%d_" % longest)
        s, st, _, _ = al.align(big, pen, score_only=True)
        np.testing.assert_array_equal(s, big_want[0])
        np.testing.assert_array_equal(st, big_want[1])


def test_call_order_where_it_stores_higher_scores(pkg, oracle_mod):
    """Reads of 200 bases with two mismatches under 16/6/2 (scaled score 16):
    the ordered stores end at 14, the kernel in call order holds them."""
    from paper_2204_02085_gb300 import synth

    rng = np.random.Generator(np.random.PCG64(8))
    t = rng.choice(list(b"ACGT"), size=(3000, 200)).astype(np.uint8)
    p = t.copy()
    swap = dict(zip(b"ACGT", b"GTAC"))
    for row in p:
        for i in rng.choice(np.arange(10, 190, 9), size=2, replace=False):
            row[i] = swap[row[i]]
    b = synth.from_pairs([(x.tobytes(), y.tobytes()) for x, y in zip(p, t)])
    want = oracle_mod.wfa_batch(b, (16, 6, 2), nthreads=16)
    assert np.mean(want[0] == 32) > 0.5  # (a mismatch may also be a gap each way)
    big, big_want = _tiled(b, want, 23)
    with pkg.Aligner(0, 1 << 30) as al:
        _check(al.align(big, (16, 6, 2)), big_want)
        assert al.variant_name(al.timing()["short_variant"]) == "g4_l255_c197_i16"
        assert al.timing()["deferred_pairs"] == 0


class _Device:
    """A batch on the device, and room for its results."""

    def __init__(self, b, words):
        import torch

        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
        self.ins = [t(b.patterns), None, t(b.pattern_lengths), t(b.texts), None, t(b.text_lengths)]
        self.s = torch.full((b.n,), -9, dtype=torch.int32, device="cuda:0")
        self.st = torch.full((b.n,), 9, dtype=torch.int8, device="cuda:0")
        self.w = torch.zeros(max(int(words), 1), dtype=torch.int32, device="cuda:0")
        self.off = torch.full((b.n + 1,), -1, dtype=torch.int64, device="cuda:0")
        torch.cuda.synchronize()

    def run(self, al, **kw):
        self.s.fill_(-9)
        self.off.fill_(-1)
        assert al.align_device(*self.ins, self.s, self.st, self.w, self.off, **kw) == 0
        if kw.get("score_only"):
            return self.s.cpu().numpy(), self.st.cpu().numpy()
        off = self.off.cpu().numpy()
        return self.s.cpu().numpy(), self.st.cpu().numpy(), self.w.cpu().numpy()[:off[-1]].view(np.uint32), off


def _substituted(n, length, subs, seed):
    from paper_2204_02085_gb300 import synth

    rng = np.random.Generator(np.random.PCG64(seed))
    t = rng.choice(list(b"ACGT"), size=(n, length)).astype(np.uint8)
    p = t.copy()
    for i in range(n):
        at = rng.choice(length, size=int(rng.integers(0, subs + 1)), replace=False)
        p[i, at] = rng.choice(list(b"ACGT"), size=len(at))
    return synth.from_pairs([(x.tobytes(), y.tobytes()) for x, y in zip(p, t)])


@pytest.mark.parametrize("n", [37, 4096, 6000])
@pytest.mark.parametrize("length", [100, 200])
def test_penalties_beyond_the_band_keep_short_reads(pkg, oracle_mod, n, length):
    """Under a gap open of 41 the band kernels take no pair; reads with a few
    substituted bases stay with the short-read kernels all the same."""
    b = _substituted(n, length, 3, n + length)
    want = oracle_mod.wfa_batch(b, (4, 41, 1), nthreads=16)
    with pkg.Aligner(0, 1 << 28) as al:
        d = _Device(b, want[3][-1])
        for kw in ({}, {"graph": True}, {"graph": True}):
            _check(d.run(al, pen=(4, 41, 1), **kw), want)
            assert al.timing()["deferred_pairs"] == 0
        _check(al.align(b, (4, 41, 1)), want)
        assert al.timing()["deferred_pairs"] == 0


@pytest.mark.parametrize("ends", [(0, 0, 0, 0), (0, 0, 30, 30)])
@pytest.mark.parametrize("pen", [(19, 39, 3), (97, 103, 41), (4, 0, 33)])
def test_penalties_beyond_the_band(pkg, oracle_mod, pen, ends):
    """What the short-read kernels leave under such penalties: medium and long
    pairs on the arena kernels, one call, host and device, graph replays."""
    from paper_2204_02085_gb300 import synth

    parts = [synth.random_pairs(60, 60, 240, seed=1, edit_rate=0.03), synth.random_pairs(20, 300, 900, seed=2, edit_rate=0.04),
             synth.random_pairs(5, 2100, 2600, seed=3, edit_rate=0.02)]
    b = synth.from_pairs([p.pair(i) for p in parts for i in range(p.n)])
    want = oracle_mod.wfa_batch(b, pen, nthreads=16, ends=ends)
    with pkg.Aligner(0, 4 << 30) as al:
        al.set_ends_free(*ends)
        _check(al.align(b, pen), want)
        d = _Device(b, want[3][-1])
        for kw in ({}, {"graph": True}, {"graph": True}, {"score_only": True}):
            got = d.run(al, pen=pen, **kw)
            if "score_only" in kw:
                np.testing.assert_array_equal(got[0], want[0])
            else:
                _check(got, want)


def test_small_replays_time_their_phases(pkg):
    """The phases of a small call, eager and replayed: of a replay, which has
    no host work between them, the alignment is the larger part, and the
    phases make up the call."""
    b = _substituted(4096, 200, 12, 4)
    with pkg.Aligner(0, 1 << 28) as al:
        d = _Device(b, 64 * b.n)
        for i, kw in enumerate(({}, {"graph": True}, {"graph": True}, {"graph": True})):
            d.run(al, timing=True, **kw)
            t = al.timing()
            assert t["deferred_pairs"] == 0
            assert t["align_ms"] > 0 and t["cigar_ms"] > 0
            if i >= 2:  # (the call before captures)
                assert t["align_ms"] > 0.4 * t["total_ms"]
            assert t["align_ms"] + t["general_ms"] + t["cigar_ms"] <= 1.001 * t["total_ms"]


@pytest.mark.parametrize("hard", [0, 1, 40])
def test_timed_calls_run_the_same_kernels(pkg, oracle_mod, hard):
    """WFA_GPU_TIMING only measures: as many kernels as without, with no pair
    deferred, one the sample does not see, and many; the phases make up the
    call."""
    from paper_2204_02085_gb300 import synth

    b = synth.uniform_reads(6000, 100, 2, seed=12)
    pairs = [b.pair(i) for i in range(b.n)]
    unrelated = synth.random_pairs(hard, 100, 100, seed=13) if hard else None
    for j in range(hard):
        pairs[(5990 + 211 * j) % 6000] = unrelated.pair(j)
    b = synth.from_pairs(pairs)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=16)
    with pkg.Aligner(0, 1 << 28) as al:
        d = _Device(b, want[3][-1])
        _check(d.run(al), want)
        launches = al.timing()["kernel_launches"]
        assert al.timing()["deferred_pairs"] == hard
        _check(d.run(al, timing=True), want)
        t = al.timing()
        assert t["kernel_launches"] == launches and t["deferred_pairs"] == hard
        assert t["align_ms"] > 0 and t["cigar_ms"] > 0 and (t["general_ms"] > 0.01) == (hard > 0)
        assert t["h2d_ms"] + t["align_ms"] + t["general_ms"] + t["cigar_ms"] <= 1.001 * t["total_ms"]


def _launches(al):
    return al.timing()["kernel_launches"]


def test_direct_pairs_that_outgrow_their_slice(pkg, oracle_mod):
    """Small calls of unrelated pairs of some 500 bases under 3/0/2: 600 rows of
    ten blocks, more than the 64 KiB a warp gets of 2 MiB, within the whole of
    it."""
    from paper_2204_02085_gb300 import synth

    b = synth.random_pairs(32, 470, 500, seed=41)
    pen = (3, 0, 2)
    want = oracle_mod.wfa_batch(b, pen, nthreads=16)
    count = []
    for arena in (1 << 30, 2 << 20):
        with pkg.Aligner(0, arena) as al:
            d = _Device(b, want[3][-1])
            for kw in ({}, {"graph": True}, {"graph": True}):
                _check(d.run(al, pen=pen, **kw), want)
                count.append(_launches(al))
            assert al.timing()["deferred_pairs"] < 16  # (those whose rows do not fit a warp)
            _check(al.align(b, pen), want)
    assert all(small > big for big, small in zip(count[:3], count[3:]))


@pytest.mark.parametrize("n", [16, 4200])
def test_band_pairs_that_outgrow_their_slice(pkg, oracle_mod, n):
    """Unrelated medium pairs in 4 MiB: more choice bits than a team's 256 KiB;
    eager, replayed and through host memory, the retries lay the CIGARs out
    again."""
    from paper_2204_02085_gb300 import synth

    hard = synth.random_pairs(16, 640, 670, seed=42)
    b = synth.from_pairs([hard.pair(i) for i in range(16)] + [(b"ACGTTG" * 15, b"ACGTTG" * 15)] * (n - 16))
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=16)
    count = []
    for arena in (1 << 30, 4 << 20):
        with pkg.Aligner(0, arena) as al:
            d = _Device(b, want[3][-1])
            for kw in ({}, {"graph": True}, {"graph": True}):
                _check(d.run(al, **kw), want)
                count.append(_launches(al))
            assert al.timing()["deferred_pairs"] == 16
            _check(al.align(b, (4, 6, 2)), want)
    assert all(small > big for big, small in zip(count[:3], count[3:]))


def test_longest_band_pairs(pkg, oracle_mod):
    """Lengths around the band kernels' last two sizes (12,000 and 32,000
    bases), the longest handed to the arena kernels."""
    from paper_2204_02085_gb300 import synth

    pairs = []
    for j, n in enumerate((12_000, 12_001, 31_999, 32_000)):
        b = synth.random_pairs(2, n, n, seed=50 + j, edit_rate=0.004)
        pairs += [(p[:n], t) for p, t in (b.pair(0), b.pair(1))]
    pairs += [(pairs[4][1][:31_990], pairs[4][1]), (pairs[4][1], pairs[4][1][9:])]
    b = synth.from_pairs(pairs)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=10)
    with pkg.Aligner(0, 4 << 30) as al:
        _check(al.align(b, (4, 6, 2)), want)
        s, st, _, _ = al.align(b, (4, 6, 2), score_only=True)
        np.testing.assert_array_equal(s, want[0])
        np.testing.assert_array_equal(st, want[1])


def test_many_long_pairs_on_four_warps(pkg, oracle_mod):
    """More long pairs than blocks of four warps: no blocks of eight, narrow
    pairs a warp each, wide ones on teams of four."""
    from paper_2204_02085_gb300 import synth

    easy = synth.random_pairs(60, 2049, 2300, seed=60, edit_rate=0.01)
    wide = synth.random_pairs(24, 2049, 2300, seed=61, edit_rate=0.18)
    b = synth.from_pairs([easy.pair(i % 60) for i in range(1140)] + [wide.pair(i) for i in range(24)])
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=16)
    with pkg.Aligner(0, 4 << 30) as al:
        _check(al.align(b, (4, 6, 2)), want)
        s, _, _, _ = al.align(b, (4, 6, 2), score_only=True)
        np.testing.assert_array_equal(s, want[0])


@pytest.mark.parametrize("pen", [(10, 3, 2), (9, 1, 2)])
@pytest.mark.parametrize("ends", [(0, 0, 300, 300), (40, 40, 40, 40), (0, 7, 9, 0)])
def test_free_ends_with_dear_mismatches(pkg, oracle_mod, pen, ends):
    """Scores without a wavefront between older gaps (x well above o + 2 e):
    the rows left out there keep gap cells of lower scores."""
    from paper_2204_02085_gb300 import synth

    parts = [synth.random_pairs(80, 1, 300, seed=70, edit_rate=0.05), synth.random_pairs(20, 260, 300, seed=71),
             _windows(60, 200, 120, 0.05, 72)]
    b = synth.from_pairs([p.pair(i) for p in parts for i in range(p.n)])
    want = oracle_mod.wfa_batch(b, pen, nthreads=16, ends=ends)
    with pkg.Aligner(0, 1 << 30) as al:
        al.set_ends_free(*ends)
        _check(al.align(b, pen), want)  # a warp per pair from bytes to CIGAR
        big, big_want = _tiled(b, want, 30)
        _check(al.align(big, pen), big_want)  # the deferred pairs on the band kernels


def test_dear_gaps_reserve_no_more_than_their_bases(pkg, oracle_mod):
    """Under 1/0/31 a gap of 130 bases scores 4,030 and a mismatch 1: the pool's
    room for a CIGAR is bounded by the bases, not by the score alone, and 1,000
    such pairs fit as 20 do (no retry: as many kernels)."""
    from paper_2204_02085_gb300 import synth

    rng = np.random.Generator(np.random.PCG64(80))

    def seq(n):
        return rng.choice(list(b"ACGT"), size=n).astype(np.uint8).tobytes()

    pairs = []
    for _ in range(20):
        t = seq(600)
        pairs.append((t, t[:300] + seq(130) + t[300:]))
    b = synth.from_pairs(pairs)
    want = oracle_mod.wfa_batch(b, (1, 0, 31), nthreads=16)
    big, big_want = _tiled(b, want, 50)
    count = []
    for one, w in ((b, want), (big, big_want)):
        with pkg.Aligner(0, 1 << 30) as al:  # (a context's first call: a retry would grow the pool)
            _check(_Device(one, w[3][-1]).run(al, pen=(1, 0, 31)), w)
            assert al.timing()["deferred_pairs"] == one.n
            count.append(_launches(al))
    assert count[0] == count[1]
