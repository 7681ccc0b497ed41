"""Parity of the lane kernel over the diagonals within each pair's bound
(ordered input), per length class (bytes up to 127 and 191 bases, 16-bit rows
up to 255): lengths at the class borders and at word borders of the bit
planes, end diagonals spread from -14 to 14 so that a warp needs several
passes, bounds above and at the store's, unrelated and empty pairs, other
bytes than A/C/G/T, lower case, batch sizes around the groups; compiled-in
and run-time penalties.  Integer results: equal to the oracle bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PENS = [(4, 6, 2), (1, 0, 1), (3, 0, 2), (5, 8, 3), (16, 6, 2), (97, 103, 41)]


@pytest.fixture(scope="module")
def pkg():
    import paper_2204_02085_gb300 as p

    p.load()
    return p


def _pairs(longest, count, seed):
    rng = np.random.Generator(np.random.PCG64(seed))

    def seq(n):
        return bytes(rng.choice(list(b"ACGT"), size=n).astype(np.uint8)) if n else b""

    lens = sorted({0, 1, 2, 31, 32, 33, 63, 64, 65, longest - 33, longest - 32, longest - 31, longest - 1, longest})
    out = [(b"", b""), (b"", seq(5)), (seq(9), b""), (seq(longest), seq(longest)), (seq(longest), seq(longest - 20)),
           (b"ACGTNACGT" * 3, b"ACGTAACGT" * 3), (seq(40).lower(), seq(41)), (seq(60) + b"-", seq(61)),
           (seq(30), b"\x00" + seq(29))]
    while len(out) < count:
        n = int(rng.choice(lens)) if rng.random() < 0.3 else int(rng.integers(longest // 2, longest + 1))
        p = bytearray(seq(n))
        t = bytearray(p)
        for _ in range(int(rng.integers(0, 6))):
            i = int(rng.integers(0, len(t) + 1))
            kind = int(rng.integers(0, 3))
            if kind == 0 and i < len(t):
                t[i] = int(rng.choice(list(b"ACGT")))
            elif kind == 1:
                t[i:i] = seq(int(rng.choice([1, 1, 2, 7, 14])))
            else:
                del t[i:i + int(rng.choice([1, 1, 2, 7, 14]))]
        out.append((bytes(p), bytes(t[:longest])))
    return out


def _check(got, want):
    for i in (0, 1, 3, 2):
        np.testing.assert_array_equal(got[i], want[i])


@pytest.mark.parametrize("pen", PENS)
@pytest.mark.parametrize("longest", [127, 191, 255])
def test_lane_band(pkg, oracle_mod, longest, pen):
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_pairs(longest, 5000, longest + sum(pen)))
    want = oracle_mod.wfa_batch(b, pen, nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, pen), want)
        s, st, _, _ = al.align(b, pen, score_only=True)
        np.testing.assert_array_equal(s, want[0])
        np.testing.assert_array_equal(st, want[1])


@pytest.mark.parametrize("count", [9, 33, 511, 512, 513, 1024, 1025])
@pytest.mark.parametrize("cap", [0, 1, 16, 24, 34])
def test_lane_band_counts_and_bounds(pkg, oracle_mod, monkeypatch, count, cap):
    from paper_2204_02085_gb300 import synth

    with pkg.Aligner(0, 1 << 28) as al:
        index = next(i for i in range(64) if al.variant_name(i) == "lane_l127_c197")
    monkeypatch.setenv("WFA_GPU_SHORT_VARIANT", str(index))
    b = synth.from_pairs(_pairs(127, count, count + cap))
    want = oracle_mod.wfa_batch(b, (4, 6, 2), max_score=cap, nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, (4, 6, 2), max_score=cap), want)


@pytest.mark.parametrize("store", ["lane_l127_c40", "lane_l127_c104", "lane_l127_t18", "lane_ct241_l127_c64"])
@pytest.mark.parametrize("walk_from", ["0", "99"])
def test_lane_band_stores(pkg, oracle_mod, monkeypatch, store, walk_from):
    """Each store, with and without the greedy bound."""
    from paper_2204_02085_gb300 import synth

    monkeypatch.setenv("WFA_GPU_LANE_SORT_MIN", walk_from)
    b = synth.from_pairs(_pairs(127, 3000, 17))
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        index = next(i for i in range(64) if al.variant_name(i) == store)
    monkeypatch.setenv("WFA_GPU_SHORT_VARIANT", str(index))
    with pkg.Aligner(0, 1 << 28) as al:
        got = al.align(b, (4, 6, 2))
        assert al.variant_name(al.timing()["short_variant"]) == store
        _check(got, want)


@pytest.mark.parametrize("count", [16384, 16385, 17408, 17411])
@pytest.mark.parametrize("pen", [(4, 6, 2), (1, 0, 1), (5, 8, 3)])
@pytest.mark.parametrize("walk_from", ["0", "99"])
def test_lane_band_groups(pkg, oracle_mod, monkeypatch, count, pen, walk_from):
    """The ordering's group sizes: the last batch of small groups, the first of
    512 and 1,024, whole and ragged last groups of each."""
    from paper_2204_02085_gb300 import synth

    monkeypatch.setenv("WFA_GPU_LANE_SORT_MIN", walk_from)
    b = synth.from_pairs(_pairs(127, count, 23))
    want = oracle_mod.wfa_batch(b, pen, nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, pen), want)


@pytest.mark.parametrize("longest", [191, 255])
def test_lane_band_groups_of_wide_classes(pkg, oracle_mod, longest):
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_pairs(longest, 16901, longest))
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
    with pkg.Aligner(0, 1 << 28) as al:
        _check(al.align(b, (4, 6, 2)), want)
