"""Parity of the band kernels (deferred pairs: a score bound per pair, then
the wavefronts on the diagonals that can reach the end within it): lengths
around the class borders, one-sided pairs, unrelated pairs (bounds far from
the optimum's shape), penalties whose rows are deep or beyond the band
kernel's limit, score bounds at and below the optimum, free ends wider and
narrower than the band, graph replays whose contents change class.
Integer results: equal to the oracle bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PENS = [(4, 6, 2), (5, 8, 3), (1, 0, 1), (2, 0, 5), (97, 103, 41)]


@pytest.fixture(scope="module")
def pkg():
    import paper_2204_02085_gb300 as p

    p.load()
    return p


def _pairs(seed):
    """Pairs the short kernels do not take, edges first."""
    rng = np.random.Generator(np.random.PCG64(seed))

    def seq(n):
        return bytes(rng.choice(list(b"ACGT"), size=n).astype(np.uint8)) if n else b""

    def edited(t, k):
        p = bytearray(t)
        for _ in range(k):
            i = int(rng.integers(0, len(p) + 1))
            kind = int(rng.integers(0, 3))
            if kind == 0 and i < len(p):
                p[i] = int(rng.choice(list(b"ACGT")))
            elif kind == 1:
                p[i:i] = seq(int(rng.choice([1, 1, 2, 30])))
            else:
                del p[i:i + int(rng.choice([1, 1, 3, 40]))]
        return bytes(p)

    out = [(b"", seq(300)), (seq(300), b""), (seq(1), seq(260)), (seq(260), seq(1)), (seq(700), seq(90))]
    for n in (256, 271, 272, 511, 1000, 2047, 2048, 2049, 2100):
        t = seq(n)
        out += [(edited(t, n // 25), t), (t, t)]
    out += [(seq(300), seq(310)), (seq(280), seq(400))]  # unrelated
    unit = seq(50)
    out += [(seq(100) + unit * 2 + seq(100), seq(100) + unit * 6 + seq(90))]
    t = seq(900)
    out += [(t[:400] + t[700:], t), (t, t[:100] + seq(300) + t[100:])]  # gaps wider than the bound's window
    return out


def _check(got, want):
    for g, w in zip((got[0], got[1], got[3], got[2]), (want[0], want[1], want[3], want[2])):
        np.testing.assert_array_equal(g, w)


@pytest.mark.parametrize("pen", PENS)
def test_band_pairs(pkg, oracle_mod, pen):
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_pairs(sum(pen)))
    want = oracle_mod.wfa_batch(b, pen, nthreads=8)
    with pkg.Aligner(0, 1 << 30) as al:
        for kw in ({}, {"plain": True}):
            _check(al.align(b, pen, **kw), want)
        s, st, _, _ = al.align(b, pen, score_only=True)
    np.testing.assert_array_equal(s, want[0])
    np.testing.assert_array_equal(st, want[1])


@pytest.mark.parametrize("pen", PENS[:3])
def test_band_score_bounds(pkg, oracle_mod, pen):
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_pairs(7))
    scores = np.sort(oracle_mod.wfa_batch(b, pen, nthreads=8, want_cigar=False)[0])
    with pkg.Aligner(0, 1 << 30) as al:
        for cap in sorted({1, int(scores[len(scores) // 2]), int(scores[len(scores) // 2]) - 1, int(scores[-1])}):
            _check(al.align(b, pen, max_score=cap), oracle_mod.wfa_batch(b, pen, max_score=cap, nthreads=8))


@pytest.mark.parametrize("ends", [(0, 0, 500, 500), (3, 0, 0, 40), (0, 7, 9, 0), (3000, 3000, 3000, 3000)])
def test_band_free_ends(pkg, oracle_mod, ends):
    from paper_2204_02085_gb300 import synth

    b = synth.from_pairs(_pairs(11))
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8, ends=ends)
    with pkg.Aligner(0, 1 << 30) as al:
        al.set_ends_free(*ends)
        _check(al.align(b, (4, 6, 2)), want)


def test_band_graph_contents_change_class(pkg, oracle_mod):
    """A graph captured on medium pairs replayed on contents with a longer
    pair than its shared memory was sized for: the arena kernels finish it."""
    import torch

    from paper_2204_02085_gb300 import synth

    dev = torch.device("cuda:0")
    rng = np.random.Generator(np.random.PCG64(5))
    total, n = 13_000, 12
    base = rng.choice(list(b"ACGT"), size=total).astype(np.uint8)
    with pkg.Aligner(0, 1 << 30) as al:
        bufs = dict(pat=torch.zeros(total, dtype=torch.uint8, device=dev),
                    txt=torch.zeros(total, dtype=torch.uint8, device=dev),
                    plen=torch.zeros(n, dtype=torch.int32, device=dev),
                    tlen=torch.zeros(n, dtype=torch.int32, device=dev),
                    s=torch.zeros(n, dtype=torch.int32, device=dev), st=torch.zeros(n, dtype=torch.int8, device=dev),
                    w=torch.zeros(1 << 14, dtype=torch.int32, device=dev),
                    off=torch.zeros(n + 1, dtype=torch.int64, device=dev))
        for first in (600, 600, 5000, 300):
            lens = np.full(n, 500)
            lens[0] = first
            text = base[:lens.sum()].copy()
            pattern = text.copy()
            pattern[37::41] = ord("A")
            offs = np.concatenate([[0], np.cumsum(lens)[:-1]])
            b = synth.Batch(pattern, offs, lens.astype(np.int32), text, offs, lens.astype(np.int32))
            for name, a in (("pat", pattern), ("txt", text)):
                bufs[name][:len(a)] = torch.from_numpy(a).to(dev)
            for name in ("plen", "tlen"):
                bufs[name].copy_(torch.from_numpy(lens.astype(np.int32)))
            torch.cuda.synchronize()
            rc = al.align_device(bufs["pat"], None, bufs["plen"], bufs["txt"], None, bufs["tlen"], bufs["s"],
                                 bufs["st"], bufs["w"], bufs["off"], graph=True)
            assert rc == pkg.WFA_GPU_OK
            want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
            off = bufs["off"].cpu().numpy()
            _check((bufs["s"].cpu().numpy(), bufs["st"].cpu().numpy(),
                    bufs["w"].cpu().numpy()[:off[-1]].astype(np.uint32), off), want)
