"""Parity of the small-call path (up to 4,096 pairs: a warp per pair, one
block for the offsets and one for the CIGAR offsets) on device pointers,
eager and replayed from a graph, against the oracle: one pair, block and item
borders of the scans, the last small batch and the first that is not, mixed
with pairs it defers (longer than its limit), empty pairs and other bytes;
offsets passed or not; a capacity one word short; rejected lengths."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2204_02085_gb300 as p

    p.load()
    return p


def _batch(n, seed):
    from paper_2204_02085_gb300 import synth

    core = synth.uniform_reads(n, 100, 4, seed=seed)
    pairs = [core.pair(i) for i in range(n)]
    extra = synth.random_pairs(4, 505, 900, seed=seed, edit_rate=0.05)
    odd = [(b"", b""), (b"", b"ACGT"), (b"ACGNT", b"ACGTT")] + [extra.pair(i) for i in range(extra.n)]
    for j, p in enumerate(odd[:max(0, n - 1)]):
        pairs[(j * 37 + n // 2) % n] = p
    return synth.from_pairs(pairs)


class _Call:
    def __init__(self, b, cap, offsets):
        import torch

        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
        n = b.n
        self.ins = [t(b.patterns), t(b.pattern_offsets) if offsets else None, t(b.pattern_lengths), t(b.texts),
                    t(b.text_offsets) if offsets else None, t(b.text_lengths)]
        self.s = torch.full((n,), -9, dtype=torch.int32, device="cuda:0")
        self.st = torch.full((n,), 9, dtype=torch.int8, device="cuda:0")
        self.w = torch.zeros(max(cap, 1), dtype=torch.int32, device="cuda:0")
        self.off = torch.full((n + 1,), -1, dtype=torch.int64, device="cuda:0")
        torch.cuda.synchronize()

    def run(self, al, **kw):
        return al.align_device(*self.ins, self.s, self.st, self.w, self.off, **kw)

    def check(self, want):
        np.testing.assert_array_equal(self.s.cpu().numpy(), want[0])
        np.testing.assert_array_equal(self.st.cpu().numpy(), want[1])
        off = self.off.cpu().numpy()
        np.testing.assert_array_equal(off, want[3])
        np.testing.assert_array_equal(self.w.cpu().numpy()[:off[-1]].view(np.uint32), want[2])


@pytest.mark.parametrize("n", [1, 4, 5, 127, 1023, 4095, 4096, 4097])
@pytest.mark.parametrize("graph", [False, True])
def test_small_calls(pkg, oracle_mod, n, graph):
    b = _batch(n, 300 + n)
    want = oracle_mod.wfa_batch(b, (4, 6, 2), nthreads=8)
    cap = int(want[3][-1])
    with pkg.Aligner(0, 1 << 28) as al:
        for offsets in (False, True):
            c = _Call(b, cap, offsets)
            for _ in range(3 if graph else 1):
                assert c.run(al, graph=graph) == pkg.WFA_GPU_OK
                c.check(want)
        short = _Call(b, cap - 1, False)
        if cap > 1:
            assert short.run(al, graph=graph) == pkg.WFA_GPU_ECIGAR_CAPACITY
            assert int(short.off[-1]) == cap
        assert c.run(al, score_only=True) == pkg.WFA_GPU_OK
        np.testing.assert_array_equal(c.s.cpu().numpy(), want[0])
        c.ins[2][n // 2] = -3
        with pytest.raises(pkg.WfaGpuError):
            c.run(al)


@pytest.mark.parametrize("ends", [(0, 0, 40, 40), (5, 9, 0, 3)])
@pytest.mark.parametrize("pen", [(4, 6, 2), (1, 0, 1), (97, 103, 41)])
def test_small_calls_free_ends_and_penalties(pkg, oracle_mod, ends, pen):
    b = _batch(200, 77)
    with pkg.Aligner(0, 1 << 28) as al:
        for e in ((0, 0, 0, 0), ends):
            al.set_ends_free(*e)
            for cap in (0, 24):
                want = oracle_mod.wfa_batch(b, pen, max_score=cap, nthreads=8, ends=e)
                c = _Call(b, int(want[3][-1]), False)
                assert c.run(al, pen=pen, max_score=cap) == pkg.WFA_GPU_OK
                c.check(want)
