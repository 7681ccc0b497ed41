"""The output spans of the CIGAR compaction, on the CPU: a small program with
the kernel's own arithmetic (nothing is launched) writes every word of a
launch, for calls of one piece and for later chunks of a call, whose words
start past the chunks before them."""
import subprocess

import pytest

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "launch.h"
using namespace wfa;
// pairs, words of each, words before the launch, warps
int main(int, char** v) {
  const int64_t n = atoll(v[1]), each = atoll(v[2]), first = atoll(v[3]), nwarps = atoll(v[4]);
  const CompactSpans s{n, first, first + n * each};
  printf("%d\\n", s.by_words() ? 1 : 0);
  if (!s.by_words()) return 0;
  std::vector<int> written(s.last + 1, 0);
  for (int64_t w = 0; w < nwarps; ++w)
    for (int64_t w0 = s.begin(w); w0 < s.last; w0 += nwarps * CompactSpans::kSpan)
      for (int64_t at = w0; at < w0 + CompactSpans::kSpan && at < s.last; ++at) ++written[at];
  int64_t before = 0, once = 0;
  for (int64_t i = 0; i < s.last; ++i)
    if (i < s.first) before += written[i];
    else once += written[i] == 1;
  printf("%lld %lld\\n", (long long)before, (long long)once);
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    from paper_2204_02085_gb300 import build

    work = tmp_path_factory.mktemp("spans")
    src, exe = str(work / "spans.cu"), str(work / "spans")
    with open(src, "w") as f:
        f.write(PROGRAM)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-cudart", "shared", "-I" + build.INCLUDE,
                        "-I" + build.CSRC, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return lambda *a: [int(x) for x in subprocess.run([exe, *map(str, a)], capture_output=True, text=True,
                                                      check=True).stdout.split()]


@pytest.mark.parametrize("first", [0, 1, 255, 256, 5_000_003])
@pytest.mark.parametrize("n,each", [(1, 65), (1, 10_000), (3, 257), (700, 100)])
@pytest.mark.parametrize("warps", [1, 16, 2432])
def test_spans_cover_the_launch_and_nothing_before_it(ask, first, n, each, warps):
    assert ask(n, each, first, warps) == [1, 0, n * each]


@pytest.mark.parametrize("first", [0, 64, 33_554_433])
def test_short_cigars_are_cut_by_pairs_whatever_lies_before(ask, first):
    """512K pairs of 9 words, after more words than 64 a pair of the chunk."""
    assert ask(1 << 19, 9, first, 16) == [0]
    assert ask(1 << 19, 64, first, 16) == [0]
