"""The host rules of the ordered lane kernel, on the CPU: a small program
linked with the library asks them with made-up arguments (nothing is
launched)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    from paper_2204_02085_gb300 import build

    build.build()
    work = tmp_path_factory.mktemp("rules")

    def run(body):
        src, exe = str(work / "rules.cu"), str(work / "rules")
        with open(src, "w") as f:
            f.write('#include <cstdio>\n#include "launch.h"\nusing namespace wfa;\nint main() {\n' + body + "\n}\n")
        cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-cudart", "shared", "-I" + build.INCLUDE, "-I" + build.CSRC,
               src, "-o", exe, build.OUT, "-Xlinker", "-rpath=" + os.path.dirname(build.OUT)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()

    return run


def test_ordered_only_with_room_for_the_planes(ask):
    """A variant of a longer class than the planes were sized for (a forced
    one) is not run on ordered input, and its launcher refuses it."""
    got = ask("""
      uint32_t w; int2 s;
      for (int room : {127, 191, 255})
        for (int lmax : {127, 191, 255}) {
          AlignArgs a{};
          a.n = 5000; a.xs = 2; a.oes = 4; a.es = 1; a.g = 2;
          a.lane_words = &w; a.lane_slots = &s; a.lane_planes = lane_plane_words(room);
          ShortVariant v{};
          v.kind = 1; v.max_len = lmax;
          const bool ok = lane_ordered(a, v);
          printf("%d %d ", ok ? 1 : 0, short_launches(a, v));
          if (!ok) printf("%d ", launch_lane_ordered(a, v, nullptr) == cudaErrorInvalidValue ? 1 : 0);
        }""")
    yes, no = ["1", "2"], ["0", "1", "1"]
    assert got == yes + no + no + yes + yes + no + yes + yes + yes
