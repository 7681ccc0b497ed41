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
            f.write('#include <cstdio>\n#include <ctime>\n#include "lane_band.cuh"\nusing namespace wfa;\nint main() {\n' + body + "\n}\n")
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


SETUP = """
      AlignArgs a{};
      a.n = 5000; a.xs = 5; a.oes = 11; a.es = 3; a.g = 1;
      auto variant = [](int lmax, int store, int cell) {
        ShortVariant v{};
        v.kind = 1; v.max_len = lmax; v.band_store = store; v.band_cell = cell;
        v.band_smem = 2 * (store + 128);
        return v;
      };
      auto ask = [&](const ShortVariant& v) { LaneBand lb; lane_band_plan(a, v, &lb); return lb; };
"""


def test_plan_is_the_length_class_s_own(ask):
    """Two classes with stores of the same bytes have plans of their own,
    whichever was asked for first: the masks of the longer one leave less room
    for rows.  (127 and 191 bases differ by 64: any table that keeps answers
    by the low bits of the class sees the same entry.)"""
    got = ask(SETUP + """
      for (int first = 0; first < 2; ++first) {
        a.xs = 2 + first;
        const int p = ask(variant(first ? 191 : 127, 12928, 1)).s_store;
        const int q = ask(variant(first ? 127 : 191, 12928, 1)).s_store;
        printf("%d ", first ? q > p : p > q);
      }""")
    assert got == ["1", "1"]


def test_plans_of_a_call_are_worked_out_once(ask):
    """The candidate stores of four penalty sets asked for in turn, as calls
    under them do: after the first round the answers are kept (a plan takes
    tens of microseconds to work out, an answer well under one)."""
    got = ask(SETUP + """
      const int stores[5] = {kLaneStore8, kLaneStore10, kLaneStore12, kLaneStore16, kLaneStore18};
      const int pens[4][3] = {{5, 11, 3}, {3, 4, 2}, {2, 4, 1}, {6, 8, 3}};
      auto round = [&]() {
        int sum = 0;
        for (auto& p : pens)
          for (int store : stores) {
            a.xs = p[0]; a.oes = p[1]; a.es = p[2];
            sum += ask(variant(127, store, 1)).s_store;
          }
        return sum;
      };
      const int first = round();
      timespec t0, t1;
      clock_gettime(CLOCK_MONOTONIC, &t0);
      bool same = true;
      for (int i = 0; i < 500; ++i) same = round() == first && same;
      clock_gettime(CLOCK_MONOTONIC, &t1);
      printf("%d %f", same ? 1 : 0, ((t1.tv_sec - t0.tv_sec) * 1e6 + (t1.tv_nsec - t0.tv_nsec) * 1e-3) / (500 * 20));""")
    assert got[0] == "1"
    assert float(got[1]) < 2.0, got  # us an answer


def test_empty_sequences_have_no_bytes(ask):
    """The ordering pass loads the aligned 16-byte chunks that hold a base: of
    an empty sequence none, wherever its offset points."""
    got = ask("""
      for (int h = 0; h < 16; ++h) {
        int most = 0;
        bool ok = lane_chunks(h, 0) == 0;
        for (int len = 1; len <= 255; ++len) {
          int chunks = 0;
          for (int c = 0; c < 17; ++c) chunks += 16 * c < h + len && 16 * c + 16 > h;
          ok = ok && lane_chunks(h, len) == chunks;
        }
        printf("%d ", ok ? 1 : 0);
      }""")
    assert got == ["1"] * 16
