// lane_band.cu -- the ordering pass and the lane kernel over the diagonals
// within the pairs' bounds (lane_band.cuh): kernels, plans and launchers.
#include <algorithm>
#include <cstring>

#include "lane_band.cuh"
#include "launch.h"

namespace wfa {

namespace {

constexpr int kLaneBandWarps = 2;              // of a block: small blocks fill an SM's shared memory best
constexpr int kLaneBandSmem = 96 * 1024;       // more than any variant asks for

// The lane kernels' ordering pass: a block per group of pairs
// (lane_band.cuh).
template <int LMAX, int GROUP, int PER>
__global__ void __launch_bounds__(GROUP / PER, LMAX <= 127 && GROUP == 512 ? 4 : GROUP >= 512 ? 2 : 1)
    lane_order_kernel(const AlignArgs a, int cap, int walk) {
  extern __shared__ __align__(16) unsigned char smem[];
  lane_order_body<LMAX, GROUP, PER>(a, cap, walk != 0, smem);
}

// One lane per pair on the ordering pass's output, over the diagonals within
// the pairs' bounds.
template <typename U, int LMAX, int PX, int POE, int PE, int GROUP>
__global__ void __launch_bounds__(32 * kLaneBandWarps) lane_band_kernel(const AlignArgs a, const LaneBand lb) {
  extern __shared__ __align__(16) unsigned char smem[];
  lane_band_body<U, LMAX, PX, POE, PE, GROUP>(a, lb, smem);
}

// Pairs of a group of the ordering pass, two a thread.  1,024 where pairs are
// bounded one by one: larger groups sort better (5M pairs at E = 4 %: 2.05 ms
// a call against 2.13 in groups of 512).  512 where they are sorted by end
// diagonal alone, which 512 do as well, in four blocks an SM that wait for
// each other's loads less (E = 2 %: 0.93 ms against 0.96), and above 127
// bases, whose planes are larger.  128, one a thread, for calls of up to 16K
// pairs, whose time is a group's latency.
constexpr int kSmallGroup = 128;
constexpr int64_t kSmallGroupPairs = 1 << 14;
int group_for(int lmax, int64_t n, bool walk) {
  return n <= kSmallGroupPairs ? kSmallGroup : lmax <= 127 && walk ? 1024 : 512;
}

using LaneBandKernel = void (*)(const AlignArgs, const LaneBand);

// The kernel of a sequence class and scaled penalties: compiled in for
// 2/4/1 (4/6/2 and its multiples) and 1/1/1 (the edit distance), else read at
// run time.
LaneBandKernel lane_band_kernel_of(int lmax, int group, int x, int oe, int e) {
  const bool p241 = x == 2 && oe == 4 && e == 1, p111 = x == 1 && oe == 1 && e == 1;
  if (lmax <= 127) {
    if (p241)
      return group == 1024  ? lane_band_kernel<uint8_t, 127, 2, 4, 1, 1024>
             : group == 512 ? lane_band_kernel<uint8_t, 127, 2, 4, 1, 512>
                            : lane_band_kernel<uint8_t, 127, 2, 4, 1, 0>;
    return p111 && group == 512 ? lane_band_kernel<uint8_t, 127, 1, 1, 1, 512>
                                : lane_band_kernel<uint8_t, 127, 0, 0, 0, 0>;
  }
  if (lmax <= 191)
    return p241 ? lane_band_kernel<uint8_t, 191, 2, 4, 1, 0> : lane_band_kernel<uint8_t, 191, 0, 0, 0, 0>;
  return lane_band_kernel<uint16_t, 255, 0, 0, 0, 0>;
}

int sm_count(int device) {
  int v = 0;
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device);
  return v > 0 ? v : 1;
}

template <int LMAX, int GROUP, int PER>
cudaError_t plan_order(int device, int* grid) {
  auto k = lane_order_kernel<LMAX, GROUP, PER>;
  const size_t smem = sizeof(LaneOrderShm<LMAX, GROUP>);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, GROUP / PER, smem);
  if (e != cudaSuccess) return e;
  *grid = sm_count(device) * (per_sm < 1 ? 1 : per_sm);
  return cudaSuccess;
}

template <int LMAX, int GROUP, int PER>
cudaError_t launch_order_as(const AlignArgs& a, int grid, int cap, int walk, cudaStream_t st) {
  lane_order_kernel<LMAX, GROUP, PER><<<grid, GROUP / PER, sizeof(LaneOrderShm<LMAX, GROUP>), st>>>(a, cap, walk);
  return cudaGetLastError();
}

// grid[0], [1], [2]: groups of 1,024 (up to 127 bases), 512 and 128.
template <int LMAX>
cudaError_t plan_orders(int device, int grid[3]) {
  cudaError_t e;
  if constexpr (LMAX <= 127)
    if ((e = plan_order<LMAX, 1024, 2>(device, &grid[0]))) return e;
  if ((e = plan_order<LMAX, 512, 2>(device, &grid[1]))) return e;
  return plan_order<LMAX, kSmallGroup, 1>(device, &grid[2]);
}

template <int LMAX>
cudaError_t launch_order(const AlignArgs& a, const ShortVariant& v, int group, int cap, int walk, cudaStream_t st) {
  const int64_t groups = (a.n + group - 1) / group;
  const int most = v.order_grid[group == 1024 ? 0 : group == 512 ? 1 : 2];
  const int grid = groups < most ? (int)groups : most;
  if constexpr (LMAX <= 127)
    if (group == 1024) return launch_order_as<LMAX, 1024, 2>(a, grid, cap, walk, st);
  return group == 512 ? launch_order_as<LMAX, 512, 2>(a, grid, cap, walk, st)
                      : launch_order_as<LMAX, kSmallGroup, 1>(a, grid, cap, walk, st);
}

}  // namespace

cudaError_t plan_lane_band(int device, ShortVariant* v, int lmax, int store) {
  v->band_smem = kLaneBandWarps * ((size_t)store + 128);
  v->band_store = store;
  v->band_cell = lmax <= 191 ? 1 : 2;
  v->max_len = lmax;
  v->kind = 1;
  const int pens[3][3] = {{2, 4, 1}, {1, 1, 1}, {0, 0, 0}};
  for (int q = 0; q < 3; ++q) {
    for (int group : {kSmallGroup, 512, 1024}) {
      const LaneBandKernel k = lane_band_kernel_of(lmax, group, pens[q][0], pens[q][1], pens[q][2]);
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kLaneBandSmem);
      if (e != cudaSuccess) return e;
      int per_sm = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 32 * kLaneBandWarps, v->band_smem);
      if (e != cudaSuccess) return e;
      v->band_grid[q] = sm_count(device) * (per_sm < 1 ? 1 : per_sm);
    }
  }
  return lmax <= 127   ? plan_orders<127>(device, v->order_grid)
         : lmax <= 191 ? plan_orders<191>(device, v->order_grid)
                       : plan_orders<255>(device, v->order_grid);
}

cudaError_t plan_ordered(int device, ShortVariant* v, int lmax, int store, bool linear, const char* name) {
  *v = ShortVariant{};
  v->name = name;
  v->linear = linear ? 1 : 0;
  return plan_lane_band(device, v, lmax, store);
}

static void lane_band_solve(const AlignArgs& a, const ShortVariant& v, LaneBand* lb) {
  *lb = LaneBand{4, 0, -1, (int)(v.band_smem / kLaneBandWarps), 0, 0u};
  if ((a.pb | a.pe | a.tb | a.te) != 0 ) return;  // global alignment only
  const int X = a.xs, OE = a.oes, E = a.es, R = X > OE ? X : OE, rows = lane_band_rows(X, OE, E);
  if (R > 31 || E > 31) return;
  // scores with a wavefront (bit s), and those after R scores, whose row
  // positions an older row wrote
  uint32_t ex = 1u, gap = 0u;
  for (int s = 1; s < 32; ++s) {
    const bool g = (s >= OE && (ex >> (s - OE) & 1u)) || (s >= E && (gap >> (s - E) & 1u));
    if (g) gap |= 1u << s;
    if (g || (s >= X && (ex >> (s - X) & 1u))) ex |= 1u << s;
  }
  const uint32_t run = ex | ~((1u << R) - 1u);
  int from[kLaneBoundMax + 1], back[kLaneBoundMax + 1], open[kLaneBoundMax + 1], fresh[kLaneBoundMax + 1];
  for (int s = 0; s <= kLaneBoundMax; ++s) {
    lane_band_start(s, OE, E, &from[s], &back[s]);
    lane_band_end(s, OE, E, &open[s], &fresh[s]);
  }
  // the largest bound whose rows and choices fit, with the end diagonals of
  // a warp spread over a few about 0, or any one of them
  for (int T = 0; T <= kLaneBoundMax; ++T) {
    int pitch = 0, words = 0;
    for (int d = 0; d <= T; ++d) {  // (lower end diagonals mirror the higher)
      int lo_all = 1 << 20, hi_all = -(1 << 20), sum = 0;
      for (int s = 0; s <= T; ++s) {
        int lo, hi;
        if (!(run >> s & 1u)) continue;
        lane_band_span(from[s], back[s], open[T - s], fresh[T - s], d ? d : -1, d ? d : 2, &lo, &hi);
        if (lo > hi) continue;
        sum += lane_band_choice_words(hi - lo + 1);
        lo_all = lo < lo_all ? lo : lo_all;
        hi_all = hi > hi_all ? hi : hi_all;
      }
      words = sum > words ? sum : words;
      pitch = hi_all - lo_all + 3 > pitch ? hi_all - lo_all + 3 : pitch;
    }
    if (pitch > kLaneBandWidth + 2) break;
    const long row_bytes = (long)rows * pitch * 32 * v.band_cell;
    const long bits = 128L * words;
    const long masks = (long)(pitch - 2) * lane_plane_words(v.max_len) * 128;
    const long events = 64L * (T / (X < OE ? X : OE) + 1);  // the walk's scratch lies over the rows
    if (masks + row_bytes + bits > v.band_store || events > row_bytes) break;
    lb->pitch = pitch;
    lb->words = words;
    lb->s_store = T;
  }
  lb->run = run;
}

void lane_band_plan(const AlignArgs& a, const ShortVariant& v, LaneBand* lb) {
  // a pure function of these few numbers, 1 to 16 us to work out and asked for
  // some ten times a call: each thread keeps its last answers, the stores of
  // several penalty sets (kept by a hash, most stores of a call shared an
  // entry and were worked out again in every call: 200,000 reads of 100 bases
  // at 0.5 % edits under 5/8/3 245 us a call, now 140; under 4/6/2 162, now 131)
  struct Memo {
    int64_t key[4];
    LaneBand lb;
  };
  constexpr unsigned kMemo = 64;
  static thread_local Memo memo[kMemo] = {};
  static thread_local unsigned oldest = 0;
  const int64_t key[4] = {((int64_t)a.xs << 32) | a.oes, ((int64_t)a.es << 32) | v.band_store,
                          ((int64_t)v.band_smem << 8) | v.band_cell,
                          ((int64_t)v.max_len << 2) | ((a.pb | a.pe | a.tb | a.te) == 0 ? 1 : 2)};
  for (const Memo& mm : memo)
    if (std::memcmp(mm.key, key, sizeof key) == 0) {
      *lb = mm.lb;
      return;
    }
  Memo& mm = memo[oldest++ % kMemo];
  lane_band_solve(a, v, &mm.lb);
  std::memcpy(mm.key, key, sizeof key);
  *lb = mm.lb;
}

// Ordered input only for sequences in device memory (the ordering pass
// reads each pair's bytes with its own loads, which page-locked host memory
// read in place over the link would turn into many small transfers).
bool lane_ordered(const AlignArgs& a, const ShortVariant& v) {
  return a.n > 0 && v.kind == 1 && a.lane_slots && a.lane_words && lane_plane_words(v.max_len) <= a.lane_planes &&
         !a.host_seqs;
}

cudaError_t launch_lane_ordered(const AlignArgs& a, const ShortVariant& v, cudaStream_t st) {
  if (!lane_ordered(a, v)) return cudaErrorInvalidValue;
  LaneBand lb;
  lane_band_plan(a, v, &lb);
  // bounds above the store's mean "deferred" (or over the caller's largest
  // score): the greedy walk stops there
  const int cap = std::max(0, std::min(lb.s_store, a.s_cap));
  const int walk = lb.s_store >= a.lane_sort_min ? 1 : 0;
  const int group = lb.group = group_for(v.max_len, a.n, walk != 0);
  const int64_t groups = (a.n + group - 1) / group;
  const cudaError_t e = v.max_len <= 127   ? launch_order<127>(a, v, group, cap, walk, st)
                        : v.max_len <= 191 ? launch_order<191>(a, v, group, cap, walk, st)
                                           : launch_order<255>(a, v, group, cap, walk, st);
  if (e != cudaSuccess) return e;
  const int64_t need = (groups * group + 32 * kLaneBandWarps - 1) / (32 * kLaneBandWarps);
  const int q = a.xs == 2 && a.oes == 4 && a.es == 1 ? 0 : a.xs == 1 && a.oes == 1 && a.es == 1 ? 1 : 2;
  lane_band_kernel_of(v.max_len, group, a.xs, a.oes, a.es)<<<(unsigned)std::min<int64_t>(v.band_grid[q], need),
                                                      32 * kLaneBandWarps, v.band_smem, st>>>(a, lb);
  return cudaGetLastError();
}

}  // namespace wfa
