// band_path.cuh -- the gap-affine WFA over the diagonals that can matter:
// pairs the short-read kernels defer (medium and long reads, high scores,
// ends-free calls with wide ends).
//
// A pair is run in two steps.
//
// 1. An upper bound T on its scaled score (BandSearch): the recurrences on a
//    window of 32 diagonals, one per lane, that follows the cell
//    furthest along both sequences.  The score it ends with is the cost of a
//    real alignment, so the optimum is at most T.
// 2. The exact wavefronts (band_forward), but only on diagonals from which
//    the end can still be reached within T: at score s a cell on diagonal k
//    needs at least e * d more, d the distance from k to the nearest end
//    diagonal (a gap in progress is extended for e a diagonal), so row s
//    spans the diagonals with e * d <= T - s among those a start reaches.
//    Every step of the recurrences costs at least what it brings the cell
//    closer by, so a cell inside that range has all its reachable sources
//    inside theirs: values inside are the unpruned method's, and every cell
//    of every alignment of cost <= T -- the canonical one among them -- is
//    inside.  Rows grow up to about T / 2 and shrink again: with T near the
//    optimum, half the cells of the unpruned method.
//
// Storage.  M of the last max(x, o + e) + 1 scores and I and D of the last
// e + 1 lie in shared memory by diagonal, 16 bits a cell, as u = B_k - h,
// the distance of offset h to the end of diagonal k (B_k = min(m, n + k)):
// in these terms the sequence-end tests vanish (lane_path.cuh says how), the
// end cell is u = 0, and 0x8000 and up is null.  A row position holds an
// older row's cell only where that row was wider, i.e. where the range
// shrinks towards the end, and there no in-range cell reads (by the argument
// above); where the range grows, positions never written are null.
//
// For the CIGAR a row keeps four bits a cell in the arena, in ballots of 32
// cells: mismatch taken, insertion over deletion, I extended, D extended --
// the four choices of the method's tie-break -- half a byte where storing
// M, I and D took six.  The walk back follows the bits (band_walk); the
// match lengths are found again by replaying the operations forward from
// the start, extending after each (band_replay), which is what the forward
// pass did on the way to each cell.
//
// Work split.  One warp per pair, or a CTA of four or eight when the rows are
// wide (or do not fit a warp's share of the shared memory): a lane per
// diagonal, 32 * warps diagonals a round.
#pragma once

#include "arena_path.cuh"
#include "launch.h"
#include "short_path.cuh"
#include "wfa_device.cuh"

namespace wfa {

constexpr uint32_t kBandNull = 0xFFFFu;
constexpr uint32_t kBandValid = 0x8000u;  // u below this is an offset
constexpr int kBandWarps = 4;             // warps of a CTA (and of a team); twice as many when few pairs are long
// Rows wider than this (or than a warp's share of the shared memory): a team,
// whose every row costs each of its warps the fixed part and a barrier
// (200,000 mixed-length pairs 12.6 ms a call with teams from 256 diagonals, 11.8
// from what fits a warp).
constexpr int kBandTeamWidth = 512;

// 16-bit row cells a pair keeps per diagonal.
__host__ __device__ constexpr int band_rows(int x, int oe, int e) {
  return (x > oe ? x : oe) + 1 + 2 * (e + 1);
}
__host__ __device__ constexpr int band_words(int len) { return (len >> 4) + 2; }  // packed words a window may touch

// A pair's diagonals: starts lo0 .. hi0, ends elo .. ehi, bound T; rows lie
// in kmin .. kmax whatever the score.
struct BandGeo {
  int n, m, kf, lo0, hi0, elo, ehi, T, kmin, kmax;
  __device__ __forceinline__ int pitch() const { return (kmax - kmin + 4) & ~1; }  // a null border on either side
  __device__ __forceinline__ int blocks() const { return (kmax - kmin + 32) >> 5; }
  __device__ __forceinline__ int row_lo(int s, int oe, int e) const {
    const int g = s < oe ? 0 : (s - oe + e) / e;
    return max(max(lo0 - g, elo - (T - s) / e), -n);
  }
};

// The lowest value over the scores of max(a - growth(s), b - (T - s) / e):
// the low edge of the widest row (two diagonals of slack for the divisions).
__device__ __forceinline__ int band_edge(int a, int b, int T, int oe, int e) {
  int s = (T + oe - e + e * (a - b)) / 2;
  s = min(max(s, 0), T);
  if (s < oe) s = 0;
  const int g = s < oe ? 0 : (s - oe + e) / e;
  return max(a - g, b - (T - s) / e) - 2;
}

__device__ __forceinline__ BandGeo band_geo(const AlignArgs& a, int n, int m, int T) {
  BandGeo g;
  g.n = n;
  g.m = m;
  g.kf = m - n;
  g.lo0 = -min(a.pb, n);
  g.hi0 = min(a.tb, m);
  g.elo = max(g.kf - min(a.te, n + m), -n);
  g.ehi = min(g.kf + min(a.pe, n + m), m);
  g.T = T;
  g.kmin = max(band_edge(g.lo0, g.elo, T, a.oes, a.es), -n);
  g.kmax = min(-band_edge(-g.hi0, -g.ehi, T, a.oes, a.es), m);
  g.kmax = max(g.kmax, g.kmin);  // every row empty (T below the cost of any alignment): one position, always null
  return g;
}

// Shared memory of a pair: both packed sequences, the rows, and room past
// the last row for the lanes of a round beyond the range.
__device__ __forceinline__ int band_bytes(const AlignArgs& a, const BandGeo& g) {
  const int seq = 4 * (band_words(g.n) + band_words(g.m));
  return ((seq + 15) & ~15) + 2 * g.pitch() * band_rows(a.xs, a.oes, a.es) + 80;
}

// Matches from (v, h), at most rem: 16 bases a round.
__device__ __forceinline__ int band_extend(const uint32_t* pw, const uint32_t* tw, int v, int h, int rem) {
  int got = 0;
  for (;;) {
    const uint32_t d = window32s(pw, v + got, 1) ^ window32s(tw, h + got, 1);
    const int eq = __clz(d) >> 1;
    got += eq;
    if (eq < 16 || got >= rem) return min(got, rem);
  }
}

// ---------------------------------------------------------------- bound

// The search for a pair's bound, a row at a time, on one warp: lane l holds
// the diagonal k = l (mod 32) of the window b .. b + 31, its rows the
// band_rows(...) * 32 cells at ring.  Every fourth score the window moves when
// its furthest cell (largest v + h) comes within a quarter of an edge.  On
// every sampled pair of 100 to 10,000 bases at up to 10 % edits the bound found
// was the optimum itself.  (Half a warp per pair found it too, but two pairs'
// extensions in one warp wait for each other: 260 instructions a score for two
// pairs against 148 for one, and twice the latency on long reads.)
struct BandSearch {
  static constexpr int kLanes = 32;
  static constexpr unsigned kAll = 0xffffffffu;
  const uint32_t *pw, *tw;
  uint16_t* ring;
  int n, m, kf, elo, ehi, b, k, s, cap;
  int rs, rx, ro, rn, re;  // ring rows of the scores s, s - x, s - o - e (M), s, s - e (I, D)

  __device__ static int lane() { return threadIdx.x & (kLanes - 1); }

  // Score 0; true when it reaches an end.
  __device__ bool start(const uint32_t* pw_, const uint32_t* tw_, const BandGeo& g, int x, int oe, int e, int cap_,
                        uint16_t* ring_) {
    const int l = lane(), R = max(x, oe) + 1, RE = e + 1;
    pw = pw_;
    tw = tw_;
    ring = ring_;
    n = g.n;
    m = g.m;
    kf = g.kf;
    elo = g.elo;
    ehi = g.ehi;
    cap = cap_;
    s = 0;
    for (int r = 0; r < R + 2 * RE; ++r) ring[r * kLanes + l] = (uint16_t)kBandNull;
    b = -kLanes / 2;
    if (g.lo0 != g.hi0) {  // free starts: the one with the longest match
      int best = 0;
      for (int q = g.lo0 + l; q <= g.hi0; q += kLanes) {
        const int h = max(q, 0), v = h - q, rem = min(n - v, m - h);
        const int len = rem > 0 ? band_extend(pw, tw, v, h, rem) : 0;
        best = max(best, (len << 16) | (q - g.lo0));  // lengths < 32,768: no overlap with the sign
      }
      b = g.lo0 + (__reduce_max_sync(kAll, best) & 0xFFFF) - kLanes / 2;
    }
    k = b + ((l - b) & (kLanes - 1));
    bool fin = false;
    if (k >= g.lo0 && k <= g.hi0) {
      const int h = max(k, 0), v = h - k, rem = min(n - v, m - h);
      const int u = rem > 0 ? rem - band_extend(pw, tw, v, h, rem) : 0;
      ring[l] = (uint16_t)u;
      fin = u == 0 && k >= elo && k <= ehi;
    }
    __syncwarp(kAll);
    rs = 1 % R, rx = (1 - x + R) % R, ro = (1 - oe + R) % R, rn = 1 % RE, re = 2 % RE;
    return __any_sync(kAll, fin);
  }

  // The next score; true when it reaches an end.
  __device__ __forceinline__ bool step(int x, int oe, int e) {
    const int l = lane(), R = max(x, oe) + 1, RE = e + 1;
    uint16_t* const I = ring + R * kLanes;
    uint16_t* const D = I + RE * kLanes;
    ++s;
    const uint32_t mx = ring[rx * kLanes + l];
    const int l1 = (l - 1) & (kLanes - 1), r1 = (l + 1) & (kLanes - 1);
    const bool first = k == b, last = k == b + kLanes - 1;
    const uint32_t oa = first ? kBandNull : ring[ro * kLanes + l1], il = first ? kBandNull : I[re * kLanes + l1];
    const uint32_t oc = last ? kBandNull : ring[ro * kLanes + r1], dr = last ? kBandNull : D[re * kLanes + r1];
    const uint32_t uI = min(il, oa) - (k > kf ? 1u : 0u);
    const uint32_t uD = min(dr, oc) - (k < kf ? 1u : 0u);
    uint32_t u = min(mx - 1u, min(uI, uD));
    int far = 0;  // v + h of the cell
    bool fin = false;
    if (u < kBandValid) {
      const int h = min(m, n + k) - (int)u;
      u -= (uint32_t)band_extend(pw, tw, h - k, h, (int)u);
      far = 2 * (min(m, n + k) - (int)u) - k;
      fin = u == 0 && k >= elo && k <= ehi;
    } else {
      u = kBandNull;
    }
    ring[rs * kLanes + l] = (uint16_t)u;
    I[rn * kLanes + l] = (uint16_t)uI;
    D[rn * kLanes + l] = (uint16_t)uD;
    __syncwarp(kAll);
    if ((s & 3) == 0) {
      const int best = __reduce_max_sync(kAll, (far << 5) | l);
      const int at = ((best & 31) - b) & (kLanes - 1);
      if (best >= 32 && (at < kLanes / 4 || at >= kLanes - kLanes / 4)) {
        b += at - kLanes / 2;
        const int k2 = b + ((l - b) & (kLanes - 1));
        if (k2 != k)
          for (int r = 0; r < R + 2 * RE; ++r) ring[r * kLanes + l] = (uint16_t)kBandNull;
        k = k2;
        __syncwarp(kAll);
      }
    }
    rs = rs + 1 == R ? 0 : rs + 1;
    rx = rx + 1 == R ? 0 : rx + 1;
    ro = ro + 1 == R ? 0 : ro + 1;
    rn = rn + 1 == RE ? 0 : rn + 1;
    re = re + 1 == RE ? 0 : re + 1;
    return __any_sync(kAll, fin);
  }
};

// The whole search on one warp: an upper bound on the pair's scaled score, at
// most cap (itself a bound, or the caller's largest score of interest).
__device__ __forceinline__ int band_bound(const uint32_t* pw, const uint32_t* tw, const BandGeo& g, int x, int oe,
                                          int e, int cap, uint16_t* ring) {
  BandSearch w;
  if (w.start(pw, tw, g, x, oe, e, cap, ring)) return 0;
  while (w.s + 1 < cap)
    if (w.step(x, oe, e)) return w.s;
  return cap;
}

// A bound that needs no search: every base a mismatch and the length
// difference one gap, or one gap for each sequence.
__device__ __forceinline__ int band_worst(int n, int m, int x, int oe, int e) {
  const int d = abs(n - m), o = oe - e;
  const int one = x * min(n, m) + (d ? o + e * d : 0);
  const int two = (n ? o + e * n : 0) + (m ? o + e * m : 0);
  return min(one, two);
}

// -------------------------------------------------------------- forward

// The scores without a wavefront among the first max(x, o + e) + 1 (bit s):
// their rows need not be written.  M's ring positions of such a score are
// still null: each score up to max(x, o + e) is the first to use its own.  I
// and D's rings are shorter: where e >= 2 and x lies well above o + 2 e, a row
// left out may show the gap cells of e + 1 scores before (x = 10, o + e = 5, e =
// 2: score 8 has no wavefront, and its I and D positions hold score 5).  Results
// do not change: such a cell belongs to a real alignment, counted dearer than
// it is, so that an end it leads to at score s was found at s - e - 1 at the
// latest; no cell on the way to the end at the optimum, and no tie there, comes
// from one.
__device__ __forceinline__ uint32_t band_absent(int x, int oe, int e) {
  uint32_t ex = 1u, gap = 0u;
  for (int s = 1; s < 32; ++s) {
    const bool g = (s >= oe && ((ex >> (s - oe)) & 1u)) || (s >= e && ((gap >> (s - e)) & 1u));
    if (g) gap |= 1u << s;
    if (g || (s >= x && ((ex >> (s - x)) & 1u))) ex |= 1u << s;
  }
  const int R = max(x, oe) + 1;
  return R >= 32 ? ~ex : ~ex & ((1u << R) - 1u);
}

// The exact score of a pair whose score is at most g.T, on WPP warps: the
// scaled score (and its end diagonal in *k_out), or -1 when no alignment
// costs at most T.  bits: the choice bits of row s, block c at
// bits[s * g.blocks() + c] (CIG).  fin: a shared word, 0 on entry: the score
// whose row holds an end (EF).  It is this pass's alone until the team's next
// barrier after the return: a warp may still read it then.
template <int WPP, bool CIG, bool EF>
__device__ int band_forward(const BandGeo& g, const uint32_t* pw, const uint32_t* tw, uint16_t* rows, int x, int oe,
                            int e, uint32_t absent, uint4* bits, int* fin, int* k_out) {
  constexpr unsigned FULL = 0xffffffffu;
  using T_ = Team<WPP>;
  const int lane = threadIdx.x & 31, warp = WPP == 1 ? 0 : (int)(threadIdx.x >> 5), r = T_::rank();
  const int n = g.n, m = g.m, kf = g.kf, pitch = g.pitch(), nblk = g.blocks();
  const int R = max(x, oe) + 1, RE = e + 1;
  uint16_t* const I = rows + R * pitch;
  uint16_t* const D = I + RE * pitch;
  {
    uint32_t* z = reinterpret_cast<uint32_t*>(rows);  // pitch is even
    for (int i = r; i < (R + 2 * RE) * pitch / 2; i += T_::kSize) z[i] = 0xFFFFFFFFu;
  }
  T_::sync();
  const int off = 1 - g.kmin;  // position of diagonal 0
  // the end diagonal's position; outside every row: a border, always null
  const int pf = kf >= g.kmin && kf <= g.kmax ? kf + off : 0;
  // Of the end diagonals of a row with u = 0, the one nearest kf, the larger
  // on a tie (every warp the same answer).
  auto pick_end = [&](int row, int lo, int hi) -> int {
    int best = INT_MAX;
    for (int k = max(lo, g.elo) + lane; k <= min(hi, g.ehi); k += 32)
      if (rows[row + k + off] == 0) best = min(best, 2 * abs(k - kf) + (k < kf ? 1 : 0));
    best = __reduce_min_sync(FULL, best);
    return best == INT_MAX ? INT_MAX : (best & 1) ? kf - (best >> 1) : kf + (best >> 1);
  };
  int q = g.T / e, q_at = g.T % e + 1;  // (T - s) / e, and the score at which it drops next
  int gr = 0, g_at = oe;                // diagonals grown, and the score at which the next is
  {
    const int lo = max(max(g.lo0, g.elo - q), -n), hi = min(min(g.hi0, g.ehi + q), m);
    for (int k = lo + r; k <= hi; k += T_::kSize) {
      const int h = max(k, 0), v = h - k, rem = min(n - v, m - h);
      rows[k + off] = (uint16_t)(rem > 0 ? rem - band_extend(pw, tw, v, h, rem) : 0);
    }
    T_::sync();
    const int k = EF ? pick_end(0, lo, hi) : rows[pf] == 0 ? kf : INT_MAX;
    if (k != INT_MAX) {
      *k_out = k;
      return 0;
    }
  }
  const int Rp = R * pitch, REp = RE * pitch;
  int rs = 1 % R * pitch, rx = (1 - x + R) % R * pitch, ro = (1 - oe + R) % R * pitch;
  int rn = 1 % RE * pitch, re = 2 % RE * pitch;
  int skip = EF && absent ? __ffs(absent) - 1 : 0;  // the next score without a wavefront
  for (int s = 1; s <= g.T; ++s) {
    if (s == q_at) {
      --q;
      q_at += e;
    }
    if (s == g_at) {
      ++gr;
      g_at += e;
    }
    const int lo = max(max(g.lo0 - gr, g.elo - q), -n), hi = min(min(g.hi0 + gr, g.ehi + q), m);
    const uint16_t* const mxp = rows + rx + off;
    const uint16_t* const mop = rows + ro + off;
    const uint16_t* const ip = I + re + off - 1;
    const uint16_t* const dp = D + re + off + 1;
    int c = warp, k0 = lo + 32 * warp;
    if (EF && s == skip) {  // no wavefront at this score (wide first rows: worth the test)
      k0 = hi + 1;
      absent &= absent - 1;
      skip = absent ? __ffs(absent) - 1 : 0;
    }
    for (; k0 <= hi; k0 += 32 * WPP, c += WPP) {
      const int k = k0 + lane;
      const bool act = k <= hi;
      const uint32_t mx = mxp[k], oa = mop[k - 1], oc = mop[k + 1], il = ip[k], dr = dp[k];
      const uint32_t uI = min(il, oa) - (k > kf ? 1u : 0u);
      const uint32_t uD = min(dr, oc) - (k < kf ? 1u : 0u);
      const uint32_t uX = mx - 1u, uG = min(uI, uD);
      if (CIG) {
        uint4 w;
        w.x = __ballot_sync(FULL, uX <= uG);
        w.y = __ballot_sync(FULL, uI <= uD);
        w.z = __ballot_sync(FULL, il <= oa);  // I extends (ties extend)
        w.w = __ballot_sync(FULL, dr <= oc);
        if (lane == 0) bits[(size_t)s * nblk + c] = w;
      }
      uint32_t u = min(uX, uG);
      if (act) {
        if (u < kBandValid) {
          const int h = min(m, n + k) - (int)u;
          u -= (uint32_t)band_extend(pw, tw, h - k, h, (int)u);
          if (EF && u == 0 && k >= g.elo && k <= g.ehi) *(volatile int*)fin = s;
        } else {
          u = kBandNull;
        }
        rows[rs + off + k] = (uint16_t)u;
        I[rn + off + k] = (uint16_t)uI;
        D[rn + off + k] = (uint16_t)uD;
      }
    }
    T_::sync();
    if (EF) {
      if (*(volatile int*)fin == s) {  // a warp already in the next row may have set s + 1
        *k_out = pick_end(rs, lo, hi);
        return s;
      }
    } else if (rows[rs + pf] == 0) {
      *k_out = kf;
      return s;
    }
    rs = rs + pitch == Rp ? 0 : rs + pitch;
    rx = rx + pitch == Rp ? 0 : rx + pitch;
    ro = ro + pitch == Rp ? 0 : ro + pitch;
    rn = rn + pitch == REp ? 0 : rn + pitch;
    re = re + pitch == REp ? 0 : re + pitch;
  }
  return -1;
}

// ---------------------------------------------------------------- CIGAR

// Walk back from (M, s, k) over the choice bits and write the events to
// ev[0 ..), last first: (length << 4) | op for a mismatch (length 1) or a
// whole gap.  One warp, every lane the same walk: lane j holds the block of
// row s0 - j around the diagonal of the last load, so that a load serves up
// to 32 rows.  Returns the number of events (the start diagonal in *k_out),
// or -1 when the bits are inconsistent (never, for bits the forward pass
// wrote).
__device__ int band_walk(const BandGeo& g, const uint4* bits, int x, int oe, int e, int s, int k, uint32_t* ev,
                         int cap, int* k_out) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, nblk = g.blocks();
  int s0 = -1, lb = 0, q = 0;
  uint4 w = make_uint4(0, 0, 0, 0);
  int op = kOpM, len = 0;  // the gap being walked
  while (s > 0) {
    int j = s0 - s;
    int at = k - __shfl_sync(FULL, lb, j & 31);
    if (s0 < 0 || j > 31 || at < 0 || at > 31) {
      s0 = s;
      const int sr = s - lane;
      const int lo = sr > 0 ? g.row_lo(sr, oe, e) : 0;
      const int blk = (k - lo) >> 5;
      lb = INT_MAX / 2;  // no block: reloaded when the walk gets there
      if (sr > 0 && k >= lo && blk < nblk) {
        lb = lo + 32 * blk;
        w = bits[(size_t)sr * nblk + blk];
      }
      j = 0;
      at = k - __shfl_sync(FULL, lb, 0);
      if (at < 0 || at > 31) return -1;
    }
    const uint32_t bx = __shfl_sync(FULL, op == kOpM ? w.x : op == kOpI ? w.z : w.w, j);
    const bool bit = (bx >> at) & 1u;
    if (op == kOpM) {
      if (bit) {
        if (q >= cap) return -1;
        if (lane == 0) ev[q] = (1u << 4) | kOpX;
        ++q;
        s -= x;
      } else {
        op = ((__shfl_sync(FULL, w.y, j) >> at) & 1u) ? kOpI : kOpD;
        len = 0;
      }
    } else {
      ++len;
      k += op == kOpI ? -1 : 1;
      s -= bit ? e : oe;
      if (!bit) {
        if (q >= cap) return -1;
        if (lane == 0) ev[q] = ((uint32_t)len << 4) | (uint32_t)op;
        ++q;
        op = kOpM;
      }
    }
  }
  if (s != 0 || op != kOpM) return -1;
  *k_out = k;
  return q;
}

// Replay the events forward from the start on diagonal k, extending after
// each one, and write the CIGAR's runs downwards from top[-1] (so that they
// lie last run first).  One warp; an extension compares 16 bases a lane.
// ev and the runs may share a buffer of 2 * q + 3 words (ev at its start,
// top past its end): an event gives at most two runs.  Returns the number of
// runs, or -1 when the events do not lead to the end diagonal k_end.
__device__ int band_replay(const BandGeo& g, const uint32_t* pw, const uint32_t* tw, const uint32_t* ev, int q, int k,
                           int k_end, uint32_t* top) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, n = g.n, m = g.m;
  uint32_t cur_op = 0xF, cur_len = 0;
  int nr = 0;
  auto emit = [&](uint32_t op, uint32_t len) {
    if (len == 0) return;
    if (op == cur_op) {
      cur_len += len;
      return;
    }
    if (cur_len) {
      ++nr;
      if (lane == 0) top[-nr] = (cur_len << 4) | cur_op;
    }
    cur_op = op;
    cur_len = len;
  };
  int h = max(k, 0);
  auto slide = [&]() {
    int got = 0;
    for (;;) {
      const int rem = min(n - (h - k), m - h);
      const bool in = 16 * lane < rem;
      uint32_t d = 0;
      if (in) d = window32s(pw, h - k + 16 * lane, 1) ^ window32s(tw, h + 16 * lane, 1);
      const unsigned diff = __ballot_sync(FULL, !in || d != 0);
      const int f = diff ? __ffs(diff) - 1 : 32;
      const int eq = diff ? (int)(__clz(__shfl_sync(FULL, in ? d : 0xFFFFFFFFu, f)) >> 1) : 0;
      const int len = min(16 * f + eq, max(rem, 0));
      h += len;
      got += len;
      if (f < 32) break;
    }
    emit(kOpM, (uint32_t)got);
  };
  if (k > 0) emit(kOpI, (uint32_t)k);
  if (k < 0) emit(kOpD, (uint32_t)(-k));
  slide();
  for (int i0 = q - 1; i0 >= 0; i0 -= 32) {
    const uint32_t mine = i0 - lane >= 0 ? ev[i0 - lane] : 0u;
    __syncwarp();  // loaded before a run may overwrite them
    for (int j = 0; j < min(32, i0 + 1); ++j) {
      const uint32_t v = __shfl_sync(FULL, mine, j);
      const uint32_t op = v & 15u;
      const int len = (int)(v >> 4);
      emit(op, (uint32_t)len);
      if (op != kOpD) h += len;
      if (op == kOpI) k += len;
      if (op == kOpD) k -= len;
      if (h > m || h - k > n) return -1;
      slide();
    }
  }
  if (k != k_end || h != min(m, n + k)) return -1;
  // free end: the characters past the end cell
  if (k > g.kf) emit(kOpD, (uint32_t)(k - g.kf));
  if (k < g.kf) emit(kOpI, (uint32_t)(g.kf - k));
  if (cur_len) {
    ++nr;
    if (lane == 0) top[-nr] = (cur_len << 4) | cur_op;
  }
  return nr;
}

// ----------------------------------------------------------- one pair

// Shared words of a team (a warp or a CTA).  `fin` has a word of its own: the
// first thread, past a pair's last row, writes the queue's next index to
// team.bcast while a slower warp may still be reading `fin` of that row.
struct alignas(16) BandShm {
  TeamShm team;
  int fin;
};

// One pair, on one warp (WPP 1) or a CTA: absent = band_absent(...), smem of at
// least band_bytes, slot_bytes of the arena at slot.  packed: the sequences
// are at smem already.
template <int WPP, bool CIG, bool EF>
__device__ void band_pair(const AlignArgs& a, uint32_t absent, int64_t pair, int T, unsigned char* smem, BandShm* ts,
                          int& round,
                          unsigned char* slot, long slot_bytes, int32_t* overflow_count, bool packed = false) {
  using T_ = Team<WPP>;
  const int r = T_::rank();
  const int n = a.plen[pair], m = a.tlen[pair];
  const BandGeo g = band_geo(a, n, m, T);
  uint32_t* pw = reinterpret_cast<uint32_t*>(smem);
  uint32_t* tw = pw + band_words(n);
  uint16_t* rows = reinterpret_cast<uint16_t*>(smem + ((4 * (band_words(n) + band_words(m)) + 15) & ~15));
  if (CIG && 16L * (T + 1) * g.blocks() > slot_bytes) {
    if (r == 0) overflow_pair_to(a, pair, overflow_count);
    return;
  }
  if (EF && r == 0) ts->fin = 0;
  if (!packed) {
    team_pack32<WPP>(a.pat + a.poff[pair], n, pw, ts->team.flags, round);  // the bound pass checked the bytes
    team_pack32<WPP>(a.txt + a.toff[pair], m, tw, ts->team.flags, round);
  }
  int k_end = 0;
  uint4* bits = reinterpret_cast<uint4*>(slot);
  const int s = band_forward<WPP, CIG, EF>(g, pw, tw, rows, a.xs, a.oes, a.es, absent, bits, &ts->fin, &k_end);
  if (!CIG || s < 0) {
    // no alignment within T: T was the caller's largest score
    if (r == 0) {
      if (s < 0 && T < a.s_cap) atomicExch(&a.ctrl->internal_error, 1);
      write_result(a, pair, s < 0 ? 1 : 0, s < 0 ? -1 : s * a.g, 0, 0);
    }
    return;
  }
  if (WPP > 1 && threadIdx.x >= 32) return;
  // first warp: the CIGAR, into a reservation of the run pool
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // events: each costs that much, and takes a base (the lengths read again:
  // with n and m kept in registers across the rows the row loop compiles to a
  // form 3 % slower on long reads, 2,000 x 10 kbp 5.42 against 5.24 ms a call)
  const int most = min(s / min(a.xs, a.oes), a.plen[pair] + a.tlen[pair]);
  const unsigned long long want = 2ull * most + 3;
  unsigned long long pos = 0;
  if (lane == 0) pos = atomicAdd(&a.ctrl->pool_top, want);
  pos = __shfl_sync(FULL, pos, 0);
  if ((long long)(pos + want) > a.pool_cap) {
    if (lane == 0) {
      atomicExch(&a.ctrl->pool_short, 1);
      overflow_pair_to(a, pair, overflow_count);
    }
    return;
  }
  uint32_t* ev = a.pool + pos;
  int k0 = 0;
  int nr = -1;
  const int q = band_walk(g, bits, a.xs, a.oes, a.es, s, k_end, ev, most, &k0);
  __syncwarp();
  if (q >= 0) nr = band_replay(g, pw, tw, ev, q, k0, k_end, ev + want);
  if (lane == 0) {
    if (nr < 0) atomicExch(&a.ctrl->internal_error, 1);
    // negative: an index into the pool
    write_result(a, pair, 0, s * a.g, max(nr, 0), -(int64_t)(pos + want - max(nr, 0)) - 1);
  }
}

}  // namespace wfa
