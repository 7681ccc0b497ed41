// lane_band.cuh -- short pairs, one lane each, over the diagonals that can
// matter: an ordering pass that packs, bounds and sorts the pairs, and the
// lane-per-pair kernel that runs on its output.
//
// The ordering pass bounds each pair's scaled score from above by a greedy
// alignment (T) and sorts every group of pairs by (T, end diagonal m - n), so
// that the 32 pairs of a warp have nearly the same bound and end diagonal;
// for stores of low scores T is the store's last score for every pair.
// The kernel then runs the wavefronts in lockstep, one lane per pair, but a
// row holds only diagonals that lie on some alignment of cost <= T: those a
// start reaches (a gap of d costs o + e d) from which an end diagonal is
// still within reach (a cell d diagonals from the nearest end diagonal of
// the warp's pairs needs o + e d more, or e d when the gap that closes the
// distance is already open).  At T = 16, 12 and 8 under 4/6/2 (scaled
// 2/4/1) that is 85, 37 and 9 cells where the unpruned rows have 195, 104
// and 37.  Every step of the recurrences costs at least what it brings the
// cell closer by, so the sources of a cell inside the range are inside
// theirs: values inside are the unpruned method's, and so are the score and
// the canonical alignment, whose cells all are.
//
// Storage, [position][32 lanes], a lane touching only its own column: M of
// the last max(x, o + e) scores and I and D of the last e, by diagonal and
// in place (a cell's sources to the left, already overwritten, are carried
// in registers), as u = B_k - h (lane_path.cuh), unsigned and wrapping to
// null past an end.  A row position holds an older row's value only where
// rows shrink, and there no cell inside the range reads it.
//
// Extension reads mismatch masks: once per pass, for every diagonal of the
// rows, one bit a position (set: the bases differ, or an end is reached),
// from the sequences' two bit planes, 32 positions a word.  A cell then finds
// its next mismatch with two loads, a funnel shift and a count of leading
// zeros; comparing packed windows in every cell took 22 instructions, and 45
// for every further 32 bases of a long match, which some lane of the 32 has
// in nearly every row.
//
// For the CIGAR
// each cell leaves four choice bits (mismatch taken, insertion over
// deletion, I extended, D extended), a word or two a row; the walk back
// follows them to the events and a replay from the start finds
// the match lengths, extending after each event as the forward pass did.
#pragma once

#include "lane_path.cuh"
#include "launch.h"
#include "short_path.cuh"
#include "wfa_device.cuh"

namespace wfa {

// ------------------------------------------------------------ ordering

// Sort keys: the bound times eight, plus the end diagonal clamped to
// -4 .. 3 (in alternate directions for odd and even bounds, so that
// neighbouring keys have neighbouring end diagonals); empty slots take the
// last key.
constexpr int kLaneKeys = 256;
constexpr int kLaneBoundMax = kLaneKeys / 8 - 2;  // largest bound (and stored score)

// Matches from pattern position v and text position h, up to 32, from the bit
// planes of both sequences (P: the pattern's NP words of plane 0, then of
// plane 1, then the text's; word j at P[j * 32]; position i in bit
// 31 - i % 32 of word i / 32).  Positions past a sequence's end count as
// whatever lies there: callers clamp.  Reads up to word 4 * NP of P.
template <int NP>
__device__ __forceinline__ int plane_match32(const uint32_t* P, int v, int h) {
  const uint32_t* p = P + (v >> 5) * 32;
  const uint32_t* t = P + (2 * NP + (h >> 5)) * 32;
  const uint32_t a = __funnelshift_l(p[32], p[0], v), b = __funnelshift_l(p[(NP + 1) * 32], p[NP * 32], v);
  const uint32_t c = __funnelshift_l(t[32], t[0], h), d = __funnelshift_l(t[(NP + 1) * 32], t[NP * 32], h);
  return __clz((a ^ c) | (b ^ d));
}

// The furthest offset of diagonal k from offset h: 32 bases a round.
template <int NP>
__device__ __forceinline__ int plane_extend(const uint32_t* P, int n, int m, int k, int h) {
  for (;;) {
    const int rem = min(n - (h - k), m - h);
    if (rem <= 0) return h;
    const int eq = plane_match32<NP>(P, h - k, h);
    if (eq >= rem) return h + rem;
    h += eq;
    if (eq < 32) return h;
  }
}

// Cost of a greedy alignment, an upper bound on the optimal scaled score,
// followed only up to cap (a higher bound changes nothing: such a pair
// passes the store): from the furthest point of diagonal 0, repeatedly take
// one edit and extend.  Of the mismatch, one inserted and one deleted base
// (each priced as a fresh event) the one whose first 32 bases end furthest
// along v + h, less its cost, is taken -- the mismatch at once when at least
// four matches follow it or it reaches an end -- and extended.  The rest of
// the longer sequence at an end is one gap.  (Extending all three to their
// ends first took twice the instructions for the same bounds.)
template <int NP>
__device__ __forceinline__ int lane_estimate(const uint32_t* P, int n, int m, int X, int OE, int E, int cap) {
  int k = 0, h = plane_extend<NP>(P, n, m, 0, 0), cost = 0;
#pragma unroll 1
  while (cost < cap) {  // every edit costs at least 1
    const int v = h - k, rp = n - v, rt = m - h;
    if (rp <= 0 || rt <= 0) {
      const int rem = rp + rt;
      return min(cost + (rem > 0 ? OE + E * (rem - 1) : 0), cap);
    }
    const int rx = min(rp, rt) - 1;
    const int ex = min(plane_match32<NP>(P, v + 1, h + 1), rx);
    const int ei = min(plane_match32<NP>(P, v, h + 1), min(rp, rt - 1));
    const int ed = min(plane_match32<NP>(P, v + 1, h), min(rp - 1, rt));
    // v + h after the window, less the edit's cost, counted from v + h
    const int gx = 2 * ex + 2 - X, gi = 2 * ei + 1 - OE, gd = 2 * ed + 1 - OE;
    const bool px = ex >= 4 || ex == rx || (gx >= gi && gx >= gd), pi = !px && gi >= gd;
    const int len = px ? ex : pi ? ei : ed;
    cost += px ? X : OE;
    k += px ? 0 : pi ? 1 : -1;
    h += len + (px || pi ? 1 : 0);
    if (len == 32) h = plane_extend<NP>(P, n, m, k, h);
  }
  return cap;
}

// 16 ASCII bytes -> the two bit planes of their codes, 16 bits each, first
// byte in the top bit (bits 1 and 2 of the byte, in either case distinct for
// A, C, G and T: the planes tell bases apart, which is all the comparisons
// need), one plane in the upper half, one in the lower; and whether a byte is
// not A/C/G/T: the upper-case letter of each byte's code is picked from
// "ACTG" by a byte permute with the codes as selectors and compared with the
// byte folded to upper case.  Only when some byte differs is the per-byte
// mask (bit i: byte i) worked out.  The 2-bit codes are gathered first, four
// with one multiply, and the planes parted from all 16 at once (an unshuffle
// in four steps): gathering each plane by itself took a third more
// instructions.
__device__ __forceinline__ uint32_t lane_planes16(uint4 v, uint32_t* bad16) {
  const uint32_t q[4] = {v.x, v.y, v.z, v.w};
  uint32_t code = 0u, xs[4], any = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t w = q[i];
    const uint32_t c = (w >> 1) & 0x03030303u;  // byte j's code in bits 8j, 8j + 1
    const uint32_t sel = __byte_perm(c | (c >> 4), 0u, 0x4420u);  // nibble j = byte j's code
    xs[i] = (w & 0xDFDFDFDFu) ^ __byte_perm(0x47544341u, 0u, sel);  // zero byte <=> valid
    any |= xs[i];
    code = __funnelshift_l(c * 0x40100401u, code, 8);  // the product's top byte: 4 codes, first in the top bits
  }
  uint32_t t;
  t = (code ^ (code >> 1)) & 0x22222222u;
  code ^= t ^ (t << 1);
  t = (code ^ (code >> 2)) & 0x0C0C0C0Cu;
  code ^= t ^ (t << 2);
  t = (code ^ (code >> 4)) & 0x00F000F0u;
  code ^= t ^ (t << 4);
  t = (code ^ (code >> 8)) & 0x0000FF00u;
  code ^= t ^ (t << 8);
  uint32_t bad = 0u;
  if (any) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t x = xs[i];
      const uint32_t hb = ((((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x) >> 7) & 0x01010101u;  // 1 per nonzero byte
      bad |= ((hb * 0x01020408u) >> 24 & 0xFu) << (4 * i);
    }
  }
  *bad16 = bad;
  return code;
}

// Aligned 16-byte chunks that hold a base of a sequence starting h bytes into
// the first (none of an empty one, whose address need not be anyone's).
__host__ __device__ inline int lane_chunks(int h, int len) { return len > 0 ? (h + len + 15) >> 4 : 0; }

// One lane packs one sequence of at most 32 * NP - 1 bases from device memory
// into NP words of each bit plane (word j of plane q at out[(q * NP + j) *
// 32]): every aligned 16-byte chunk holding a base is loaded at once, then
// the words are cut from the chunks' planes.  Returns whether a byte of the
// sequence is not A/C/G/T.
template <int NP>
__device__ __forceinline__ bool lane_pack_planes(const char* seq, int len, uint32_t* out) {
  constexpr int NCH = 2 * NP + 1;
  const unsigned long long a0 = reinterpret_cast<uintptr_t>(seq), b0 = a0 & ~15ull;
  const int h = (int)(a0 - b0);
  const int nch = lane_chunks(h, len);
  uint4 raw[NCH];
#pragma unroll
  for (int c = 0; c < NCH; ++c)  // all loads first: their latencies overlap
    raw[c] = c < nch ? __ldg(reinterpret_cast<const uint4*>(b0 + 16ull * c)) : make_uint4(0u, 0u, 0u, 0u);
  uint32_t code[NCH], bad[NCH];
#pragma unroll
  for (int c = 0; c < NCH; ++c) {
    code[c] = 0u;
    bad[c] = 0u;
    if (c < nch) code[c] = lane_planes16(raw[c], &bad[c]);
  }
  uint32_t any_bad = 0u;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    // 32 positions: chunks 2j, 2j + 1 and the first h bytes of 2j + 2
    const uint32_t a = code[2 * j], b = code[2 * j + 1], c = code[2 * j + 2];
    const uint32_t w0 = __byte_perm(b, a, 0x7632), w1 = __byte_perm(b, a, 0x5410);  // plane 0, plane 1
    out[j * 32] = __funnelshift_l(c & 0xFFFF0000u, w0, h);
    out[(NP + j) * 32] = __funnelshift_l(c << 16, w1, h);
    const uint32_t bb = bad[2 * j] | bad[2 * j + 1] | bad[2 * j + 2];
    if (bb) {  // rare: are the bad bytes among the sequence's?
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int first = h - 16 * (2 * j + q), last = first + len;  // the sequence in the chunk
        const uint32_t in = (last >= 16 ? 0xFFFFu : last <= 0 ? 0u : (1u << last) - 1u) &
                            ~(first <= 0 ? 0u : first >= 16 ? 0xFFFFu : (1u << first) - 1u);
        any_bad |= bad[2 * j + q] & in;
      }
    }
  }
  return any_bad != 0u;
}

// Shared memory of the ordering pass: per warp the bit planes of its 32
// pairs; per key its count and its first slot.
template <int LMAX, int GROUP>
struct LaneOrderShm {
  static constexpr int NP = lane_plane_words(LMAX);
  static constexpr int kGroup = GROUP;
  uint32_t planes[kGroup / 32][4 * NP * 32];  // per warp: word j of lane l at [j * 32 + l] (cnt behind the last: see
                                              // plane_match32)
  int cnt[2][kLaneKeys];  // alternate groups use alternate halves
  int start[kLaneKeys];
  int2 slot[kGroup];        // the group's slots in order
  uint16_t from[kGroup];    // and which of its pairs each one holds
};

// The ordering pass (a block of GROUP / PER threads, PER pairs of a group each;
// sequences in device memory, each lane reading its own pair's aligned
// 16-byte chunks).  Large groups: two pairs a thread and two blocks an SM or
// more, so that one packs while another waits for its bytes or its slowest
// warp (with one block of GROUP threads half the issue slots were idle).  Bound
// by instruction issue and the loads' latency: 1M pairs of 100 bases take 76 us
// sorted by end diagonal, 117 us with the walk.  cap: the largest bound of
// interest (the last score the store holds, or the caller's largest); pairs
// above it get it.  walk = false: every pair at cap, sorted by end diagonal
// alone (for stores so small that the greedy walk would cost more than it
// saves).  Pairs longer than LMAX are deferred and pairs with a byte other than
// A/C/G/T get their status here; both, and the slots past the last pair, become
// empty slots (pair -1).
template <int LMAX, int GROUP, int PER>
__device__ void lane_order_body(const AlignArgs& a, int cap, bool walk, unsigned char* smem) {
  using S_t = LaneOrderShm<LMAX, GROUP>;
  constexpr int NP = S_t::NP, G = S_t::kGroup;
  constexpr unsigned FULL = 0xffffffffu;
  if (*(volatile int32_t*)&a.ctrl->bad_input) return;  // inputs rejected by the validation kernel
  auto& S = *reinterpret_cast<S_t*>(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t groups = (a.n + G - 1) / G;
  constexpr int kThreads = G / PER;
  for (int i = threadIdx.x; i < 2 * kLaneKeys; i += kThreads) (&S.cnt[0][0])[i] = 0;
  __syncthreads();
  int half = 0;
  for (int64_t gi = blockIdx.x; gi < groups; gi += gridDim.x, half ^= 1) {
    // this group's counts are in half `half` (zero: cleared while the group
    // before used the other half)
    int* cnt = S.cnt[half];
    int key[PER], at[PER];
    int2 slot[PER];
#pragma unroll 1
    for (int q = 0; q < PER; ++q) {
      const int64_t pair = gi * G + q * kThreads + threadIdx.x;
      uint32_t* const P = S.planes[q * (kThreads / 32) + warp] + lane;
      bool active = pair < a.n;
      int T = cap, kq = kLaneKeys - 1;
      int n = 0, m = 0;
      int64_t po = 0, to = 0;
      if (active) {
        n = a.plen[pair];
        m = a.tlen[pair];
        po = a.poff[pair];  // with the lengths: one round trip for all four
        to = a.toff[pair];
        if (n > LMAX || m > LMAX) {
          defer_pair(a, pair);
          active = false;
        }
      }
      if (active) {
        const bool bad =
            lane_pack_planes<NP>(a.pat + po, n, P) | lane_pack_planes<NP>(a.txt + to, m, P + 2 * NP * 32);
        if (bad) {
          write_result(a, pair, 2, -1, 0, 0);
          active = false;
        }
      }
      if (active) {
        if (walk) T = lane_estimate<NP>(P, n, m, a.xs, a.oes, a.es, cap);
        const int d = min(max(m - n, -4), 3) + 4;
        kq = 8 * T + (T & 1 ? 7 - d : d);
      }
      const unsigned same = __match_any_sync(FULL, kq);
      const int leader = __ffs(same) - 1;
      int first = 0;
      if (lane == leader) first = atomicAdd(&cnt[kq], __popc(same));
      const int rank = __shfl_sync(FULL, first, leader) + __popc(same & ((1u << lane) - 1u));
      const int2 sl = make_int2(active ? (int)pair : -1, active ? n | (m << 8) | (T << 16) : 0);
      if (q == 0) key[0] = kq, at[0] = rank, slot[0] = sl;
      else key[PER - 1] = kq, at[PER - 1] = rank, slot[PER - 1] = sl;
    }
    __syncthreads();
    // every warp is past its reads of the other half (the group before)
    for (int i = threadIdx.x; i < kLaneKeys; i += kThreads) S.cnt[half ^ 1][i] = 0;
    if (warp == 0) {
      constexpr int Q = kLaneKeys / 32;
      int v[Q], sum = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        v[q] = cnt[Q * lane + q];
        sum += v[q];
      }
      int incl = sum;
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += o;
      }
      int run = incl - sum;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        S.start[Q * lane + q] = run;
        run += v[q];
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int to = S.start[key[q]] + at[q];
      S.slot[to] = slot[q];
      S.from[to] = (uint16_t)(q * kThreads + threadIdx.x);
    }
    __syncthreads();
    // a thread writes whole slots, so that a warp's stores are consecutive:
    // written from where the pairs were packed, a store touched up to 32
    // sectors, and the pass waited for them
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int to = q * kThreads + threadIdx.x, from = S.from[to];
      const uint32_t* const P = S.planes[from >> 5] + (from & 31);
      uint32_t* out = a.lane_words + gi * (4 * NP * G) + to;
#pragma unroll
      for (int j = 0; j < 4 * NP; ++j) out[j * G] = P[j * 32];  // (an empty slot's are never used)
      a.lane_slots[gi * G + to] = S.slot[to];
    }
    __syncthreads();  // the planes are the next group's
  }
}

// ------------------------------------------------------------ the kernel

// How far the gaps of a row reach: of score s, a start to -g .. g and a gap
// back towards 0 up to b; with `left` still to spend, an open gap covers `gap`
// diagonals and one still to open m.
__host__ __device__ inline void lane_band_start(int s, int oe, int e, int* g, int* b) {
  *g = s < oe ? 0 : (s - (oe - e)) / e;
  *b = s < 2 * oe ? -1 : (s - 2 * (oe - e)) / e - 2;
}
__host__ __device__ inline void lane_band_end(int left, int oe, int e, int* gap, int* m) {
  *gap = left / e;
  *m = left < oe ? 0 : (left - (oe - e)) / e;
}

// The lowest and highest diagonal of such a row (lo > hi: no cell) for end
// diagonals kl .. kh.
__host__ __device__ inline void lane_band_span(int g, int b, int gap, int m, int kl, int kh, int* lo, int* hi) {
  const int h1 = g < kh + m ? g : kh + m, h2 = b < kh + gap ? b : kh + gap;
  const int l1 = -g > kl - m ? -g : kl - m, l2 = -b > kl - gap ? -b : kl - gap;
  *hi = h1 > h2 ? h1 : h2;
  *lo = l1 < l2 ? l1 : l2;
}

// Row s of a pair set with bound T, start diagonal 0 and end diagonals kl ..
// kh.
__host__ __device__ inline void lane_band_row(int s, int T, int kl, int kh, int oe, int e, int* lo, int* hi) {
  if (T < s) {
    *lo = 1;
    *hi = 0;
    return;
  }
  int g, b, gap, m;
  lane_band_start(s, oe, e, &g, &b);
  lane_band_end(T - s, oe, e, &gap, &m);
  lane_band_span(g, b, gap, m, kl, kh, lo, hi);
}

// Words of choices a row of w cells keeps: four bits a cell, in one word up to
// eight cells and two up to 16.
__host__ __device__ constexpr int lane_band_choice_words(int w) { return w <= 0 ? 0 : w <= 8 ? 1 : 2; }
constexpr int kLaneBandWidth = 16;  // widest row
constexpr int kLaneBlock = 2;       // cells of a row whose loads go together, and one at the end of odd rows
template <int V>
struct IntC {
  static constexpr int value = V;
};

// Rows of a store: M of the last R scores, then I and D of the last e.
__host__ __device__ constexpr int lane_band_rows(int x, int oe, int e) { return (x > oe ? x : oe) + 2 * e; }

// Pairs of the ordering pass, one per lane, in batches of 32 slots taken
// from a queue (within a group the batches' costs rise with the bounds).
// PX, POE, PE: the scaled penalties when known at compile time, else 0; GROUP
// likewise (the loads of a batch at constant strides: 2 % of an E = 2 % call).
// Pairs whose score passes their bound's cap are deferred (or over the
// caller's bound), as are pairs whose CIGAR needs more than kSlot runs.  A
// batch whose end diagonals spread too far for the store (around the border
// of two bounds) runs in two or more passes.
// Bound by instruction issue and the latency between a cell's steps (67 and
// 64 % of the issue slots by instructions and duration); with the large store
// by the 16 warps an SM its 12.9 KB a warp leave.  1M pairs of 100 bases: E =
// 2 % 144 -> 90 us, E = 4 % 508 -> 276 us (75 and 220 warp instructions a pair),
// before: every diagonal a row can hold (lane_path.cuh).
template <typename U, int LMAX, int PX, int POE, int PE, int GROUP>
__device__ __forceinline__ void lane_band_body(const AlignArgs& a, const LaneBand& lb, unsigned char* smem) {
  constexpr int NP = lane_plane_words(LMAX);
  const int64_t G = GROUP ? GROUP : lb.group;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr uint32_t kNull = sizeof(U) == 1 ? 0xFFu : 0xFFFFu;
  // a null loses at most one a score; LMAX and the null range stay apart
  static_assert(LMAX + kLaneBoundMax < (int)kNull, "null offsets");
  if (*(volatile int32_t*)&a.ctrl->bad_input) return;  // inputs rejected by the validation kernel
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // shared memory of the warp: the rows' table, the masks (word j of
  // diagonal kmin + d at masks[(d * NP + j) * 32]), the rows, the choices
  int32_t* const tab = reinterpret_cast<int32_t*>(smem + warp * lb.warp_bytes);  // row s: lo, hi (bytes), first choice word << 16
  const int X = PX ? PX : a.xs, OE = POE ? POE : a.oes, E = PE ? PE : a.es;
  const int R = X > OE ? X : OE, pitch = lb.pitch;
  uint32_t* const masks = reinterpret_cast<uint32_t*>(tab + 32) + lane;
  unsigned char* const store = reinterpret_cast<unsigned char*>(tab + 32) + (pitch - 2) * NP * 128;
  U* const M = reinterpret_cast<U*>(store) + lane;
  U* const I = M + R * pitch * 32;
  U* const D = I + E * pitch * 32;
  const int row_bytes = lane_band_rows(X, OE, E) * pitch * 32 * (int)sizeof(U);
  uint32_t* const bits = reinterpret_cast<uint32_t*>(store + row_bytes) + lane;  // choice word j at bits[j * 32]
  uint16_t* const ev = reinterpret_cast<uint16_t*>(store) + lane;  // events of the walk, over the rows
  const bool cig = !a.score_only;
  const int64_t total = (a.n + G - 1) & ~(G - 1);
  int2 nsl = make_int2(-1, 0);
  uint32_t pl[4 * NP];  // the batch's bit planes, until its masks are built
  auto grab = [&]() -> int64_t {
    int b = 0;
    if (lane == 0) b = atomicAdd(&a.ctrl->lane_next, 1);
    return (int64_t)__shfl_sync(FULL, b, 0) * 32;
  };
  auto fetch = [&](int64_t f) {
    if (f >= total) return;
    nsl = a.lane_slots[f + lane];
    const uint32_t* src = a.lane_words + (f & ~(G - 1)) * (4 * NP) + (f & (G - 1)) + lane;
#pragma unroll
    for (int j = 0; j < 4 * NP; ++j) pl[j] = src[j * G];
  };
  int64_t next = grab();
  fetch(next);
  while (next < total) {
    const int64_t pair = nsl.x;
    bool todo = pair >= 0;
    const int n = nsl.y & 255, m = (nsl.y >> 8) & 255, kf = m - n;
    const int Tl = nsl.y >> 16;
    next = grab();
    if (!__any_sync(FULL, todo)) fetch(next);
    while (__any_sync(FULL, todo)) {
    // the pass's geometry: lane s works out row s
    bool active = todo;
    const int pivot = __shfl_sync(FULL, kf, __ffs(__ballot_sync(FULL, todo)) - 1);
    int T, kmin, ndiag, words;
    for (;;) {
      T = __reduce_max_sync(FULL, active ? Tl : -1);
      const int kl = __reduce_min_sync(FULL, active ? kf : 1 << 20);
      const int kh = __reduce_max_sync(FULL, active ? kf : -(1 << 20));
      int lo, hi;
      lane_band_row(lane, T, kl, kh, OE, E, &lo, &hi);
      const bool empty = lo > hi || !((lb.run >> lane) & 1u);
      const int w = empty ? 0 : hi - lo + 1;
      const int mine = lane_band_choice_words(w);
      int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(FULL, incl, d);
        if (lane >= d) incl += o;
      }
      words = __shfl_sync(FULL, incl, 31);
      kmin = __reduce_min_sync(FULL, w ? lo : 1 << 20);
      const int kmax = __reduce_max_sync(FULL, w ? hi : -(1 << 20));
      ndiag = kmax - kmin + 1;
      // (rows are as wide as the store's positions allow, at most 16)
      if (words == 0 || (ndiag + 2 <= pitch && words <= lb.words)) {
        tab[lane] = ((w ? lo : 1) & 255) | (((w ? hi : 0) & 255) << 8) | ((incl - mine) << 16);
        __syncwarp();
        break;
      }
      // without the pairs whose end diagonal is furthest from the first's
      const int far = __reduce_max_sync(FULL, active ? abs(kf - pivot) : 0);
      if (far == 0) {  // one end diagonal, and still too wide: not with bounds up to the store's
        if (active) defer_pair(a, pair);
        todo = todo && !active;
        active = false;
        words = 0;
        break;
      }
      if (abs(kf - pivot) == far) active = false;
    }
    todo = todo && !active;
    if (words > 0) {
      // the masks of the rows' diagonals, from the planes in registers;
      // position i of diagonal k compares pattern i + max(-k, 0) with text
      // i + max(k, 0)
      const int kmax = kmin + ndiag - 1;
      for (int k = kmin; k <= kmax; ++k) {
        const int len = min(m - max(k, 0), n - max(-k, 0));
        uint32_t* const out = masks + (k - kmin) * NP * 32;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          // (the words past the last are never compared: len < 32 * NP)
          const uint32_t p0 = pl[j], p1 = pl[NP + j], t0 = pl[2 * NP + j], t1 = pl[3 * NP + j];
          const uint32_t q0 = j + 1 < NP ? pl[j + 1] : 0u, q1 = j + 1 < NP ? pl[NP + j + 1] : 0u;
          const uint32_t u0 = j + 1 < NP ? pl[2 * NP + j + 1] : 0u, u1 = j + 1 < NP ? pl[3 * NP + j + 1] : 0u;
          const uint32_t d = k >= 0 ? (p0 ^ __funnelshift_l(u0, t0, k)) | (p1 ^ __funnelshift_l(u1, t1, k))
                                    : (t0 ^ __funnelshift_l(q0, p0, -k)) | (t1 ^ __funnelshift_l(q1, p1, -k));
          const int left = min(max(len - 32 * j, 0), 32);
          out[j * 32] = d | (left == 32 ? 0u : 0xFFFFFFFFu >> left);
        }
      }
    }
    // the next batch's slot and planes load while this pass computes
    if (!__any_sync(FULL, todo)) fetch(next);
    // the next set bit of diagonal k's mask from position i, up to 32 on
    auto matches = [&](int k, int i) -> int {
      const uint32_t* w = masks + ((k - kmin) * NP + (i >> 5)) * 32;
      return __clz(__funnelshift_l(w[32], w[0], i));
    };
    int s_fin = -1;
    bool run = active && words > 0;
    if (words > 0) {
      {
        uint4* z = reinterpret_cast<uint4*>(store);
        for (int i = lane; i < row_bytes / 16; i += 32) z[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
        __syncwarp();
      }
      const int off = 1 - kmin;  // position of diagonal 0
      // score 0
      if ((signed char)(tab[0] & 255) <= (signed char)(tab[0] >> 8)) {
        uint32_t u = kNull;
        if (run) {
          int i = 0, eq;
          do i += eq = matches(0, i);
          while (eq == 32);
          u = (uint32_t)(min(m, n) - i);
          if (kf == 0 && u == 0) {
            s_fin = 0;
            run = false;
          }
        }
        M[off * 32] = (U)u;
      }
      // a lane's end diagonal; outside every row: the border, always null
      const int pf = kf + off >= 1 && kf + off < pitch - 1 ? kf + off : 0;
      int rs = 1 % R, rx = (R + 1 - X % R) % R, ro = (R + 1 - OE % R) % R, re = 1 % E;
      for (int s = 1; s <= T && __any_sync(FULL, run); ++s) {
        if ((lb.run >> s) & 1u) {
          const int t = tab[s];
          const int lo = (signed char)(t & 255), hi = (signed char)((t >> 8) & 255);
          if (lo <= hi) {
          U* const ms = M + (rs * pitch + off) * 32;
          const U* const mx = M + (rx * pitch + off) * 32;
          const U* const mo = M + (ro * pitch + off) * 32;
          U* const ir = I + (re * pitch + off) * 32;
          U* const dr = D + (re * pitch + off) * 32;
          // sources to the left of the cell: M_{s-o-e} and I_{s-e} on k - 1,
          // M_{s-o-e} on k
          uint32_t oa = mo[(lo - 1) * 32], ob = mo[lo * 32], il = ir[(lo - 1) * 32];
          // pending extensions, and the row's choices: mismatch taken,
          // insertion over deletion, I extended, D extended
          uint32_t pend = 0, cx = 0, ci = 0, ce = 0, cd = 0, bit = 1;
          // N cells at once: every load before the stores, which the compiler
          // has to take for aliases of the next cells' sources (1M pairs of 150
          // bases 701 -> 681 us a call, 5M of 100 at E = 4 % 2,030 -> 1,998; three
          // or four at once no faster)
          auto cells = [&](int k, auto count) {
            constexpr int N = count.value;
            uint32_t o[N + 2], dn[N], in[N + 1], u[N];
            int at[N];
            bool valid[N];
            o[0] = oa;
            o[1] = ob;
            in[0] = il;
#pragma unroll
            for (int j = 0; j < N; ++j) {
              o[j + 2] = mo[(k + j + 1) * 32];
              dn[j] = dr[(k + j + 1) * 32];
              in[j + 1] = ir[(k + j) * 32];
              u[j] = (uint32_t)mx[(k + j) * 32] - 1u;
            }
#pragma unroll
            for (int j = 0; j < N; ++j) {
              const bool ei = in[j] <= o[j], ed = dn[j] <= o[j + 2];  // extension (ties extend)
              const uint32_t uI = (ei ? in[j] : o[j]) - (k + j > kf ? 1u : 0u);
              const uint32_t uD = (ed ? dn[j] : o[j + 2]) - (k + j < kf ? 1u : 0u);
              const uint32_t ug = min(uI, uD);
              if (u[j] <= ug) cx |= bit << j;
              if (uI <= uD) ci |= bit << j;
              if (ei) ce |= bit << j;
              if (ed) cd |= bit << j;
              u[j] = min(u[j], ug);
              valid[j] = u[j] <= (uint32_t)LMAX && run;
              at[j] = valid[j] ? min(m, n + k + j) - max(k + j, 0) - (int)u[j] : 0;
              ir[(k + j) * 32] = (U)uI;
              dr[(k + j) * 32] = (U)uD;
            }
            int eq[N];
#pragma unroll
            for (int j = 0; j < N; ++j) eq[j] = matches(k + j, at[j]);
#pragma unroll
            for (int j = 0; j < N; ++j) {
              if (valid[j] && eq[j] == 32) pend |= bit << j;
              ms[(k + j) * 32] = (U)(valid[j] ? u[j] - (uint32_t)eq[j] : u[j]);
            }
            oa = o[N];
            ob = o[N + 1];
            il = in[N];
            bit <<= N;
          };
          int k = lo;
          for (; k + kLaneBlock <= hi + 1; k += kLaneBlock) cells(k, IntC<kLaneBlock>());
          if (k <= hi) cells(k, IntC<1>());
          if (cig) {
            uint32_t* const b = bits + (t >> 16) * 32;
            if (hi - lo < 8) {
              b[0] = cx + (ci << 8) + (ce << 16) + (cd << 24);
            } else {
              b[0] = cx + (ci << 16);
              b[32] = ce + (cd << 16);
            }
          }
          // the cells whose 32 bases all matched: every lane through its own
          while (__any_sync(FULL, pend != 0)) {
            if (pend) {
              const int k = lo + __ffs(pend) - 1;
              const uint32_t u = ms[k * 32];
              const int eq = matches(k, min(m, n + k) - max(k, 0) - (int)u);
              ms[k * 32] = (U)(u - (uint32_t)eq);
              if (eq < 32) pend &= pend - 1;
            }
          }
          if (run && M[(rs * pitch + pf) * 32] == 0) {
            s_fin = s;
            run = false;
          }
          }
        }
        rs = rs + 1 == R ? 0 : rs + 1;
        rx = rx + 1 == R ? 0 : rx + 1;
        ro = ro + 1 == R ? 0 : ro + 1;
        re = re + 1 == E ? 0 : re + 1;
      }
      __syncwarp();  // the rows are the walk's scratch from here
    }
    if (active && s_fin < 0) {
      // no alignment within the bound, which was the caller's largest score
      // or the store's (then the band kernels take the pair)
      if (a.s_cap <= lb.s_store) write_result(a, pair, 1, -1, 0, 0);
      else defer_pair(a, pair);
    } else if (active && !cig) {
      write_result(a, pair, 0, s_fin * a.g, 0, 0);
    } else if (active) {
      // walk back over the choices: a word (length << 2) | op per event
      int s = s_fin, k = kf, q = 0, op = kOpM, len = 0;
      bool bad = false;
      while (s > 0 && !bad) {
        const int t = tab[s];
        const int lo = (signed char)(t & 255), hi = (signed char)((t >> 8) & 255);
        bad = k < lo || k > hi;
        const int i = bad ? 0 : k - lo;
        const uint32_t* const b = bits + (t >> 16) * 32;
        // the cell's four choices, 8 or 16 bits apart
        const bool wide = hi - lo >= 8;
        const uint32_t b0 = b[0] >> i, b1 = wide ? b[32] >> i : b0 >> 16;
        if (op == kOpM && (b0 & 1u)) {
          ev[q++ * 32] = (uint16_t)((1 << 2) | kOpX);
          s -= X;
          continue;
        }
        if (op == kOpM) {
          op = b0 & (wide ? 0x10000u : 0x100u) ? kOpI : kOpD;
          len = 0;
        }
        ++len;
        k += op == kOpI ? -1 : 1;
        if (b1 & (op == kOpI ? 1u : wide ? 0x10000u : 0x100u)) {
          s -= E;
        } else {
          s -= OE;
          ev[q++ * 32] = (uint16_t)((len << 2) | op);
          op = kOpM;
        }
      }
      bad = bad || s != 0 || k != 0 || op != kOpM;
      // replay from the start; runs downwards from the slot's end, so that
      // they lie last run first
      uint32_t* const top = a.runs + (pair + 1) * kSlot;
      uint32_t cur_op = 0xF, cur_len = 0;
      int nr = 0;
      auto emit = [&](uint32_t o, int l) {
        if (l <= 0) return;
        if (o == cur_op) {
          cur_len += (uint32_t)l;
          return;
        }
        if (cur_len && ++nr <= kSlot) top[-nr] = (cur_len << 4) | cur_op;
        cur_op = o;
        cur_len = (uint32_t)l;
      };
      int h = 0;
      for (int i = bad ? -1 : q;; --i) {
        if (i < 0) break;
        if (i < q) {
          const int v = ev[i * 32], o = v & 3, l = v >> 2;
          emit((uint32_t)o, l);
          if (o != kOpD) h += l;
          if (o == kOpI) k += l;
          if (o == kOpD) k -= l;
          if (h > m || h - k > n) {
            bad = true;
            break;
          }
        }
        int at = h - max(k, 0), eq;
        const int from = at;
        do at += eq = matches(k, at);
        while (eq == 32);
        emit(kOpM, at - from);
        h += at - from;
      }
      if (cur_len && ++nr <= kSlot) top[-nr] = (cur_len << 4) | cur_op;
      if (bad || h != m || k != kf) {
        atomicExch(&a.ctrl->internal_error, 1);
        write_result(a, pair, 0, s_fin * a.g, 0, pair * kSlot);
      } else if (nr > kSlot) {
        defer_pair(a, pair);  // more runs than a slot holds
      } else {
        write_result(a, pair, 0, s_fin * a.g, nr, (pair + 1) * kSlot - nr);
      }
    }
    __syncwarp();  // the shared memory is the next pass's
    }
  }
}

}  // namespace wfa
