// launch.h -- host-side launchers of the library's kernels (C++ linkage,
// internal to libwfa_gpu.so; the public interface is include/wfa_gpu.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "wfa_device.cuh"

namespace wfa {

// Bins of a sample's scaled scores: one each, the last that much or more.
constexpr int kSampleBins = 32;

// Per-call device control block, zeroed before each batch.
struct Ctrl {
  int32_t bad_input;        // a length or offset out of range
  int32_t internal_error;   // stored wavefronts inconsistent in a backtrace
  int32_t defer_count;      // deferred pairs: medium (at most kMediumMaxLen bases)
  int32_t defer_long_count; // and long
  int32_t next_medium;      // work-queue heads of the arena kernels
  int32_t next_long;
  int32_t retry_count;      // pairs of the current retry list
  int32_t next_retry;
  int32_t overflow_count;   // pairs that outgrew their slice of the arena, or the CIGAR pool
  int32_t pool_short;       // the CIGAR pool ran out
  unsigned long long pool_top;  // words used in the CIGAR pool
  long long pat_extent;     // max(offset + length) over patterns
  long long txt_extent;     // max(offset + length) over texts
  int32_t max_len;          // longest pattern or text
  int32_t lane_next;        // work-queue head of the lane kernel on ordered input
  // the band kernels (band_path.cuh): queue heads, and the deferred pairs by
  // who takes them: teams and single warps of the band kernel, or the arena
  // kernels (medium and long pairs)
  int32_t bound_next, team_next, warp_next;
  int32_t team_count, warp_count, arena_count, arena_long_count;
  int32_t pad;
  int32_t sample[kSampleBins];  // scores of a sample (launch_sample_scores)
};
static_assert(sizeof(Ctrl) % 4 == 0 && sizeof(Ctrl) <= 1024, "moved in words, by one small block at most");

struct AlignArgs {
  int64_t n;
  const char* pat;
  const int64_t* poff;
  const int32_t* plen;
  const char* txt;
  const int64_t* toff;
  const int32_t* tlen;
  int xs, oes, es;  // penalties divided by g
  int g;            // gcd(x, o, e)
  int s_cap;        // largest scaled score reported (INT_MAX: none)
  int score_only;
  int host_seqs;  // sequences read in place from page-locked host memory
  // ends-free alignment: free leading / trailing pattern (pb, pe) and text
  // (tb, te) characters; all 0 for a global alignment
  int pb, pe, tb, te;
  int32_t* score;
  int8_t* status;
  int32_t* nruns;
  int64_t* run_src;   // where a pair's runs (last run first) are: >= 0 an
                      // index into `runs`, < 0 the index -src-1 into `pool`
  uint32_t* runs;     // [n * kSlot] per-pair slots of the short kernel
  uint32_t* pool;     // runs of band- and arena-kernel pairs, reserved by atomics
  int64_t pool_cap;   // words in the pool
  int32_t* defer_list;       // [n] deferred medium pairs
  int32_t* defer_long_list;  // [n] deferred long pairs
  int32_t* overflow_list;    // [n]
  Ctrl* ctrl;
  // lane-per-pair kernel input order (both null: pairs in call order).  Each
  // group of G (LaneBand::group) consecutive pairs is packed
  // and sorted by a bound on its score; slot q of group j holds its pair's
  // bit planes at lane_words[(j * 4 * NP + w) * G + q] (NP =
  // lane_plane_words(...): the pattern's NP words of plane 0, of plane 1, then
  // the text's) and (pair or -1, n | m << 8 | bound << 16) at
  // lane_slots[j * G + q].
  uint32_t* lane_words;
  int2* lane_slots;
  int lane_planes;    // plane words lane_words has room for per sequence and plane: the NP of the largest class it takes
  int lane_sort_min;  // smallest store (largest bound) whose ordering bounds each pair
};

// Packed 16-base words per sequence (of at most 127 bases) the lane kernel in
// call order reads, and 32-base words per bit plane of a sequence of at most
// lmax bases the one on ordered input reads (a position past the last base
// included).
constexpr int kLaneWords = 127 / 16 + 2;
__host__ __device__ constexpr int lane_plane_words(int lmax) { return lmax / 32 + 1; }
// Most pairs the ordering sorts together.
constexpr int kLaneGroupMax = 1024;

// longest sequence handled by a one-warp arena team; longer pairs go to a
// one-CTA team
constexpr int kMediumMaxLen = 2048;
// A one-CTA arena team (pairs longer than kMediumMaxLen) has 8 warps when
// few long pairs are deferred (each pair's latency sets the call's) and 4
// when they outnumber the 8-warp teams that fit (more teams in flight).
constexpr int kLongTeamWide = 8;
constexpr int kLongTeamNarrow = 4;

constexpr int kSlot = 16;  // CIGAR runs a short-kernel pair may keep

// Fused short-read kernel (pack + wavefronts in shared memory + backtrace),
// one instantiation per variant.  kind 0: the running pairs of a warp share
// its lanes cell by cell (short_path.cuh); kind 1: one lane per pair, the
// warp's 32 pairs in lockstep over a host-built geometry (lane_path.cuh).
struct ShortVariant {
  const void* kernel;
  const char* name;
  int grid, block, pairs_per_block;
  size_t smem;
  int max_len;  // longest sequence the variant takes
  int cells;    // wavefront cells stored per pair
  int scap;     // largest score index of the geometry table
  int linear;   // 1: gap-linear model only (o = 0; M stored, I and D derived)
  int ends_free;  // 1: for ends-free calls only
  int kind;     // 0 shared-lane, 1 lane-per-pair
  int rw;       // kind 1: positions of each in-place I and D row
  int ct_x, ct_oe, ct_e;  // kind 1: scaled penalties compiled in (0: any)
  // kind 1, ordered input (lane_band.cu): bytes of masks, rows and choices a
  // warp of the kernel over the diagonals within the bound keeps, the cell
  // size of its rows, its shared memory, its resident blocks (for scaled
  // penalties 2/4/1, 1/1/1 and any others) and the ordering pass's (with the
  // walk, without it, and in small groups).
  // `kernel` takes call order (null: the variant runs on ordered input only)
  int band_store, band_cell, band_grid[3], order_grid[3];
  size_t band_smem;
};
struct ShortPlan {
  ShortVariant v[32];
  int count;
};
cudaError_t short_plan(int device, ShortPlan* plan);
cudaError_t launch_short(const AlignArgs& a, const ShortVariant& v, cudaStream_t st);
// Kernels launch_short enqueues: the ordering pass and the lane kernel for a
// lane variant with lane_slots set (sequences in device memory), else one.
int short_launches(const AlignArgs& a, const ShortVariant& v);

// Geometry of the lane-per-pair kernel for one call (a kernel parameter):
// the uniform table of scores 0..31, the last score the kernel stores (-1:
// it takes no pair, e.g. ends-free calls), and where the in-place I and D
// rows keep each score: I_s[k] at position (s mod e) * span_i + k - s/e +
// off_i, D_s[k] at (s mod e) * span_d + k + s/e + off_d.
// rows[s]: score s's row as the forward pass with the table read at run
// time takes it (every lane of every warp the same, so it is worked out
// once on the host): its diagonals and store cells, where its sources lie,
// and the items whose sources all lie inside their rows.
struct alignas(16) LaneRow {
  int32_t lo, w, base;  // first diagonal, width, store cell of item 0
  int32_t ax, wx, cx;   // row s - x: its first item, its width, the cell of item 0
  int32_t ao, wo, co;   // row s - o - e, likewise
  int32_t pi0, pd0;     // I and D row positions of item 0
  int32_t a, b;         // items a .. b - 1 need no range test
  int32_t ex;           // 1: the score has an M wavefront
  int32_t pad[2];
};
struct LaneGeo {
  UGeo tab[32];
  LaneRow rows[32];
  int32_t s_store, off_i, off_d, span_i, span_d, pad[3];
};
// Fills g for the call's penalties and a variant of `cells` cells and
// in-place rows of `rw` positions (lane_layout in lane_path.cuh: the last
// stored score is the largest whose wavefronts fit the cells, are at most 32
// diagonals wide, fit the rows, and whose row reads each find the previous
// score's value or a position not yet written).
void lane_geometry(const AlignArgs& a, int cells, int rw, LaneGeo* g);

// What the lane kernel over the diagonals within the bound needs of a call
// (a kernel parameter): row positions, words of choices, the largest
// bound its store holds (-1: it takes no pair), the shared memory of a warp,
// and the scores whose rows run (bit s; a score without a wavefront whose rows nobody wrote is left
// out).
struct LaneBand {
  int32_t pitch, words, s_store, warp_bytes;
  int32_t group;  // pairs of a group of the ordering pass (a power of two)
  uint32_t run;
};
void lane_band_plan(const AlignArgs& a, const ShortVariant& v, LaneBand* lb);
// Whether launch_short runs the ordering pass and the band kernel of v: only
// where lane_words has room for the planes of v's length class.
bool lane_ordered(const AlignArgs& a, const ShortVariant& v);
cudaError_t launch_lane_ordered(const AlignArgs& a, const ShortVariant& v, cudaStream_t st);
// Fill the ordered half of a lane variant, or a variant that has no other,
// for sequences of up to lmax bases and `store` bytes a warp.
cudaError_t plan_lane_band(int device, ShortVariant* v, int lmax, int store);
cudaError_t plan_ordered(int device, ShortVariant* v, int lmax, int store, bool linear, const char* name);
// The bytes of rows (cells of `cell` bytes), choices and `diags` diagonals'
// masks, and what bounds of 8, 10, 12, 16 and 18 take under scaled penalties
// 2/4/1, and of 6 under 1/1/1 (the edit distance), for up to 127 bases.
constexpr int lane_band_store(int rows, int choices, int diags, int lmax, int cell = 1) {
  return rows * cell + choices + diags * lane_plane_words(lmax) * 128;
}
constexpr int kLaneStore8 = lane_band_store(1536, 896, 6, 127), kLaneStore10 = lane_band_store(1920, 1152, 8, 127),
              kLaneStore12 = lane_band_store(2304, 1408, 10, 127), kLaneStore16 = lane_band_store(3072, 2688, 14, 127),
              kLaneStore18 = lane_band_store(3456, 3328, 16, 127), kLaneStoreLin6 = lane_band_store(960, 896, 8, 127);

// Every pair onto the arena work lists (arena-only calls).
cudaError_t launch_route_all(const AlignArgs& a, cudaStream_t st);

// Resident teams per SM of an arena kernel with teams of team_warps warps
// (1: one-warp teams of medium pairs; kLongTeamWide or kLongTeamNarrow:
// one-CTA teams of long pairs).
cudaError_t arena_occupancy(int team_warps, int* teams_per_sm);
// An arena kernel over the pairs list[0 .. *count), taken through the
// work-queue head *next by `nteams` teams with slot_bytes of the arena each;
// pairs that do not fit go to a.overflow_list.
cudaError_t launch_arena(int team_warps, const AlignArgs& a, const int32_t* list, const int32_t* count,
                         int32_t* next, int32_t* overflow_count, unsigned char* arena, long slot_bytes, int nteams,
                         cudaStream_t st);

constexpr int kBandMaxPen = 31;     // scaled penalties the band kernels take: rows kept per pair
constexpr int kBandMaxLen = 32000;  // sequences they take are shorter: a row cell's offset fits 15 bits
// The band kernels over the deferred pairs (a.defer_list, a.defer_long_list
// and their counts in a.ctrl): each pair's score bound, the pairs ordered by
// cost (largest first; in call order when `ordered` is false), then the band
// kernel over those it takes.  The rest -- sequences of kBandMaxLen bases and
// more, scaled penalties above kBandMaxPen, rows wider than a team's shared
// memory -- end up in arena_list / arena_long_list (ctrl->arena_count,
// arena_long_count), pairs that outgrow their arena slice in
// a.overflow_list.  Counts are read on the device, so that the launches can
// be captured into a graph.
struct BandPlan {
  // by the longest sequence of the call, ascending: CTAs per SM and shared
  // memory of the band kernel
  static constexpr int kSizes = 4;
  int max_len[kSizes], warps[kSizes], per_sm[kSizes], smem[kSizes];
  int nsm;
};
struct BandBufs {
  int32_t* key;    // [n] by pair: score bound, and its bin in the order
  int32_t* order;  // [n] the band kernel's pairs: teams' first, then single warps'
  int32_t* arena_list;
  int32_t* arena_long_list;
  int32_t* aux;  // kBandAux ints of scratch
};
constexpr int kBandBins = 128;
constexpr int kBandAux = 2 * kBandBins;
cudaError_t band_plan(int device, BandPlan* plan);
// pairs: at most this many are deferred, nlong of them long; max_len: the
// longest sequence among the call's (sizes the shared memory; a longer pair in
// a replay still ends up right, in the arena lists).
cudaError_t launch_band(const AlignArgs& a, const BandPlan& plan, const BandBufs& b, int64_t pairs, int64_t nlong,
                        int max_len, bool ordered, unsigned char* arena, long arena_bytes, cudaStream_t st);
// Kernels it enqueues: under scaled penalties above kBandMaxPen only those
// that order the arena lists.
int band_launches(const AlignArgs& a);
// Calls of at most kDirectPairs pairs: every pair on a warp of its own, what
// does not fit deferred.
constexpr int kDirectPairs = 4096;
// Scores of the first pairs of a global call (a.n of them; those of at most
// lmax bases, scaled penalties up to kBandMaxPen), found by the band kernels'
// search for a bound, counted in ctrl->sample.
cudaError_t launch_sample_scores(const AlignArgs& a, int lmax, cudaStream_t st);
cudaError_t launch_direct(const AlignArgs& a, const BandPlan& plan, unsigned char* arena, long arena_bytes,
                          cudaStream_t st);

// Offsets of back-to-back patterns and texts (both exclusive scans of the
// lengths, [n] = totals) and the checks and extents of launch_validate, in
// one pass of three kernels; ctrl must be zeroed first.
cudaError_t launch_offsets_validate(const int32_t* plen, const int32_t* tlen, int64_t n, int64_t* poff,
                                    int64_t* toff, int64_t* tmp, Ctrl* ctrl, cudaStream_t st);

// Calls of at most kDirectPairs pairs, one block each: the control block
// zeroed, the offsets that are missing (poff / toff null: the exclusive scans
// to out_poff / out_toff) and the checks and extents of launch_validate; and
// the CIGAR offsets (out[n] = the total) with the control block and the
// total in their host mirrors (device addresses; off null: score only).
cudaError_t launch_small_front(int64_t n, const int64_t* poff, const int32_t* plen, const int64_t* toff,
                               const int32_t* tlen, int64_t* out_poff, int64_t* out_toff, Ctrl* ctrl, cudaStream_t st);
cudaError_t launch_small_finish(int64_t n, const int32_t* nruns, int64_t* off, const Ctrl* ctrl, Ctrl* h_ctrl,
                                int64_t* h_total, cudaStream_t st);

// Validate lengths / offsets, record max(offset + length) extents.
cudaError_t launch_validate(int64_t n, const int64_t* poff, const int32_t* plen, const int64_t* toff,
                            const int32_t* tlen, Ctrl* ctrl, cudaStream_t st);

// Elements per tile of the prefix-sum kernels (one tile sum each in tmp).
constexpr int kScanTile = 2048;

// Exclusive prefix sums into out[0..n] (out[n] = total).  `kind`:
//   0: values in[i];  1: ceil(in[i]/32) + 1 (packed words per sequence).
// tmp must hold scan_tmp_elems(n) int64.
int64_t scan_tmp_elems(int64_t n);
cudaError_t launch_scan(const int32_t* in, int64_t n, int kind, int64_t* out, int64_t* tmp, cudaStream_t st);

// The output words of a compaction: off[0] .. off[n] of its n pairs.  off[0] is
// not 0 for a chunk of a call: the words before it are other chunks', maybe on
// their way to the host.
struct CompactSpans {
  int64_t n, first, last;
  static constexpr int64_t kSpan = 256;  // words a warp takes at a time
  // cut by words, not by pairs: 64 words and more a pair
  __host__ __device__ constexpr bool by_words() const { return last - first > 64 * n; }
  // first word of a warp's first span
  __host__ __device__ constexpr int64_t begin(int64_t warp) const { return first + warp * kSpan; }
};
// CIGAR compaction: pair i's runs (stored last first, see run_src) to
// out[off[i] .. off[i+1]) in order; writes nothing if off[n] > cap or the
// inputs were rejected (ctrl may be NULL).
cudaError_t launch_compact(int64_t n, const int32_t* nruns, const int64_t* run_src, const uint32_t* runs,
                           const uint32_t* pool, const int64_t* off, uint32_t* out, int64_t cap, const Ctrl* ctrl,
                           cudaStream_t st);

// p[0 .. count) += v (int64).
cudaError_t launch_add(int64_t* p, int64_t count, int64_t v, cudaStream_t st);

// Small transfers as one-block kernels.  A copy engine serves the copies of
// every stream in order, so a small copy queued behind another stream's
// bulk copy (a chunk of input bases, a chunk of outputs) waits for all of
// it; a kernel's loads and stores do not.  launch_put_ctrl writes v (a
// kernel argument) to dst; launch_copy_small copies bytes (a multiple of 4,
// at most 4 KiB, both addresses 4-byte aligned; dst may be the device
// address of page-locked host memory).
cudaError_t launch_put_ctrl(Ctrl* dst, const Ctrl& v, cudaStream_t st);
cudaError_t launch_copy_small(void* dst, const void* src, size_t bytes, cudaStream_t st);

// Standalone packer: sequence i -> words[woff[i] ..], invalid[i].
cudaError_t launch_pack(int64_t n, const char* seqs, const int64_t* off, const int32_t* len, const int64_t* woff,
                        uint64_t* words, int8_t* invalid, cudaStream_t st);

}  // namespace wfa
