// band.cu -- the band kernels (band_path.cuh) and their launcher: score
// bounds of the deferred pairs, their order, and the exact wavefronts.
#include <algorithm>

#include "band_path.cuh"
#include "launch.h"

namespace wfa {

namespace {

// Bins of the order: kClassBins for each taker, dearest first.
enum { kTeam = 0, kWarp = 1, kArena = 2, kArenaLong = 3, kClasses = 4 };
constexpr int kClassBins = 31;
constexpr int kNoBin = kBandBins - 1;  // nothing left to do for the pair
static_assert(kClasses * kClassBins <= kNoBin, "bins");
constexpr int kKeyBits = 24;  // a key: bound | bin << kKeyBits
static_assert(kBandMaxPen * kBandMaxLen < (1 << kKeyBits), "a bound fits its key");

// Cost classes half a power of two wide, the largest first.
__device__ __forceinline__ int cost_bin(int cls, unsigned cost) {
  const int lz = 31 - __clz(max(cost, 1u));
  const int half = lz > 0 ? (int)((cost >> (lz - 1)) & 1u) : 0;
  const int i = min(max(2 * lz + half - 6, 0), kClassBins - 1);
  return cls * kClassBins + (kClassBins - 1 - i);
}

// The arena kernels' pairs by length, longest first, in even steps up to the
// call's longest: reads of one batch differ by less than a power of two.
__device__ __forceinline__ int arena_bin(int cls, int len, int max_len) {
  const int i = (int)((long long)len * kClassBins / ((long long)max(max_len, len) + 1));
  return cls * kClassBins + (kClassBins - 1 - i);
}

// The deferred pairs, long ones first (their bounds take longest).
__device__ __forceinline__ int32_t deferred(const AlignArgs& a, int i, int nlong) {
  return i < nlong ? a.defer_long_list[i] : a.defer_list[i - nlong];
}

// One warp per pair: the bound on its score and with it the shared memory
// its rows need, which says who takes it.  Bound by the latency of its
// rows (about 70 instructions a score, one row after the other): as many
// warps as the shared memory for the packed sequences allows.
__global__ void __launch_bounds__(32 * kBandWarps) bound_kernel(const AlignArgs a, int32_t* key, int32_t* hist,
                                                                int warp_smem, int row_smem, int team_smem,
                                                                int ordered) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned FULL = 0xffffffffu;
  if (*(volatile const int32_t*)&a.ctrl->bad_input) return;
  const int lane = threadIdx.x & 31;
  unsigned char* my = smem + (threadIdx.x >> 5) * warp_smem;
  const int nlong = *(volatile const int32_t*)&a.ctrl->defer_long_count;
  const int total = nlong + *(volatile const int32_t*)&a.ctrl->defer_count;
  const bool pen_ok = a.xs <= kBandMaxPen && a.oes <= kBandMaxPen && a.es <= kBandMaxPen;
  const int ring_bytes = 64 * band_rows(a.xs, a.oes, a.es);
  const int max_len = *(volatile const int32_t*)&a.ctrl->max_len;
  int round = 0, flags[3];
  for (;;) {
    int i = 0;
    if (lane == 0) i = atomicAdd(&a.ctrl->bound_next, 1);
    i = __shfl_sync(FULL, i, 0);
    if (i >= total) return;
    const int32_t pair = deferred(a, i, nlong);
    const int n = a.plen[pair], m = a.tlen[pair];
    int T = 0, bin = arena_bin(max(n, m) > kMediumMaxLen ? kArenaLong : kArena, max(n, m), max_len);
    const bool lens_ok = n < kBandMaxLen && m < kBandMaxLen;
    if (pen_ok && lens_ok && ring_bytes + 4 * (band_words(n) + band_words(m)) <= warp_smem) {
      uint16_t* ring = reinterpret_cast<uint16_t*>(my);
      uint32_t* pw = reinterpret_cast<uint32_t*>(my + ring_bytes);
      uint32_t* tw = pw + band_words(n);
      const bool okp = team_pack32<1>(a.pat + a.poff[pair], n, pw, flags, round);
      const bool okt = team_pack32<1>(a.txt + a.toff[pair], m, tw, flags, round);
      if (!(okp && okt)) {
        if (lane == 0) {
          write_result(a, pair, 2, -1, 0, 0);
          key[pair] = kNoBin << kKeyBits;
        }
        continue;
      }
      BandGeo g = band_geo(a, n, m, 0);
      T = band_bound(pw, tw, g, a.xs, a.oes, a.es, min(band_worst(n, m, a.xs, a.oes, a.es), a.s_cap), ring);
      __syncwarp();
      g = band_geo(a, n, m, T);
      const int need = band_bytes(a, g), width = g.kmax - g.kmin + 1;
      const unsigned cost = (unsigned)(T + 1) * (unsigned)g.blocks();
      if (need <= row_smem && width <= kBandTeamWidth) bin = cost_bin(kWarp, cost);
      else if (need <= team_smem) bin = cost_bin(kTeam, cost);
    }
    if (!ordered) bin -= bin % kClassBins;
    if (lane == 0) {
      key[pair] = T | bin << kKeyBits;
      atomicAdd(&hist[bin], 1);
    }
  }
}

// The deferred pairs into their takers' lists, bin by bin: a block counts
// its pairs per bin in shared memory and reserves room for each bin with one
// global atomic (one per pair on so few addresses took 45 us for 178,000
// pairs).
constexpr int kPlaceBlock = 256, kPlaceItems = 8;
__global__ void __launch_bounds__(kPlaceBlock) place_kernel(const AlignArgs a, const int32_t* key, const int32_t* hist,
                                                            int32_t* cursor, int32_t* order, int32_t* arena_list,
                                                            int32_t* arena_long_list) {
  __shared__ int s_hist[kBandBins], s_start[kBandBins], s_count[kBandBins], s_base[kBandBins];
  const int nlong = a.ctrl->defer_long_count, total = nlong + a.ctrl->defer_count;
  if (*(volatile const int32_t*)&a.ctrl->bad_input || total == 0) return;
  const int t = threadIdx.x;
  if (t < kBandBins) s_hist[t] = hist[t];
  __syncthreads();
  if (t < kClasses * kClassBins) {
    // the band kernel's two classes share one list, the arena lists start at 0
    const int cls = t / kClassBins;
    const int first = cls < kArena ? 0 : cls * kClassBins;
    int at = 0;
    for (int b = first; b < t; ++b) at += s_hist[b];
    s_start[t] = at;
  }
  if (blockIdx.x == 0 && t < kClasses) {
    int c = 0;
    for (int b = 0; b < kClassBins; ++b) c += s_hist[t * kClassBins + b];
    int32_t* out[kClasses] = {&a.ctrl->team_count, &a.ctrl->warp_count, &a.ctrl->arena_count,
                              &a.ctrl->arena_long_count};
    *out[t] = c;
  }
  for (int i0 = blockIdx.x * kPlaceBlock * kPlaceItems; i0 < total; i0 += gridDim.x * kPlaceBlock * kPlaceItems) {
    if (t < kBandBins) s_count[t] = 0;
    __syncthreads();
    int32_t pair[kPlaceItems];
    int bin[kPlaceItems], rank[kPlaceItems];
#pragma unroll
    for (int j = 0; j < kPlaceItems; ++j) {
      const int i = i0 + j * kPlaceBlock + t;
      bin[j] = kNoBin;
      if (i < total) {
        pair[j] = deferred(a, i, nlong);
        bin[j] = key[pair[j]] >> kKeyBits;
        if (bin[j] != kNoBin) rank[j] = atomicAdd(&s_count[bin[j]], 1);
      }
    }
    __syncthreads();
    if (t < kBandBins && s_count[t]) s_base[t] = s_start[t] + atomicAdd(&cursor[t], s_count[t]);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPlaceItems; ++j) {
      if (bin[j] == kNoBin) continue;
      const int cls = bin[j] / kClassBins;
      int32_t* out = cls < kArena ? order : cls == kArena ? arena_list : arena_long_list;
      out[s_base[bin[j]] + rank[j]] = pair[j];
    }
    __syncthreads();
  }
}

// The exact wavefronts of the pairs the bound pass gave the band kernel:
// the wide ones first, each on the whole CTA, then a pair per warp.
// Persistent CTAs, pairs from queues.  Bound by instruction issue (82 % of
// the issue slots busy on mixed lengths).  Calls on the arena kernels before
// -> with the bound and the band: 200,000 mixed-length pairs (100-2,000 bp)
// 21.8 -> 11.8 ms, 4,000 x 10 kbp score-only 25.8 -> 6.6 ms, 2,000 x 10 kbp
// with CIGARs 17.7 -> 5.2 ms, 200,000 reads in 100-300 bp windows with free
// text ends 42.3 -> 2.0 ms.
// WARPS: a CTA of four, or of eight when few pairs are long (launch_band).
template <bool CIG, bool EF, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 32 / WARPS)
    band_kernel(const AlignArgs a, const int32_t* key, const int32_t* order, unsigned char* arena, long slot_bytes,
                int warp_smem) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (*(volatile const int32_t*)&a.ctrl->bad_input) return;
  const uint32_t absent = EF ? band_absent(a.xs, a.oes, a.es) : 0u;
  constexpr int kBoundMask = (1 << kKeyBits) - 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nteam = *(volatile const int32_t*)&a.ctrl->team_count;
  const int nwarp = *(volatile const int32_t*)&a.ctrl->warp_count;
  unsigned char* cta_slot = arena + (size_t)blockIdx.x * WARPS * (size_t)slot_bytes;
  if (nteam > 0) {
    BandShm* ts = reinterpret_cast<BandShm*>(smem);
    if (threadIdx.x == 0) ts->team.flags[0] = ts->team.flags[1] = ts->team.flags[2] = 0;
    __syncthreads();
    int round = 0;
    for (;;) {
      const int i = Team<WARPS>::broadcast(threadIdx.x == 0 ? atomicAdd(&a.ctrl->team_next, 1) : 0, &ts->team.bcast);
      if (i >= nteam) break;
      const int32_t pair = order[i];
      band_pair<WARPS, CIG, EF>(a, absent, pair, key[pair] & kBoundMask, smem + sizeof(BandShm), ts, round, cta_slot,
                                     WARPS * slot_bytes, &a.ctrl->overflow_count);
    }
    __syncthreads();
  }
  unsigned char* my = smem + warp * warp_smem;
  BandShm* ts = reinterpret_cast<BandShm*>(my);
  int round = 0;
  for (;;) {
    int i = 0;
    if (lane == 0) i = atomicAdd(&a.ctrl->warp_next, 1);
    i = __shfl_sync(0xffffffffu, i, 0);
    if (i >= nwarp) break;
    const int32_t pair = order[nteam + i];
    band_pair<1, CIG, EF>(a, absent, pair, key[pair] & kBoundMask, my + sizeof(BandShm), ts, round,
                          cta_slot + warp * slot_bytes, slot_bytes, &a.ctrl->overflow_count);
    __syncwarp();
  }
}

// Small calls: a warp per pair from its bytes to its CIGAR, the bound and the
// exact wavefronts one after the other, every pair of the call at once.  The
// time is one pair's latency: 37 reads of 100 bases took the ordering pass
// and the lane kernel 38 us (one lane runs a pair's cells in turn); the call
// went from 206 to 48 us with this kernel and its outputs in one wait.  Pairs
// longer than kDirectMaxLen, or whose rows do not fit, are deferred.
constexpr int kDirectMaxLen = 512;
template <bool CIG, bool EF>
__global__ void __launch_bounds__(32 * kBandWarps, 8)
    direct_kernel(const AlignArgs a, unsigned char* arena, long slot_bytes, int warp_smem) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (*(volatile const int32_t*)&a.ctrl->bad_input) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* my = smem + warp * warp_smem;
  BandShm* ts = reinterpret_cast<BandShm*>(my);
  my += sizeof(BandShm);
  const int room = warp_smem - (int)sizeof(BandShm);
  const bool pen_ok = a.xs <= kBandMaxPen && a.oes <= kBandMaxPen && a.es <= kBandMaxPen;
  const int w0 = (int)blockIdx.x * kBandWarps + warp, nw = (int)gridDim.x * kBandWarps;
  const uint32_t absent = EF ? band_absent(a.xs, a.oes, a.es) : 0u;
  int round = 0;
  for (int64_t pair = w0; pair < a.n; pair += nw) {
    const int n = a.plen[pair], m = a.tlen[pair];
    const int seq = (4 * (band_words(n) + band_words(m)) + 15) & ~15;
    bool mine = pen_ok && n <= kDirectMaxLen && m <= kDirectMaxLen && seq + 64 * band_rows(a.xs, a.oes, a.es) <= room;
    if (mine) {
      uint32_t* pw = reinterpret_cast<uint32_t*>(my);
      uint32_t* tw = pw + band_words(n);
      const bool okp = team_pack32<1>(a.pat + a.poff[pair], n, pw, ts->team.flags, round);
      const bool okt = team_pack32<1>(a.txt + a.toff[pair], m, tw, ts->team.flags, round);
      if (!(okp && okt)) {
        if (lane == 0) write_result(a, pair, 2, -1, 0, 0);
        __syncwarp();
        continue;
      }
      const int T = band_bound(pw, tw, band_geo(a, n, m, 0), a.xs, a.oes, a.es,
                               min(band_worst(n, m, a.xs, a.oes, a.es), a.s_cap),
                               reinterpret_cast<uint16_t*>(my + seq));
      __syncwarp();
      mine = band_bytes(a, band_geo(a, n, m, T)) <= room;
      if (mine)
        band_pair<1, CIG, EF>(a, absent, pair, T, my, ts, round, arena + (size_t)w0 * (size_t)slot_bytes, slot_bytes,
                              &a.ctrl->overflow_count, true);
    }
    if (!mine && lane == 0) defer_pair(a, pair);
    __syncwarp();
  }
}

// A sample's scores for the choice of a short-read store: the search for a
// bound alone, a warp per pair, up to the last bin.  The greedy bounds a lane
// works out for the ordering pass overshoot the score of 2 to 7 % of the
// paper's pairs, so that a choice by them had to leave a tenth of the pairs
// to the band kernels, at some 6 ns a pair.
__global__ void __launch_bounds__(32 * kBandWarps) sample_kernel(const AlignArgs a, int lmax, int warp_smem) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (*(volatile const int32_t*)&a.ctrl->bad_input) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t pair = (int64_t)blockIdx.x * kBandWarps + warp;
  if (pair >= a.n) return;
  const int n = a.plen[pair], m = a.tlen[pair];
  if (n > lmax || m > lmax) return;
  unsigned char* my = smem + warp * warp_smem;
  uint16_t* ring = reinterpret_cast<uint16_t*>(my);
  uint32_t* pw = reinterpret_cast<uint32_t*>(my + 64 * band_rows(a.xs, a.oes, a.es));
  uint32_t* tw = pw + band_words(n);
  int round = 0, flags[3];
  const bool okp = team_pack32<1>(a.pat + a.poff[pair], n, pw, flags, round);
  const bool okt = team_pack32<1>(a.txt + a.toff[pair], m, tw, flags, round);
  if (!(okp && okt)) return;
  const int cap = min(min(band_worst(n, m, a.xs, a.oes, a.es), a.s_cap), kSampleBins - 1);
  const int T = band_bound(pw, tw, band_geo(a, n, m, 0), a.xs, a.oes, a.es, cap, ring);
  if (lane == 0) atomicAdd(&a.ctrl->sample[T], 1);
}

using BandKernel = void (*)(const AlignArgs, const int32_t*, const int32_t*, unsigned char*, long, int);
template <int WARPS>
BandKernel band_kernel_as(bool cig, bool ef) {
  return cig ? (ef ? band_kernel<true, true, WARPS> : band_kernel<true, false, WARPS>)
             : (ef ? band_kernel<false, true, WARPS> : band_kernel<false, false, WARPS>);
}
BandKernel band_kernel_of(int warps, bool cig, bool ef) {
  return warps == kBandWarps ? band_kernel_as<kBandWarps>(cig, ef) : band_kernel_as<2 * kBandWarps>(cig, ef);
}

using DirectKernel = void (*)(const AlignArgs, unsigned char*, long, int);
DirectKernel direct_kernel_of(bool cig, bool ef) {
  return cig ? (ef ? direct_kernel<true, true> : direct_kernel<true, false>)
             : (ef ? direct_kernel<false, true> : direct_kernel<false, false>);
}

constexpr int kMaxSmem = 227 * 1024;

}  // namespace

cudaError_t band_plan(int device, BandPlan* plan) {
  cudaError_t e;
  // CTAs an SM (a CTA costs 1 KB of shared memory besides its own).  Eight of
  // four warps are what 64 registers allow, for short sequences (200,000 reads
  // in windows 1.93 ms, 2.00 with six); six for longer ones, so that rows of
  // some 460 diagonals fit a warp (mixed lengths 12.0 ms with eight, 11.8 with
  // six).  Under 4/6/2 (9 rows, 18 bytes a diagonal) a team's rows may be about
  // 1,500, 1,900 and 3,900 diagonals wide: the last size holds reads of 32,000
  // bases at up to some 4 % edits.  The second has a form with half as many
  // CTAs of eight warps, the last only that.
  const int len[BandPlan::kSizes] = {kDirectMaxLen, 12000, 12000, kBandMaxLen};
  const int warps[BandPlan::kSizes] = {kBandWarps, kBandWarps, 2 * kBandWarps, 2 * kBandWarps};
  const int want[BandPlan::kSizes] = {8, 6, 3, 3};
  int nsm = 0;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device))) return e;
  plan->nsm = nsm > 0 ? nsm : 1;
  for (int q = 0; q < 4; ++q) {
    for (int w : {kBandWarps, 2 * kBandWarps})
      if ((e = cudaFuncSetAttribute(band_kernel_of(w, q & 1, q & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kMaxSmem)))
        return e;
    if ((e = cudaFuncSetAttribute(direct_kernel_of(q & 1, q & 2), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kMaxSmem)))
      return e;
  }
  if ((e = cudaFuncSetAttribute(bound_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem))) return e;
  for (int i = 0; i < BandPlan::kSizes; ++i) {
    plan->max_len[i] = len[i];
    plan->warps[i] = warps[i];
    plan->smem[i] = (228 * 1024 / want[i] - 1024) & ~127;
    plan->per_sm[i] = want[i];
    for (int q = 0; q < 4; ++q) {
      int got = 0;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, band_kernel_of(warps[i], q & 1, q & 2),
                                                             32 * warps[i], plan->smem[i])))
        return e;
      plan->per_sm[i] = std::max(1, std::min(plan->per_sm[i], got));
    }
  }
  return cudaSuccess;
}

cudaError_t launch_sample_scores(const AlignArgs& a, int lmax, cudaStream_t st) {
  if (a.n <= 0 || std::max(a.xs, std::max(a.oes, a.es)) > kBandMaxPen) return cudaErrorInvalidValue;
  const int warp_smem = (64 * band_rows(a.xs, a.oes, a.es) + 8 * band_words(lmax) + 15) & ~15;
  if (kBandWarps * warp_smem > 48 * 1024) return cudaErrorInvalidValue;
  sample_kernel<<<(unsigned)((a.n + kBandWarps - 1) / kBandWarps), 32 * kBandWarps, kBandWarps * warp_smem, st>>>(
      a, lmax, warp_smem);
  return cudaGetLastError();
}

cudaError_t launch_direct(const AlignArgs& a, const BandPlan& plan, unsigned char* arena, long arena_bytes,
                          cudaStream_t st) {
  if (a.n <= 0) return cudaSuccess;
  const int smem = plan.smem[0];
  int64_t grid = std::min<int64_t>((int64_t)plan.nsm * plan.per_sm[0], (a.n + kBandWarps - 1) / kBandWarps);
  grid = std::max<int64_t>(1, std::min<int64_t>(grid, arena_bytes / (kBandWarps * (64L << 10))));
  const long slot = (long)(arena_bytes / (grid * kBandWarps)) & ~255L;
  const bool ef = (a.pb | a.pe | a.tb | a.te) != 0;
  direct_kernel_of(!a.score_only, ef)<<<(unsigned)grid, 32 * kBandWarps, smem, st>>>(a, arena, slot,
                                                                                     (smem / kBandWarps) & ~15);
  return cudaGetLastError();
}

int band_launches(const AlignArgs& a) { return std::max(a.xs, std::max(a.oes, a.es)) <= kBandMaxPen ? 3 : 2; }

cudaError_t launch_band(const AlignArgs& a, const BandPlan& plan, const BandBufs& b, int64_t pairs, int64_t nlong,
                        int max_len, bool ordered, unsigned char* arena, long arena_bytes, cudaStream_t st) {
  if (pairs <= 0) return cudaSuccess;
  int size = 0;
  while (size + 1 < BandPlan::kSizes && max_len > plan.max_len[size]) ++size;
  // fewer long pairs than CTAs of four warps: CTAs of eight (400 x 10 kbp with
  // CIGARs 2.7 -> 2.0 ms, 2,000 no faster: every row costs eight warps its
  // fixed part)
  if (size == 1 && max_len > kMediumMaxLen && nlong <= (int64_t)plan.nsm * plan.per_sm[1]) size = 2;
  const int warps = plan.warps[size], smem = plan.smem[size];
  const int warp_smem = (smem / warps) & ~15;
  cudaError_t e = cudaMemsetAsync(b.aux, 0, kBandAux * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  // bound pass: both packed sequences and the 32-diagonal rows a warp
  const int len = std::min(max_len, kBandMaxLen);
  const int rows = std::min(band_rows(a.xs, a.oes, a.es), band_rows(kBandMaxPen, kBandMaxPen, kBandMaxPen));
  const int bound_warp = (64 * rows + 8 * band_words(len) + 15) & ~15;
  const int bound_smem = std::min(kBandWarps * bound_warp, kMaxSmem);
  int bound_per_sm = std::min(std::max(1, 228 * 1024 / (bound_smem + 1024)), 12);
  const int64_t bound_grid = std::min<int64_t>((pairs + kBandWarps - 1) / kBandWarps, (int64_t)plan.nsm * bound_per_sm);
  bound_kernel<<<(unsigned)bound_grid, 32 * kBandWarps, bound_smem, st>>>(
      a, b.key, b.aux, (bound_smem / kBandWarps) & ~15, warp_smem - (int)sizeof(BandShm),
      smem - (int)sizeof(BandShm), ordered ? 1 : 0);
  if ((e = cudaGetLastError())) return e;
  const int64_t tiles = (pairs + kPlaceBlock * kPlaceItems - 1) / (kPlaceBlock * kPlaceItems);
  place_kernel<<<(unsigned)std::min<int64_t>(tiles, 2 * plan.nsm), kPlaceBlock, 0, st>>>(
      a, b.key, b.aux, b.aux + kBandBins, b.order, b.arena_list, b.arena_long_list);
  if ((e = cudaGetLastError()) || band_launches(a) < 3) return e;
  // CTAs: as many as are resident, at least 64 KiB of arena a warp, no more
  // than pairs (a team takes one at a time)
  int64_t grid = std::min<int64_t>((int64_t)plan.nsm * plan.per_sm[size], pairs);
  grid = std::max<int64_t>(1, std::min<int64_t>(grid, arena_bytes / (warps * (64L << 10))));
  const long slot = (long)(arena_bytes / (grid * warps)) & ~255L;
  const bool ef = (a.pb | a.pe | a.tb | a.te) != 0;
  band_kernel_of(warps, !a.score_only, ef)<<<(unsigned)grid, 32 * warps, smem, st>>>(a, b.key, b.order, arena, slot,
                                                                                     warp_smem);
  return cudaGetLastError();
}

}  // namespace wfa
