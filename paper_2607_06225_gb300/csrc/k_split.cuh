// k_split.cuh -- tiled pairs with a warp per row strip: the strips of one pair run
// at the same time on different warps, each a few columns behind the strip
// above it.
//
// A batch whose pairs do not fill the device leaves most warps idle when a warp
// takes a whole pair, and its time is that of its longest pair.  Here the unit
// of work is one strip of 32 * R rows (R = 8, or 16 in the packed tile, or 4 for one
// long banded pair), so a
// pair of M rows uses M / (32 R) warps and takes about N + lag steps instead of
// strips x N.  The cells, traceback words and results are those of k_full /
// k_pack with the same R.
//
// Queue.  Items (strip s, pair) are taken in the order of s, then of the pairs by
// strip count, from one counter (k_split_plan lays the order out): strip s's
// predecessor s - 1 is earlier in the queue, so a warp only ever waits for an item
// that a running warp holds, and the first unfinished item never waits: no
// deadlock, whatever part of the grid is resident.  With more pairs than warps
// the strips above are mostly done before the ones below start.
//
// Hand-over.  Lane 31 of strip s stores its bottom row's (H, F) of each column as
// one 64-bit word whose top 11 bits are a tag (the strip's turn in its slot);
// a relaxed 64-bit store is atomic, so the word carries its own "ready" flag and
// neither side needs a fence.  (Progress words with release stores every 16
// columns made each release wait for the lane's traceback stores: 0.46 us per
// 8-row step of an 80 kbp banded pair.)  The consumer loads up to 32 columns at
// once and takes the leading ones whose tag is right.  Two slots per pair do: strip
// s + 2 writes column c of strip s's slot only after strip s + 1 published
// its column c, which it did after reading strip s's.  In a banded pair, where
// the slots are indexed from each strip's first column, strip s + 2's index x is
// a later column than strip s's, and past strip s + 1's last column strip s + 1
// is finished.  A warp may wait for strip s while its slot still holds a word of
// strip s - 2t; then strips s - 2t + 2 .. s + 1 are all unfinished, each held by a
// warp of its own, so tags of 2047 turns never meet again within SPLIT_MAX_WARPS
// warps.
//
// Every wait is bounded by a time limit on %globaltimer; a wait that runs out sets
// the error word, after which no wait waits, and the launch's pairs report
// FILTR_ST_TIMEOUT.
#pragma once

#include "filtr_internal.h"
#include "plan.h"

namespace filtr {

constexpr int SPLIT_SLOTS = 2;
constexpr int SPLIT_TAG = 53;              // the tag's first bit
constexpr int SPLIT_TURNS = 2047;
constexpr int SPLIT_MAX_WARPS = 2 * SPLIT_TURNS - 16;
// Which batches run a warp per strip (whole calls, plain against split).
// Up to SPLIT_LATENCY_PAIRS, whose shapes the plain path launches one after the other:
// 64 protein pairs of 100-1000 3.74 / 0.57 ms, 16 banded pairs of 100-600 0.55 / 0.22.
// More pairs are planned on the device and their shapes run side by side: unbanded ones
// split up to SPLIT_MAX_PAIRS when the tallest pair has more than SPLIT_TALL_ROWS rows
// and would outlast the batch (twice a warp's share; 608 pairs of 100-1000 0.73 / 0.85),
// banded ones up to SPLIT_MAX_BANDED from SPLIT_BAND_ROWS rows and half a warp's share
// (256 of 100-1500, band 256, traceback 2.02 / 1.27 ms, 3000 of them 4.26 / 3.14; but
// 3000 scores of 100-600 0.56 / 0.62 and 20,000 of 100-1500 8.29 / 9.15).
constexpr unsigned long long SPLIT_TIMEOUT_NS = 20ull * 1000 * 1000 * 1000;  // 20 s without progress
constexpr uint32_t SPLIT_LATENCY_PAIRS = 255;
constexpr uint32_t SPLIT_MAX_PAIRS = 4096;
constexpr uint32_t SPLIT_TALL_ROWS = 2048;
constexpr uint32_t SPLIT_MAX_BANDED = 16384;
constexpr uint32_t SPLIT_BAND_ROWS = 1408;
// Captured pipelines run their shapes side by side and know only bounds.  Plain against
// split, local pairs with traceback: 64 of up to 700 0.39 / 0.36 ms, of up to 2000
// 1.59 / 0.96; 256 of up to 1000 0.62 / 0.82, of up to 2000 2.03 / 1.57; banded (256):
// 16 of up to 300 0.26 / 0.25, 256 of up to 600 0.55 / 0.64, of up to 1500 2.09 / 1.67.
// Scores only: 40 local pairs of up to 1100 0.260 / 0.271, of up to 1220 0.311 / 0.302, of
// up to 1500 0.60 / 0.37; 64 banded (60) of up to 380 0.138 / 0.149, of up to 620 0.201 / 0.187.
inline bool split_graph(bool band, bool traceback, uint32_t max_pairs, uint32_t max_len) {
  if (max_pairs <= 64) return band ? traceback || max_len > 512 : max_len > (traceback ? 1024u : 1152u);
  return band ? max_pairs <= SPLIT_MAX_PAIRS && max_len > 1024
              : max_pairs <= SPLIT_LATENCY_PAIRS && max_len > 1408;
}

struct SplitArgs {
  FullArgs f;                  // batch, parameters, outputs, traceback (order, counter unused)
  uint32_t *hdr;               // [0] pairs, [1] strips of the tallest, [2] items, [3] queue cursor
  uint32_t *sstart;            // first item of strip s, s = 0 .. hdr[1]
  uint32_t *sorted;            // pair ids, most strips first
  unsigned long long *ring;    // per pair (by rank): SPLIT_SLOTS slots of ring_stride words
  uint32_t ring_stride;
  int4 *res;                   // per item: best cell (v, i, j) and H at the corner
  int *err;
  int *timed_out;              // set to 1 with the results when err was set (nullptr: nobody asks)
  unsigned long long timeout_ns;
  int withhold;                // test hook: strip 0 never publishes (forces the timeout)
};

#ifdef __CUDACC__
namespace {

__device__ __forceinline__ unsigned long long split_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// One strip's two ends of the hand-over.  `at`: index of a column in its slot.
struct SplitLink {
  static constexpr bool FETCH = true;
  const unsigned long long *src;
  unsigned long long *dst;
  unsigned tag_src;
  unsigned long long tag_dst;  // in place
  int *err;
  unsigned long long timeout_ns;
  bool dead, mute;

  __device__ void open(const SplitArgs &a, uint32_t rank, int s) {
    unsigned long long *base = a.ring + (uint64_t)rank * SPLIT_SLOTS * a.ring_stride;
    src = base + (uint64_t)((s + SPLIT_SLOTS - 1) % SPLIT_SLOTS) * a.ring_stride;
    dst = base + (uint64_t)(s % SPLIT_SLOTS) * a.ring_stride;
    tag_src = s > 0 ? (unsigned)((s - 1) / SPLIT_SLOTS % SPLIT_TURNS + 1) : 0u;
    tag_dst = (unsigned long long)(s / SPLIT_SLOTS % SPLIT_TURNS + 1) << SPLIT_TAG;
    err = a.err;
    timeout_ns = a.timeout_ns;
    dead = false;
    mute = a.withhold != 0 && s == 0;
  }
  // lane x loads word at + x (x < left); returns how many leading words are
  // ready, waiting for the first
  __device__ int poll(int at, int left, unsigned long long &w) {
    const int x = threadIdx.x & 31;
    unsigned long long t0 = 0;
    for (;;) {
      w = 0;
      if (x < left)
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(src + at + x) : "memory");
      const unsigned ready = __ballot_sync(0xffffffffu, (unsigned)(w >> SPLIT_TAG) == tag_src);
      if (dead) return 32;
      if (ready & 1u) return ready == 0xffffffffu ? 32 : __ffs(~ready) - 1;
      int stop = 0;
      if (x == 0) {
        const unsigned long long now = split_timer();
        if (t0 == 0) t0 = now;
        if (*(volatile int *)err) {
          stop = 1;
        } else if (now - t0 > timeout_ns) {
          atomicExch(err, 1);
          stop = 1;
        }
      }
      if (__shfl_sync(0xffffffffu, stop, 0)) {
        dead = true;
        return 32;
      }
      __nanosleep(64);
    }
  }
  __device__ void put(int at, unsigned long long v) {
    if (!mute)
      asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(dst + at), "l"(v | tag_dst) : "memory");
  }
};

// The next item: false when the queue is empty.  k: its number, s its strip,
// rank the pair's rank, p the pair.
__device__ __forceinline__ bool split_next(const SplitArgs &a, uint32_t &k, int &s, uint32_t &rank,
                                           uint32_t &p) {
  k = 0;
  if ((threadIdx.x & 31) == 0) k = atomicAdd(a.hdr + 3, 1u);
  k = __shfl_sync(0xffffffffu, k, 0);
  if (k >= a.hdr[2]) return false;
  int lo = 0, hi = (int)a.hdr[1];  // sstart[lo] <= k < sstart[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.sstart[mid] <= k)
      lo = mid;
    else
      hi = mid;
  }
  s = lo;
  rank = k - a.sstart[lo];
  p = a.sorted[rank];
  return true;
}

}  // namespace
#endif

// ---- host side (split.cu) ----------------------------------------------------
// What one split launch covers.  count: its pairs, or -1 to take them from the
// device plan's summary (captured pipeline: f.gd, f.gsum and f.gshape set).
struct SplitLaunch {
  SplitArgs a;
  bool packed;
  int R;
  int64_t count;          // pairs (an upper bound when taken from the device plan)
  uint32_t max_strips;    // upper bound of a pair's strips
  int grid;
};
// Device memory of one split launch: pairs <= n, strips <= ns, references <= max_n.
struct SplitSpace {
  size_t hdr, sstart, sorted, ring, res, bytes;
};
SplitSpace split_space(uint64_t n, uint64_t ns, uint64_t stride);
// the largest strip count a launch over several pairs sorts by
constexpr uint32_t SPLIT_MAX_STRIPS = 12000;
void split_bind(SplitArgs *a, char *mem, const SplitSpace &sp, uint32_t stride);
cudaError_t launch_split(const SplitLaunch &l, cudaStream_t st);
cudaError_t launch_split_full(const SplitArgs &a, int R, int grid, cudaStream_t st);  // R = 8; banded: or 4
cudaError_t launch_split_pack(const SplitArgs &a, int R, int grid, cudaStream_t st);
int split_full_blocks_per_sm(int R, const ScoreParams &sp);
int split_pack_blocks_per_sm(int R, const ScoreParams &sp);
inline int split_rows(bool packed, int R) { return 32 * (packed || R == 4 ? R : 8); }

}  // namespace filtr
