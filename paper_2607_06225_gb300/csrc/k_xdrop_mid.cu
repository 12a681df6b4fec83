// k_xdrop_mid.cu -- the antidiagonal sweep over Table 1's M/I/D recurrence
// (k_xdrop_impl.cuh with the gap-open source moved from H to the diagonal state
// M), with or without an X-drop threshold, in a translation unit of its own.
#include <algorithm>

#include "k_xdrop_impl.cuh"

namespace filtr {

cudaError_t launch_mid_w(const FullArgs &a, int W, int grid, uint32_t *overflow,
                         uint32_t *n_overflow, cudaStream_t s) {
  return launch_any_w<2>(a, W, grid, overflow, n_overflow, s);
}

// No more than 12 warps per SM with traceback and 16 without, though the registers hold
// 20: the sweep is bound by issue, so more pairs at once only slow each other, and the
// longest ends the launch.  Limited (and not): 2471 reads of 1-4 kbp 9.8 (12.0) ms, 2785 of 3-12
// kbp 30.7 (33.6), with traceback; 4000 of 1-3 kbp, score only, 7.75 (8.1); but 8000 14.4 (13.7).
int mid_blocks_per_sm(int W, const ScoreParams &sp) {
  return std::min(occ_any_w<2>(W, sp), std::max(1, (sp.traceback ? 12 : 16) / (W == 1 ? 4 : W)));
}

}  // namespace filtr
