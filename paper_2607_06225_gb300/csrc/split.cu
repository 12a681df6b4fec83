// split.cu -- the queue, the results and the launch of pairs run a warp per strip
// (k_split.cuh).
#include <algorithm>

#include "k_split.cuh"
#include "k_strip.cuh"
#include "plan_pair.h"

namespace filtr {
namespace {

struct SplitPlanArgs {
  const uint32_t *order;       // the pairs of the batch by shape, or nullptr (one pair, id 0)
  uint32_t begin, count;       // their slice (captured pipeline: from gsum)
  const GraphDesc *gd;
  const DevPlanSummary *gsum;
  int gshape;
  const uint32_t *q_len;
  int rows;                    // rows per strip
  uint32_t max_strips;
  SplitArgs a;
};

// Block 0: the queue's order (pairs counting-sorted by strips, most first).  Every
// block: its share of the hand-over words, cleared.
__global__ void __launch_bounds__(1024) k_split_plan(const SplitPlanArgs s) {
  extern __shared__ uint32_t hist[];  // per strip count: pairs, then pairs with more strips
  if (s.gd && s.gd->abort) return;
  uint32_t begin = s.begin, n = s.count;
  if (s.gsum) {
    begin = 0;
    for (int k = 0; k < s.gshape; ++k) begin += s.gsum->count[k];
    n = s.gsum->count[s.gshape];
  }
  const uint32_t *ql = s.gd ? s.gd->b.q_len : s.q_len;
  const uint64_t words = (uint64_t)n * SPLIT_SLOTS * s.a.ring_stride;
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < words;
       t += (uint64_t)gridDim.x * blockDim.x)
    s.a.ring[t] = 0;
  if (blockIdx.x != 0) return;
  const uint32_t tid = threadIdx.x;
  if (tid == 0) *s.a.err = 0;
  if (n == 1) {  // one pair: strip s is item s
    const uint32_t p = s.order ? s.order[begin] : 0u;
    const uint32_t ns = (uint32_t)(((uint64_t)ql[p] + s.rows - 1) / s.rows);
    for (uint32_t x = tid; x <= ns; x += blockDim.x) s.a.sstart[x] = x;
    if (tid == 0) {
      s.a.sorted[0] = p;
      s.a.hdr[0] = 1;
      s.a.hdr[1] = s.a.hdr[2] = ns;
      s.a.hdr[3] = 0;
    }
    return;
  }
  const uint32_t cap = s.max_strips;
  for (uint32_t x = tid; x <= cap; x += blockDim.x) hist[x] = 0;
  __syncthreads();
  for (uint32_t t = tid; t < n; t += blockDim.x)
    atomicAdd(&hist[min((uint32_t)(((uint64_t)ql[s.order[begin + t]] + s.rows - 1) / s.rows), cap)], 1u);
  __syncthreads();
  if (tid == 0) {
    uint32_t more = 0, tall = 0;
    for (int b = (int)cap; b >= 0; --b) {  // hist[b]: pairs with more than b strips
      const uint32_t here = hist[b];
      if (here && !tall) tall = (uint32_t)b;
      hist[b] = more;
      more += here;
    }
    uint32_t at = 0;
    for (uint32_t x = 0; x < tall; ++x) {
      s.a.sstart[x] = at;
      at += hist[x];
    }
    s.a.sstart[tall] = at;
    s.a.hdr[0] = n;
    s.a.hdr[1] = tall;
    s.a.hdr[2] = at;
    s.a.hdr[3] = 0;
  }
  __syncthreads();
  for (uint32_t t = tid; t < n; t += blockDim.x) {
    const uint32_t p = s.order[begin + t];
    const uint32_t ns = min((uint32_t)(((uint64_t)ql[p] + s.rows - 1) / s.rows), cap);
    s.a.sorted[atomicAdd(&hist[ns], 1u)] = p;  // after the pairs with more strips
  }
}

// A warp per pair: the strips' best cells and the corner make the result.
__global__ void __launch_bounds__(128) k_split_finish(const SplitArgs a, int rows) {
  const GraphDesc *gd = a.f.gd;
  if (gd && gd->abort) return;
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  const BatchDev &b = gd ? gd->b : a.f.b;
  filtr_result *out = gd ? gd->out : a.f.out;
  for (uint32_t rank = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; rank < a.hdr[0]; rank += nw) {
    const uint32_t p = a.sorted[rank];
    const int M = (int)b.q_len[p], N = (int)b.r_len[p], ns = (M + rows - 1) / rows;
    LaneBest best{0, INT_MAX, INT_MAX};
    int endH = NEG;
    for (int s = lane; s < ns; s += 32) {
      const int4 r = a.res[a.sstart[s] + rank];
      if (r.x > best.v || (r.x == best.v && (r.y < best.i || (r.y == best.i && r.z < best.j))))
        best = LaneBest{r.x, r.y, r.z};
      if (s == ns - 1) endH = r.w;
    }
    best = warp_best(best);
    endH = __shfl_sync(STRIP_FULLMASK, endH, (ns - 1) & 31);
    if (lane != 0) continue;
    filtr_result res{};
    res.cells = band_cells((uint32_t)M, (uint32_t)N, a.f.sp);
    if (*(volatile int *)a.err) {
      if (a.timed_out) *a.timed_out = 1;
      res.status = FILTR_ST_TIMEOUT;
      res.cells = 0;
    } else if (a.f.sp.mode == FILTR_LOCAL) {
      if (best.v > 0) {
        res.score = best.v;
        res.q_end = best.i;
        res.r_end = best.j;
        res.q_begin = res.r_begin = -1;
        res.status = FILTR_ST_OK;
      } else {
        res.status = FILTR_ST_EMPTY;
      }
    } else {
      int64_t lo = -(int64_t)M - 1, hi = (int64_t)N + 1;
      if (a.f.sp.use_band) band_limits(M, N, a.f.sp.band, a.f.sp.band_literal, &lo, &hi);
      res.q_end = M;
      res.r_end = N;
      if ((int64_t)N - M >= lo && (int64_t)N - M <= hi && endH > NEG_HALF)
        res.score = endH;
      else
        res.status = FILTR_ST_UNREACHABLE;
    }
    out[p] = res;
    if (a.f.fwd) a.f.fwd[p] = FwdOut{res.score, res.q_end, res.r_end, res.status};
  }
}

}  // namespace

SplitSpace split_space(uint64_t n, uint64_t ns, uint64_t stride) {
  SplitSpace s;
  size_t at = 0;
  auto part = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) / 256 * 256;
    return o;
  };
  s.hdr = part(256);
  s.sstart = part((ns + 2) * 4);
  s.sorted = part(n * 4);
  s.ring = part(n * SPLIT_SLOTS * stride * 8);
  s.res = part(n * ns * 16);
  s.bytes = at;
  return s;
}

void split_bind(SplitArgs *a, char *mem, const SplitSpace &sp, uint32_t stride) {
  a->hdr = reinterpret_cast<uint32_t *>(mem + sp.hdr);
  a->err = reinterpret_cast<int *>(mem + sp.hdr + 64);
  a->sstart = reinterpret_cast<uint32_t *>(mem + sp.sstart);
  a->sorted = reinterpret_cast<uint32_t *>(mem + sp.sorted);
  a->ring = reinterpret_cast<unsigned long long *>(mem + sp.ring);
  a->ring_stride = stride;
  a->res = reinterpret_cast<int4 *>(mem + sp.res);
}

cudaError_t launch_split(const SplitLaunch &l, cudaStream_t st) {
  SplitPlanArgs pa{};
  pa.order = l.a.f.order;
  pa.begin = 0;
  pa.count = (uint32_t)l.count;
  pa.gd = l.a.f.gd;
  pa.gsum = l.a.f.gsum;
  pa.gshape = l.a.f.gshape;
  pa.q_len = l.a.f.b.q_len;
  pa.rows = split_rows(l.packed, l.R);
  pa.max_strips = l.max_strips;
  pa.a = l.a;
  const size_t smem = l.count == 1 ? 0 : ((size_t)l.max_strips + 2) * 4;
  const uint64_t words = (uint64_t)l.count * SPLIT_SLOTS * l.a.ring_stride;
  const unsigned blocks = (unsigned)std::min<uint64_t>(304, 1 + words / 8192);
  k_split_plan<<<blocks, 1024, smem, st>>>(pa);
  cudaError_t e = cudaGetLastError();
  const int grid = std::min(l.grid, SPLIT_MAX_WARPS / FULL_WARPS);
  if (e == cudaSuccess)
    e = l.packed ? launch_split_pack(l.a, l.R, grid, st) : launch_split_full(l.a, l.R, grid, st);
  if (e != cudaSuccess) return e;
  k_split_finish<<<(unsigned)std::min<int64_t>((l.count + 3) / 4, 1 << 16), 128, 0, st>>>(l.a, pa.rows);
  return cudaGetLastError();
}

}  // namespace filtr
