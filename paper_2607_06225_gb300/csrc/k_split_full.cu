// k_split_full.cu -- a warp per row strip, int32 tile (k_split.cuh, k_strip.cuh).
#include "k_split.cuh"
#include "k_strip.cuh"
#include "plan_pair.h"

namespace filtr {
namespace {

// H in 30 bits above minus infinity (finite scores stay below 2^28), and H - F in
// 23: F opens from the row above, so a finite F is at most the largest score plus
// two opened gaps (below 2^23) short of H; the largest difference stands for an
// F of minus infinity
struct FullLink : SplitLink {
  static constexpr unsigned DMAX = 0x7fffffu;
  int jlo, prev_jlo;  // slots are indexed from each strip's first column
  __device__ int fetch(int j, int jmax, int2 &v) {
    unsigned long long w;
    const int n = poll(j - prev_jlo, jmax - j + 1, w);
    v.x = (int)(w & 0x3fffffffu) + NEG;
    const unsigned d = (unsigned)(w >> 30) & DMAX;
    v.y = d == DMAX ? NEG : v.x - (int)d;
    return n;
  }
  __device__ void out(int j, int H, int F) {
    put(j - jlo, (unsigned long long)(unsigned)(max(H, NEG) - NEG) |
                     (unsigned long long)min((unsigned)(H - F), DMAX) << 30);
  }
};

template <int R, bool LOCAL, bool AFFINE, bool TB, bool BAND>
__global__ void __launch_bounds__(FULL_WARPS * 32) k_split_full(const SplitArgs a) {
  constexpr int HS = 32 * R;
  extern __shared__ __align__(16) int8_t smem[];
  const GraphDesc *gd = a.f.gd;
  if (gd && gd->abort) return;
  const int A = a.f.sp.alphabet;
  int8_t *s_sub = smem;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < A * A; t += blockDim.x) s_sub[t] = a.f.sp.subst[t];
  __syncthreads();

  uint32_t k, rank, p;
  int s;
  while (split_next(a, k, s, rank, p)) {
    const BatchDev &b = gd ? gd->b : a.f.b;
    StripPair P;
    P.M = (int)b.q_len[p];
    P.N = (int)b.r_len[p];
    P.q = b.q_seq + b.q_off[p];
    P.r = b.r_seq + b.r_off[p];
    P.lo = -P.M - 1;
    P.hi = P.N + 1;
    if (BAND) {
      int64_t l64, h64;
      band_limits(P.M, P.N, a.f.sp.band, a.f.sp.band_literal, &l64, &h64);
      P.lo = (int)(l64 < -(int64_t)P.M - 1 ? -(int64_t)P.M - 1 : l64);
      P.hi = (int)(h64 > (int64_t)P.N + 1 ? (int64_t)P.N + 1 : h64);
    }
    P.one = (A > 0) ? 1 : 0;  // 1, unknown to the compiler
    P.o = a.f.sp.o;
    P.e = a.f.sp.e;
    P.A = A;
    P.s_sub = s_sub;
    P.prof = smem + 512 + wib * (A * HS);
    P.tb = TB ? a.f.tb + a.f.tbl[p].off : nullptr;
    const int M = P.M, N = P.N, nstrips = (M + HS - 1) / HS;
    LaneBest best{0, INT_MAX, INT_MAX};
    int endH = NEG;
    int64_t jl, jh, pjl = 1, pjh = 0;
    strip_cols((int64_t)s * HS, HS, M, N, BAND, P.lo, P.hi, &jl, &jh);
    if (jl <= jh) {  // else no band cell in this strip or below
      if (s > 0) strip_cols((int64_t)(s - 1) * HS, HS, M, N, BAND, P.lo, P.hi, &pjl, &pjh);
      int64_t base = 0;  // traceback words of the strips above
      if (TB && BAND) {
        for (int x = lane; x < s; x += 32) {
          int64_t xl, xh;
          strip_cols((int64_t)x * HS, HS, M, N, true, P.lo, P.hi, &xl, &xh);
          base += strip_tb_words(xl, xh, R);
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) base += __shfl_xor_sync(STRIP_FULLMASK, base, off);
      } else if (TB) {
        base = s * strip_tb_words(1, N, R);
      }
      FullLink io;
      io.open(a, rank, s);
      io.jlo = (int)jl;
      io.prev_jlo = (int)pjl;
      strip_pass<R, LOCAL, AFFINE, TB, BAND>(P, s, (int)jl, (int)jh, (int)pjl, (int)pjh, base, io,
                                             best, endH);
    }
    if (LOCAL) best = warp_best(best);
    if (!LOCAL && s == nstrips - 1) endH = __shfl_sync(STRIP_FULLMASK, endH, ((M - 1) % HS) / R);
    if (lane == 0) a.res[k] = make_int4(best.v, best.i, best.j, endH);
  }
}

template <int R, bool LOCAL, bool AFFINE, bool TB, bool BAND>
cudaError_t launch_sf(const SplitArgs &a, int grid, cudaStream_t st) {
  auto k = k_split_full<R, LOCAL, AFFINE, TB, BAND>;
  k<<<grid, FULL_WARPS * 32, full_smem_bytes(R, a.f.sp.alphabet), st>>>(a);
  return cudaGetLastError();
}
template <int R, bool LOCAL, bool AFFINE, bool TB, bool BAND>
int occ_sf(const ScoreParams &sp) {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_split_full<R, LOCAL, AFFINE, TB, BAND>, FULL_WARPS * 32,
                                                full_smem_bytes(R, sp.alphabet));
  return nb;
}

}  // namespace

#define FILTR_SPLIT_CASES(X) \
  X(false, false, false, false) X(false, false, false, true) X(false, false, true, false) \
  X(false, false, true, true) X(false, true, false, false) X(false, true, false, true) \
  X(false, true, true, false) X(false, true, true, true) X(true, false, false, false) \
  X(true, false, false, true) X(true, false, true, false) X(true, false, true, true) \
  X(true, true, false, false) X(true, true, false, true) X(true, true, true, false) \
  X(true, true, true, true)

cudaError_t launch_split_full(const SplitArgs &a, int R, int grid, cudaStream_t st) {
  const ScoreParams &sp = a.f.sp;
  const bool L = sp.mode == FILTR_LOCAL, AF = sp.affine != 0, T = sp.traceback != 0, B = sp.use_band != 0;
#define FILTR_CASE(l, af, t, b) \
  if (L == l && AF == af && T == t && B == b) { \
    if (R == 4 && b) return launch_sf<b ? 4 : 8, l, af, t, b>(a, grid, st); \
    if (R == 8) return launch_sf<8, l, af, t, b>(a, grid, st); \
  }
  FILTR_SPLIT_CASES(FILTR_CASE)
#undef FILTR_CASE
  return cudaErrorInvalidValue;
}

int split_full_blocks_per_sm(int R, const ScoreParams &sp) {
  const bool L = sp.mode == FILTR_LOCAL, AF = sp.affine != 0, T = sp.traceback != 0, B = sp.use_band != 0;
#define FILTR_CASE(l, af, t, b) \
  if (L == l && AF == af && T == t && B == b) { \
    if (R == 4 && b) return occ_sf<b ? 4 : 8, l, af, t, b>(sp); \
    if (R == 8) return occ_sf<8, l, af, t, b>(sp); \
  }
  FILTR_SPLIT_CASES(FILTR_CASE)
#undef FILTR_CASE
  return 0;
}

}  // namespace filtr
