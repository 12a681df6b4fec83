// k_split_pack.cu -- a warp per row strip, int16x2 tile (k_split.cuh,
// k_pack_impl.cuh).
#include "k_pack_impl.cuh"
#include "k_split.cuh"

namespace filtr {
namespace {

struct PackLink : SplitLink {
  __device__ int fetch(int j, int jmax, uint32_t &v) {
    unsigned long long w;
    const int n = poll(j - 1, jmax - j + 1, w);
    v = (uint32_t)w;
    return n;
  }
  __device__ void out(int j, uint32_t hf) { put(j - 1, hf); }
};

template <int R, bool LOCAL, bool AFFINE, bool TB>
__global__ void __launch_bounds__(FULL_WARPS * 32) k_split_pack(const SplitArgs a) {
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
    PackPair PP;
    PP.M = (int)b.q_len[p];
    PP.N = (int)b.r_len[p];
    PP.q = b.q_seq + b.q_off[p];
    PP.r = b.r_seq + b.r_off[p];
    PP.o = a.f.sp.o;
    PP.e = a.f.sp.e;
    PP.A = A;
    PP.B = pack_bias(a.f.sp.mode, a.f.sp.o, a.f.sp.e, a.f.sp.smin, a.f.sp.smax, PP.M, PP.N);
    PP.one = (A > 0) ? 1u : 0u;  // 1, unknown to the compiler
    PP.s_sub = s_sub;
    PP.prof = smem + 512 + wib * (A * pack_prof_stride(R));
    PP.tb = TB ? a.f.tb + a.f.tbl[p].off : nullptr;
    const int M = PP.M, nstrips = (M + HS - 1) / HS;
    Best best{0, INT_MAX, INT_MAX};
    int endH = 0;
    PackLink io;
    io.open(a, rank, s);
    pack_strip<R, LOCAL, AFFINE, TB>(PP, s, TB ? (int64_t)s * pack_strip_tb_words(1, PP.N, R) : 0, io, best,
                                     endH);
    if (LOCAL) {
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        const int ov = __shfl_xor_sync(PFULL, best.v, off);
        const int oi = __shfl_xor_sync(PFULL, best.i, off);
        const int oj = __shfl_xor_sync(PFULL, best.j, off);
        best_put(best, ov, oi, oj);
      }
    } else if (s == nstrips - 1) {
      endH = __shfl_sync(PFULL, endH, ((M - 1) % HS) / R);
    }
    if (lane == 0) a.res[k] = make_int4(best.v, best.i, best.j, endH);
  }
}

template <int R, bool LOCAL, bool AFFINE, bool TB>
cudaError_t launch_sp(const SplitArgs &a, int grid, cudaStream_t st) {
  auto k = k_split_pack<R, LOCAL, AFFINE, TB>;
  k<<<grid, FULL_WARPS * 32, pack_smem_bytes(R, a.f.sp.alphabet), st>>>(a);
  return cudaGetLastError();
}
template <int R, bool LOCAL, bool AFFINE, bool TB>
int occ_sp(const ScoreParams &sp) {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_split_pack<R, LOCAL, AFFINE, TB>, FULL_WARPS * 32,
                                                pack_smem_bytes(R, sp.alphabet));
  return nb;
}

template <int R>
cudaError_t launch_spr(const SplitArgs &a, int grid, cudaStream_t st) {
  const bool L = a.f.sp.mode == FILTR_LOCAL, AF = a.f.sp.affine != 0, T = a.f.sp.traceback != 0;
#define FILTR_CASE(l, af, t) \
  if (L == l && AF == af && T == t) return launch_sp<R, l, af, t>(a, grid, st);
  FILTR_PACK_CASES(FILTR_CASE)
#undef FILTR_CASE
  return cudaErrorInvalidValue;
}
template <int R>
int occ_spr(const ScoreParams &sp) {
  const bool L = sp.mode == FILTR_LOCAL, AF = sp.affine != 0, T = sp.traceback != 0;
#define FILTR_CASE(l, af, t) \
  if (L == l && AF == af && T == t) return occ_sp<R, l, af, t>(sp);
  FILTR_PACK_CASES(FILTR_CASE)
#undef FILTR_CASE
  return 0;
}

}  // namespace

cudaError_t launch_split_pack(const SplitArgs &a, int R, int grid, cudaStream_t st) {
  return R == 8 ? launch_spr<8>(a, grid, st) : R == 16 ? launch_spr<16>(a, grid, st) : cudaErrorInvalidValue;
}
int split_pack_blocks_per_sm(int R, const ScoreParams &sp) {
  return R == 8 ? occ_spr<8>(sp) : R == 16 ? occ_spr<16>(sp) : 0;
}

}  // namespace filtr
