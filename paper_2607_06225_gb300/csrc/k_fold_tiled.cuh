// k_fold_tiled.cuh -- Nussinov folding as a blocked max-plus product, two cells
// per register (int16x2), with X-drop on the spans.
//
// What bounds it.  A fold of n bases evaluates about n^3 / 6 split terms
// F(i,m) + F(m+1,j).  A kernel that walks each cell's terms one by one
// (k_fold) loads both operands of every term from the table and waits for them.
// Here most terms run as a register-tiled product from shared memory (one DPX
// add-max takes two terms), and the table holds 16-bit values (F <= n / 2 <=
// 2048).  Left are the product's fixed-latency chains and the barrier of each span
// (at 300 bases: ALU pipe 42%, shared memory 34%; 1024 sequences 8.95 -> 1.35 ms).
//
// Layout.  With half-open intervals, G(i,e) = F(i, e-1) is G(i,e) = max over
// i < m < e of G(i,m) + G(m,e).  One symmetric matrix Q[a][b] =
// G(min(a,b), max(a,b)) of 16-bit words holds the table: row i read along m gives
// G(i,m), row e read along m gives G(m,e), so both operands of a term are
// contiguous in m and a 32-bit word holds the operands of two terms.  Cells not
// computed yet, pruned or outside the domain are FOLD_NEG; a term that is not
// a split of (i, e) (m <= i or m >= e) has one operand longer than the cell
// itself, so it is FOLD_NEG too and no range needs masks.
//
// Schedule.  The spans are taken in groups of FOLD_T lengths L = Lb .. Lb+T-1.
// 1. Bulk: the terms of a group's cells whose two parts are both shorter than
//    Lb are ready before the group starts.  A warp takes 16 positions i, a
//    thread four of them by three ends e that start at its own first position
//    (so the tile follows the group's parallelogram: 21 of 24 ends are used), and
//    runs over m in chunks staged in shared memory for the whole CTA with
//    cp.async; near the top of the triangle, where few blocks remain, the warps
//    share a block's m range.
// 2. Spans: L = Lb + t adds the 2 t terms with a part of length Lb or more (the
//    other part is at most t long), from two shared tables: W, the group's own
//    cells by span, and SH, the cells of length <= T.  A thread takes two
//    neighbouring positions.  One barrier per span (Sec. 9.5's order: X-drop
//    needs the best of span k-1 before span k is pruned).
// 3. The group's rows go to Q, both ways round, as contiguous runs.
// One warp then walks the fold: each step loads 32 candidates of an unpaired run
// or 32 split points at once.
//
// T = 21 fills the thread tile's 24 ends (4 positions slant it by 3).  A taller
// group would waste less of the tile, but the span phase, whose terms grow with
// T and come from unregistered operands, takes a third of the time already.
#pragma once

#include "filtr_internal.h"

namespace filtr {
namespace {

constexpr int FOLD_T = 21;                       // spans per group
constexpr int FOLD_MC = 16;                      // staged split points per chunk
constexpr int FOLD_RS = FOLD_MC + 8;             // staged row stride (48 bytes: conflict free)
constexpr int16_t FOLD_NEG = -16384;             // two of them still fit 16 bits
constexpr uint32_t FOLD_NEG2 = 0xC000C000u;
static_assert(FILTR_FOLD_MAX_LEN / 2 + 1 < -FOLD_NEG, "F <= n / 2: a sum with a missing cell stays negative");

// halfwords of a row of Q
FILTR_HD int fold_row_stride(int n) { return (n + 8) & ~7; }
FILTR_HD uint64_t fold_q_bytes(int n) { return (uint64_t)(n + 1) * fold_row_stride(n) * 2; }
// 32-bit words of a row of the span tables W and SH for up to max_n bases: odd, so
// that a column of a table is conflict free, and a constant of the instance, so
// that the span loop addresses rows with immediates
FILTR_HD constexpr int fold_span_words(int max_n) { return (max_n + 6) / 2 | 1; }
FILTR_HD constexpr size_t fold_span_bytes(int max_n) {
  return ((size_t)(2 * FOLD_T + 3) * fold_span_words(max_n) * 4 + 15) / 16 * 16;
}
FILTR_HD constexpr size_t fold_stage_bytes(int nw, int stages) {
  return (size_t)stages * (32 * nw + 20) * FOLD_RS * 2;
}
FILTR_HD constexpr size_t fold_smem_bytes(int nw, int stages, int max_n, bool gs) {
  return fold_stage_bytes(nw, stages) + (gs ? 0 : fold_span_bytes(max_n)) + (max_n + 4 + 15) / 16 * 16;
}

struct FoldTiledArgs {
  const uint8_t *seq;
  const uint64_t *off;
  const uint32_t *len;
  const uint32_t *order;      // sequences of this launch
  const uint64_t *area_off;   // per sequence: first 16-byte unit of its area
  char *area;
  filtr_fold_result *out;
  int32_t *partner;           // nullptr without traceback
  int min_loop, use_xdrop, xdrop, warmup;
};

__device__ __forceinline__ void fold_cp16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// the halfword pair one halfword past word w[0]
__device__ __forceinline__ uint32_t fold_odd(const uint32_t *w) { return __byte_perm(w[0], w[1], 0x5432); }

// NW warps; ST staging buffers; MAXN: longest sequence; GS: the span tables live in the sequence's
// area instead of shared memory; MINB: blocks per SM the registers allow
template <int NW, int ST, int MAXN, bool GS, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) k_fold_tiled(const FoldTiledArgs a) {
  constexpr int T = FOLD_T, NT = NW * 32, ROWS = 32 * NW + 20;
  constexpr int W2 = fold_span_words(MAXN), WS = 2 * W2;
  extern __shared__ __align__(16) char smem[];
  __shared__ int red[2][3][NW];
  __shared__ unsigned long long redk[NW];
  const uint32_t p = a.order[blockIdx.x];
  const int n = (int)a.len[p];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int S = fold_row_stride(n);
  int16_t *stage = reinterpret_cast<int16_t *>(smem);
  char *after = smem + fold_stage_bytes(NW, ST);
  int16_t *Q = reinterpret_cast<int16_t *>(a.area + a.area_off[p] * 16);
  // W row 2 + t: span t of the group; rows 0 and 1: the two spans before it.
  // SH row L: the cells of length L <= T
  int16_t *W = GS ? reinterpret_cast<int16_t *>(reinterpret_cast<char *>(Q) + fold_q_bytes(n))
                  : reinterpret_cast<int16_t *>(after);
  int16_t *SH = W + (T + 2) * WS;
  uint32_t *W32 = reinterpret_cast<uint32_t *>(W), *SH32 = reinterpret_cast<uint32_t *>(SH);
  uint8_t *sx = reinterpret_cast<uint8_t *>(GS ? after : after + fold_span_bytes(MAXN));

  const uint8_t *g = a.seq + a.off[p];
  for (int t = tid; t < n + 4; t += NT) sx[t] = t < n ? g[t] : 0;
  {
    uint4 *q4 = reinterpret_cast<uint4 *>(Q);
    const int total = (n + 1) * (S / 8);
    const uint4 neg = make_uint4(FOLD_NEG2, FOLD_NEG2, FOLD_NEG2, FOLD_NEG2);
    for (int t = tid; t < total; t += NT) q4[t] = neg;
    uint32_t *w2 = reinterpret_cast<uint32_t *>(W);
    for (int t = tid; t < (2 * T + 3) * W2; t += NT) w2[t] = FOLD_NEG2;
  }
  if (a.partner)
    for (int t = tid; t < n; t += NT) a.partner[a.off[p] + t] = -1;
  __syncthreads();
  for (int t = tid; t <= n; t += NT) {  // empty intervals and single bases: 0
    Q[(size_t)t * S + t] = 0;
    W[t] = 0;
    if (t < n) {
      Q[(size_t)t * S + t + 1] = 0;
      Q[(size_t)(t + 1) * S + t] = 0;
      W[WS + t] = 0;
      SH[WS + t] = 0;
    }
  }
  __syncthreads();

  const int li = lane >> 3, lj = lane & 7;
  const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(stage);
  const bool xd = a.use_xdrop != 0;
  int lo = 0, hi = n - 1, best = 0, last_k = 0;
  int bf = 0, bk = 0, bi = 0;  // this thread's best unpruned cell: largest F, longest span, smallest i
  uint64_t cells = (uint64_t)n;
  bool ended = n < 2;
  for (int Lb = 2; Lb <= n && !ended; Lb += T) {
    // ---- bulk ---------------------------------------------------------------
    const int blk0 = max(lo - T, 0) >> 4, blk1 = min(hi, n - Lb) >> 4;
    for (int b0 = blk0; b0 <= blk1; b0 += NW) {
      const int nb = min(NW, blk1 - b0 + 1);
      int sp = 1;  // warps sharing a block's m range
      while (sp < 4 && 2 * sp * nb <= NW) sp *= 2;
      const int blk = wid % nb, part = wid / nb;
      const bool on = part < sp;
      const int r0 = b0 * 16;               // first row of A; B's first row is r0 + Lb
      const int ra = 16 * nb, rb = ra + 20; // staged rows of each
      const int m_end = min(r0 + ra + Lb, S);
      const int w_lo = r0 + 16 * blk, w_hi = w_lo + 15 + Lb;  // this warp's split points [w_lo, w_hi)
      uint32_t acc[4][3];
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int x = 0; x < 3; ++x) acc[y][x] = FOLD_NEG2;
      auto fetch = [&](int m0, int buf) {
        for (int t = tid; t < (ra + rb) * 2; t += NT) {
          const int row = t >> 1, half = (t & 1) * 8;
          const int src = min(row < ra ? r0 + row : r0 + Lb + row - ra, n);
          if (m0 < m_end && m0 + half < S)
            fold_cp16(stage_s + (uint32_t)((buf * ROWS + row) * FOLD_RS + half) * 2,
                      Q + (size_t)src * S + m0 + half);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
#pragma unroll
      for (int b = 0; b < ST - 1; ++b) fetch(r0 + b * FOLD_MC, b);
      int buf = 0;
      for (int m0 = r0; m0 < m_end; m0 += FOLD_MC, buf = buf == ST - 1 ? 0 : buf + 1) {
        asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
        __syncthreads();  // the chunk is here, and the last chunk's readers are done
        fetch(m0 + (ST - 1) * FOLD_MC, buf == 0 ? ST - 1 : buf - 1);
        const int16_t *A = stage + (buf * ROWS + 16 * blk + 4 * li) * FOLD_RS;
        const int16_t *B = stage + (buf * ROWS + ra + 16 * blk + 4 * li + lj) * FOLD_RS;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int m = m0 + 8 * h;
          if (on && m < m_end && m + 8 > w_lo && m < w_hi && ((m >> 3) & (sp - 1)) == part) {
            uint4 av[4];
#pragma unroll
            for (int y = 0; y < 4; ++y)
              av[y] = *reinterpret_cast<const uint4 *>(A + y * FOLD_RS + 8 * h);
#pragma unroll
            for (int x = 0; x < 3; ++x) {
              const uint4 bv = *reinterpret_cast<const uint4 *>(B + 8 * x * FOLD_RS + 8 * h);
#pragma unroll
              for (int y = 0; y < 4; ++y) {
                acc[y][x] = __viaddmax_s16x2(av[y].x, bv.x, acc[y][x]);
                acc[y][x] = __viaddmax_s16x2(av[y].y, bv.y, acc[y][x]);
                acc[y][x] = __viaddmax_s16x2(av[y].z, bv.z, acc[y][x]);
                acc[y][x] = __viaddmax_s16x2(av[y].w, bv.w, acc[y][x]);
              }
            }
          }
        }
      }
      __syncthreads();  // the staging is reused below and by the next round
      if (sp > 1) {  // fold the parts of each block into part 0
        uint32_t *ex = reinterpret_cast<uint32_t *>(stage);  // (sp - 1) nb < NW blocks of 12 x 32 words
        if (on && part > 0) {
          uint32_t *d = ex + ((part - 1) * nb + blk) * 12 * 32 + lane;
#pragma unroll
          for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int x = 0; x < 3; ++x) d[(y * 3 + x) * 32] = acc[y][x];
        }
        __syncthreads();
        if (part == 0)
          for (int q = 0; q < sp - 1; ++q) {
            const uint32_t *d = ex + (q * nb + blk) * 12 * 32 + lane;
#pragma unroll
            for (int y = 0; y < 4; ++y)
#pragma unroll
              for (int x = 0; x < 3; ++x) acc[y][x] = __vmaxs2(acc[y][x], d[(y * 3 + x) * 32]);
          }
        __syncthreads();
      }
      if (part == 0) {
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            const int t = lj + 8 * x - y, i = r0 + 16 * blk + 4 * li + y;
            if (t >= 0 && t < T && i <= n - Lb - t)
              W[(2 + t) * WS + i] = (int16_t)max((int)(int16_t)(acc[y][x] & 0xffffu), (int)acc[y][x] >> 16);
          }
      }
    }
    __syncthreads();
    // ---- spans ---------------------------------------------------------------
    int t = 0;
    for (; t < T && Lb + t <= n; ++t) {
      const int L = Lb + t, k = L - 1;
      const int dl = max(lo - 1, 0), dh = min(hi, n - L);
      if (dl > dh) {
        ended = true;
        break;
      }
      const int thr = (xd && k > a.warmup) ? max(best - a.xdrop, 0) : 0;
      const bool loop_ok = k - 1 >= a.min_loop;
      int tmax = -1, tlo = INT_MAX, thi = -1;
      for (int i = 2 * tid; i <= n - L; i += 2 * NT) {
        uint32_t f2 = FOLD_NEG2;
        if (i + 1 >= dl && i <= dh) {
          // (i, i+x) + (i+x, e) and (i, e-x) + (e-x, e), two x at a time; x = t + 1, reached
          // when t is odd, is a split of the bulk again (W row 1, the span before the group)
          const uint32_t *wt = W32 + (1 + t) * W2 + (i >> 1);  // W of span t - 1 at i
          f2 = wt[W2];
          const uint32_t *wd = wt;                             // ... at i + x - 1
          const uint32_t *sl = SH32 + W2 + (i >> 1);           // SH row 1 at i
          const uint32_t *sr = SH32 + W2 + ((i + L - 1) >> 1); // SH row 1 at e - 1
          if (L & 1) {
#pragma unroll 4
            for (int x = 1; x <= t; x += 2) {
              f2 = __viaddmax_s16x2(sl[0], fold_odd(wd), f2);
              f2 = __viaddmax_s16x2(wt[0], sr[0], f2);
              f2 = __viaddmax_s16x2(sl[W2], wd[1 - W2], f2);
              f2 = __viaddmax_s16x2(wt[-W2], fold_odd(sr + W2 - 1), f2);
              wt -= 2 * W2;
              wd -= 2 * W2 - 1;
              sl += 2 * W2;
              sr += 2 * W2 - 1;
            }
          } else {
#pragma unroll 4
            for (int x = 1; x <= t; x += 2) {
              f2 = __viaddmax_s16x2(sl[0], fold_odd(wd), f2);
              f2 = __viaddmax_s16x2(wt[0], fold_odd(sr), f2);
              f2 = __viaddmax_s16x2(sl[W2], wd[1 - W2], f2);
              f2 = __viaddmax_s16x2(wt[-W2], sr[W2], f2);
              wt -= 2 * W2;
              wd -= 2 * W2 - 1;
              sl += 2 * W2;
              sr += 2 * W2 - 1;
            }
          }
          if (loop_ok) {
            const uint32_t in = __vadd2(fold_odd(W32 + t * W2 + (i >> 1)), 0x00010001u);  // G(i+1, e-1) + 1
            const int a0 = sx[i], a1 = sx[i + 1], c0 = sx[i + L - 1], c1 = sx[i + L];
            uint32_t m = rna_pair(a0, c0) ? 0xffffu : 0u;
            m |= rna_pair(a1, c1) ? 0xffff0000u : 0u;
            f2 = __vmaxs2(f2, (in & m) | (FOLD_NEG2 & ~m));
          }
        }
        int v0 = (int)(int16_t)(f2 & 0xffffu), v1 = (int)f2 >> 16;
        const bool in0 = i >= dl && i <= dh && v0 >= thr, in1 = i + 1 >= dl && i + 1 <= dh && v1 >= thr;
        if (!in0) v0 = FOLD_NEG;
        if (!in1) v1 = FOLD_NEG;
        f2 = ((uint32_t)v0 & 0xffffu) | ((uint32_t)v1 << 16);
        W32[(2 + t) * W2 + (i >> 1)] = f2;
        if (L <= T) SH32[L * W2 + (i >> 1)] = f2;
        if (xd) {
          if (in0) {
            tmax = max(tmax, v0);
            tlo = min(tlo, i);
            thi = i;
            if (v0 > bf || (v0 == bf && k > bk)) bf = v0, bk = k, bi = i;
          }
          if (in1) {
            tmax = max(tmax, v1);
            tlo = min(tlo, i + 1);
            thi = i + 1;
            if (v1 > bf || (v1 == bf && k > bk)) bf = v1, bk = k, bi = i + 1;
          }
        }
      }
      cells += (uint64_t)(dh - dl + 1);
      last_k = k;
      if (!xd) {  // every cell stays
        __syncthreads();
        hi = n - 1 - k;
        continue;
      }
      int(&rd)[3][NW] = red[t & 1];
      tmax = __reduce_max_sync(0xffffffffu, tmax);
      tlo = __reduce_min_sync(0xffffffffu, tlo);
      thi = __reduce_max_sync(0xffffffffu, thi);
      if (lane == 0) {
        rd[0][wid] = tmax;
        rd[1][wid] = tlo;
        rd[2][wid] = thi;
      }
      __syncthreads();  // also publishes the span to the whole CTA
      int gmax = -1, glo = INT_MAX, ghi = -1;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        gmax = max(gmax, rd[0][w]);
        glo = min(glo, rd[1][w]);
        ghi = max(ghi, rd[2][w]);
      }
      if (gmax < 0) {  // nothing unpruned on this span
        ended = true;
        ++t;
        break;
      }
      best = gmax;
      lo = glo;
      hi = ghi;
    }
    // ---- the group's cells into Q, both ways round --------------------------------
    // (row r: G(r, r + Lb + x) forwards, G(r - Lb - x, r) backwards)
    for (int y = tid; y < (n + 1) * T; y += NT) {
      const int r = y / T, x = y - r * T;
      if (x < t && r + Lb + x <= n) Q[(size_t)r * S + r + Lb + x] = W[(2 + x) * WS + r];
      if (x < t && r - Lb - x >= 0) Q[(size_t)r * S + r - Lb - x] = W[(2 + x) * WS + r - Lb - x];
    }
    __syncthreads();
    if (!ended && Lb + T <= n) {
      for (int i = tid; i <= n; i += NT) {
        W[i] = W[T * WS + i];
        W[WS + i] = W[(T + 1) * WS + i];
      }
      __syncthreads();
    }
  }

  // the end cell: (0, n-1) if it stayed, else the best unpruned cell
  int ei = 0, ej = n - 1, status = FILTR_ST_OK, score = 0;
  if (n > 0) {
    score = (n - 1 <= last_k) ? (int)Q[n] : -1;
    if (score < 0) {
      unsigned long long key = ((unsigned long long)(bf + 1) << 40) | ((unsigned long long)bk << 20) |
                               (unsigned long long)(0xfffff - bi);
      for (int o = 16; o; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
      if (lane == 0) redk[wid] = key;
      __syncthreads();
      key = 0;
      for (int w = 0; w < NW; ++w) key = max(key, redk[w]);
      score = (int)(key >> 40) - 1;
      ei = 0xfffff - (int)(key & 0xfffff);
      ej = ei + (int)((key >> 20) & 0xfffff);
      status = FILTR_ST_DROPPED;
    }
  }
  if (tid == 0) {
    filtr_fold_result r;
    r.score = score;
    r.i_end = ei;
    r.j_end = n > 0 ? ej : 0;
    r.status = status;
    r.cells = cells;
    a.out[p] = r;
  }
  if (!a.partner || n < 2 || wid != 0) return;

  // ---- the fold below the end cell (one warp) -----------------------------------
  // W is free now; a deferred part is two halfwords, at most n of them wait
  int16_t *stack = GS ? W : reinterpret_cast<int16_t *>(after);
  int32_t *pt = a.partner + a.off[p];
  int top = 0, i = ei, e = ej + 1, f = score;
  for (;;) {
    if (e - i < 2) {  // one base or none: the next deferred part
      if (top == 0) break;
      __syncwarp();
      e = stack[--top];
      i = stack[--top];
      f = Q[(size_t)i * S + e];
      __syncwarp();
      continue;
    }
    // lane d: i unpaired d + 1 times, j unpaired d + 1 times with i paired until then
    const int16_t *ri = Q + (size_t)i * S, *re = Q + (size_t)e * S, *rn = ri + S;
    const bool in_i = i + 1 + lane < e, in_j = e - 1 - lane > i;
    const int vi = in_i ? (int)re[i + 1 + lane] : INT_MIN;
    const int vj = in_j ? (int)ri[e - 1 - lane] : INT_MIN;
    const int vn = (lane > 0 && in_j) ? (int)rn[e - lane] : INT_MIN;  // G(i+1, e-lane)
    const int vp = (int)rn[e - 1];                                      // G(i+1, e-1)
    const unsigned mi = __ballot_sync(0xffffffffu, vi == f);
    if (mi & 1u) {
      i += mi == 0xffffffffu ? 32 : __ffs(~mi) - 1;
      continue;
    }
    const unsigned mj = __ballot_sync(0xffffffffu, vj == f && vn != f);
    if (mj & 1u) {
      e -= mj == 0xffffffffu ? 32 : __ffs(~mj) - 1;
      continue;
    }
    if (rna_pair(sx[i], sx[e - 1]) && e - i - 2 >= a.min_loop && vp + 1 == f) {
      if (lane == 0) {
        pt[i] = e - 1;
        pt[e - 1] = i;
      }
      ++i;
      --e;
      --f;
      continue;
    }
    int m = -1, fr = 0;
    for (int m0 = i + 1; m0 < e && m < 0; m0 += 32) {
      const int mm = m0 + lane;
      const int x = mm < e ? (int)ri[mm] : FOLD_NEG, y = mm < e ? (int)re[mm] : FOLD_NEG;
      const unsigned hit = __ballot_sync(0xffffffffu, x >= 0 && y >= 0 && x + y == f);
      if (hit) {
        const int d = __ffs(hit) - 1;
        m = m0 + d;
        fr = __shfl_sync(0xffffffffu, y, d);
      }
    }
    if (m < 0) break;  // no term gives G(i, e): not expected
    __syncwarp();
    if (lane == 0) {
      stack[top] = (int16_t)i;
      stack[top + 1] = (int16_t)m;
    }
    top += 2;
    __syncwarp();
    i = m;
    f = fr;
  }
}

}  // namespace
}  // namespace filtr
