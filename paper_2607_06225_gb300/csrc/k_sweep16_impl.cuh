// k_sweep16_impl.cuh -- the antidiagonal X-drop / Z-drop sweep (Sec. 5.2 / 7.2,
// Sec. 9.3) with two cells in each 32-bit register (int16x2), for affine Gotoh
// H/E/F alignments.  Instantiated by k_xdrop16.cu (X-drop) and k_zdrop16.cu
// (Z-drop).  The int32 sweep (k_xdrop_impl.cuh) computes the same cells; this
// one trades its per-cell bookkeeping for packed DPX arithmetic.
//
// Values.  Under X-drop every value that can still reach an unpruned cell lies
// within about X of the previous antidiagonal's best, so a group holds values
// relative to a base score b: a real value v is the signed 16-bit v - b + C0.
// When the best drifts more than X16_REBASE from C0 the group moves b (every
// state register shifted by one DPX add with a floor at zero).  Packed 0 is
// minus infinity: every add that can fall below zero has a floor at zero or is
// followed by a maximum with a value that has, so a pruned or missing neighbour
// stays at 0, and values formed from it (at most the largest substitution score)
// stay far below every threshold.  The host sends a pair here only when its
// threshold leaves room (X < X16_MAX_DROP); a pair whose best nevertheless
// leaves the range, or whose lowest threshold falls to the floor, stops with
// status X16_OVERFLOW and is rerun by the int32 sweep.
//
// Window.  Thread t owns slots 8t .. 8t+7 (16 with G = 2: two groups of eight).
// The window is fixed to diagonals: slot p of antidiagonal k is the cell (k - c_k
// - p, c_k + p), and c_k moves by one on every other antidiagonal (phase A:
// delta = 1; phase B: delta = 0).  So the two phases are straight-line code with
// every dependency at a fixed slot offset: the diagonal neighbour always sits
// in the same slot two antidiagonals ago; in phase A the left neighbour sits in
// the same slot and the upper one a slot above, in phase B the left one a slot
// below and the upper one in the same slot.  When the live range comes near the
// window's edge, the group moves the window by whole threads (a rare shuffle of
// the state) to centre it.  Register r of each state array holds slot r in its
// low half and slot r + 4 in its high half, so only registers 0 and 3 take a byte
// permute with the edge value of the neighbouring thread.  Traceback nibbles and
// window origins are laid out as the int32 sweep's, so every walk reads both
// kernels' output alike.
//
// State.  Beside H of k - 1 and k - 2 a cell keeps what its neighbours will
// need: Ho = H - (o + e), En = max(E - e, Ho) and Fn = max(F - e, Ho), formed once
// when the cell is final; a neighbour's E is then just a view of En, and "took
// the extension" is En > Ho.  Pruning needs two masked operations per register
// (H, and the constant -e replaced by the lowest value), since Ho and the maxima
// follow from them.
//
// Scores.  DNA with one match and one mismatch score: the residues of a thread's
// slots are nibbles of one word per side (slot s at nibble s, so that slots r and
// r + 4 are 16 bits apart), moved by one funnel shift on every other
// antidiagonal, compared by one XOR and one add, and refilled 8 residues at a
// time.  Other scorings look each pair up in a shared table.
//
// Blocks.  The sweep runs in blocks of 16 antidiagonals.  A block whose live
// range cannot reach a matrix edge, the band or the window's edge within 16
// antidiagonals, and whose values cannot leave the 16-bit range, runs without any
// of those checks; the others run the same code with them (SLOW).
//
// Schedule.  Pruning antidiagonal k needs best(k-1) and the live range of k - 1;
// the raw update of k needs neither, so the reductions of k - 1 are in flight
// while the raw cells of k are computed.  The candidate range [lo(k-1) - 1,
// hi(k-1) + 1] needs no mask as long as it holds every diagonal alive on k - 2:
// a cell outside it has two dead neighbours on k - 1, so only its diagonal could
// keep it alive.  Only a range that moved inwards past one of those diagonals
// (or a local alignment, whose floor keeps any cell alive) masks its cells.
//
// Measured against the sweep with a sliding origin (one delta per antidiagonal,
// four code paths, and every bound, range and code handled per antidiagonal: 362
// warp instructions each): see the figures at x16_launch.
#include <algorithm>
#include <climits>

#pragma once

#include "filtr_internal.h"
#include "k_xdrop_layout.h"

namespace filtr {
namespace {

constexpr unsigned X16_FULL = 0xffffffffu;
constexpr int X16_C0 = 16384;
constexpr int X16_BLOCK = 16;  // antidiagonals per block (8 of each phase)
constexpr uint32_t X16_K80 = 0x80008000u;

template <int W>
struct alignas(16) X16Shared {
  int4 red[2][W];       // per warp: max H (packed), lowest live slot, highest live slot, slot of the max
  // a warp's edge values, [0] its first thread's (Fn, Ho), which the warp before
  // reads in phase A, [1] its last thread's (En, Ho), which the warp after reads in phase B
  uint2 edge[2][W][2];
  int tmp[2][W];
  uint32_t pair;
  uint4 move[W > 1 ? W * 32 : 1];  // state on its way to other threads
};

// 0xffff in each half whose bit 15 (low) / bit 31 (high) is set, else 0
__device__ __forceinline__ uint32_t x16_halfmask(uint32_t x) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(r) : "r"(x));
  return r;
}
// per half [a > b] in bit 15 / 31, for halves in [0, 0x7fff]
__device__ __forceinline__ uint32_t x16_gt(uint32_t a, uint32_t b) { return a + 0x7fff7fffu - b; }
// register view of the slots one below: slot r - 1 (low) and r + 3 (high); for
// register 0 the low half is the previous thread's slot 7 (high half of pv)
__device__ __forceinline__ uint32_t x16_down0(uint32_t x3, uint32_t pv) { return __byte_perm(x3, pv, 0x1076); }
// register view of the slots one above for register 3: slot 4 (high half of
// x0) and the next thread's slot 0 (low half of nx)
__device__ __forceinline__ uint32_t x16_up3(uint32_t x0, uint32_t nx) { return __byte_perm(x0, nx, 0x5432); }
__device__ __forceinline__ uint32_t x16_splat(int v) { return ((uint32_t)v & 0xffffu) * 0x10001u; }

// register view of the slots one below for register (g, 0) of a thread with G
// groups: the low half is slot 8g - 1 (the high half of group g - 1's register
// 3, or of the previous thread's last register, pv), the high half slot 8g + 3
template <int G>
__device__ __forceinline__ uint32_t x16_down_g(const uint32_t (&X)[4 * G], int g, uint32_t pv) {
  return x16_down0(X[4 * g + 3], g ? +X[g ? 4 * g - 1 : 0] : +pv);
}
// register view of the slots one above for register (g, 3): slot 8g + 4 (high
// half of register (g, 0)) and slot 8g + 8 (low half of group g + 1's register
// 0, or of the next thread's first register, nx)
template <int G>
__device__ __forceinline__ uint32_t x16_up_g(const uint32_t (&X)[4 * G], int g, uint32_t nx) {
  return x16_up3(X[4 * g], g < G - 1 ? +X[g < G - 1 ? 4 * g + 4 : 0] : +nx);
}

// eight residue codes (each below 4) s[at .. at + 7] as the nibbles of a word,
// first in the lowest; positions outside [0, len) read as anything
__device__ __forceinline__ uint32_t x16_nibbles(const uint8_t *s, int at, int len) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(s) + (intptr_t)at;
  const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~(uintptr_t)3);
  const int off = at - (int)(a & 3);  // position of w[0]'s first byte
  // only words that hold a residue of the sequence are read
  const uint32_t w0 = (off + 3 >= 0 && off < len) ? __ldg(w) : 0u;
  const uint32_t w1 = (off + 7 >= 0 && off + 4 < len) ? __ldg(w + 1) : 0u;
  const uint32_t w2 = (off + 11 >= 0 && off + 8 < len) ? __ldg(w + 2) : 0u;
  const int sh = (int)(a & 3) * 8;
  const uint32_t x = __funnelshift_r(w0, w1, sh), y = __funnelshift_r(w1, w2, sh);
  return __byte_perm((x & 0x03030303u) | (x >> 4 & 0x30303030u), (y & 0x03030303u) | (y >> 4 & 0x30303030u),
                     0x6420);
}
// the eight nibbles in reverse order
__device__ __forceinline__ uint32_t x16_reverse(uint32_t x) {
  x = __byte_perm(x, 0, 0x0123);
  return (x & 0x0f0f0f0fu) << 4 | (x >> 4 & 0x0f0f0f0fu);
}

// runtime knobs of the packed sweep (a test hook can switch rebasing off, so
// that long pairs leave the 16-bit range and take the int32 rerun)
struct X16Knobs {
  int rebase;  // distance of the best from C0 that moves the base; <= 0: never
};

enum : int { X16_GO = 0, X16_END, X16_WIDE, X16_OVF };  // how a step ended

// UNI: DNA with one match and one mismatch score (codes compared), else a score table
// G: groups of four registers (eight slots) per thread -- 1, or 2 for a one-warp
// group holding a 512-slot window (W = 1 only)
template <int W, int G, bool LOCAL, bool TB, bool ZD, bool UNI>
struct Sweep16 {
  static constexpr int S = 8 * G, P = 4 * G, WIN = W * 32 * S, ROW = WIN / 8;
  // a fast step needs k and c itself (else a fast block counts them as a whole)
  static constexpr bool STEP_K = LOCAL || ZD || W > 1 || !UNI;
  // the widest group's window moves by single slots: no wider one takes its pairs over
  static constexpr bool ANY_SLOT = W == XD_MAX_WARPS;
  // parameters of the pair and the thread
  X16Shared<W> &sh;
  const int8_t *s_sub;
  const uint8_t *q, *rs;
  int M, N, A, lane, warp, tid, base_slot;
  int oe, X, smax, pceil, pfloor, band_lo, band_hi;
  bool xrun, track, need_bs;
  uint32_t MA2, MI2, NOE2, NE2, CX2;
  uint32_t *tbp;     // this thread's words of the next row
  // state
  uint32_t Ha[P], Hb[P], En[P], Fn[P], Ho[P];
  uint32_t qw[UNI ? G : P], rw[UNI ? G : P];  // residue codes of the window
  uint32_t qn, rn;                            // UNI: codes to come; else the next code
  int base, c;         // real value of packed C0; origin of the last antidiagonal
  uint32_t Z2;         // local: packed zero
  uint32_t b2;         // best of the last antidiagonal in both halves, 0: nothing alive
  uint32_t brun2;      // running best (X-drop running)
  int pl, ph, pbs;     // its lowest and highest live slot, slot of its best cell
  int ol, oh;          // live slots of the antidiagonal before
  int dbest;           // Z-drop: reference diagonal
  int bv, bi, bj;      // best cell so far
  int k;               // the last antidiagonal
  uint64_t cells;
  int span;            // sum of ph - pl over the steps of a fast block
  int cornerH;
  bool corner;

  __device__ __forceinline__ Sweep16(X16Shared<W> &s) : sh(s) {}

  // pruned H, and what the cell's neighbours need of it
  __device__ __forceinline__ void finish_cell(uint32_t &H, int r, uint32_t hm, uint32_t m, uint32_t E, uint32_t F) {
    H = hm;
    Ho[r] = __viaddmax_s16x2_relu(hm, NOE2, 0u);
    const uint32_t ne = (NE2 & m) | (X16_K80 & ~m);  // -e, or lower than any value
    En[r] = __viaddmax_s16x2(E, ne, Ho[r]);
    Fn[r] = __viaddmax_s16x2(F, ne, Ho[r]);
  }

  // (low half) bit 4g + rq.., the slots' bits of eight-slot group words: slot s at bit s
  static __device__ __forceinline__ uint32_t bits8(uint32_t w) { return (w & 0xfu) | (w >> 12 & 0xf0u); }

  // residue codes of the window of antidiagonal kk with origin cc, and those to
  // come when the next antidiagonal is of phase A
  __device__ __forceinline__ void load_codes(int kk, int cc) {
    const int i0 = kk - cc - base_slot;  // row of slot 0
    const int j0 = cc + base_slot;       // column of slot 0
    if constexpr (UNI) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        qw[g] = x16_reverse(x16_nibbles(q, i0 - 8 * g - 8, M));
        rw[g] = x16_nibbles(rs, j0 + 8 * g - 1, N);
      }
    } else {
#pragma unroll
      for (int r = 0; r < P; ++r) {
        uint32_t qv = 0, rv = 0;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int pp = 8 * (r >> 2) + (r & 3) + 4 * hh;
          const int j = j0 + pp, i = i0 - pp;
          qv |= (i >= 1 && i <= M ? (uint32_t)q[i - 1] : 0u) << (16 * hh);
          rv |= (j >= 1 && j <= N ? (uint32_t)rs[j - 1] : 0u) << (16 * hh);
        }
        qw[r] = qv;
        rw[r] = rv;
      }
    }
  }
  // the codes entering in the next block (UNI), the last antidiagonal k, origin c
  __device__ __forceinline__ void load_next(uint32_t &qx, uint32_t &rx, int ahead) const {
    if constexpr (UNI) {
      // phase A steps bring r[c' + base + S - 1 ..] in, phase B steps q[k - c - base ..]
      rx = x16_nibbles(rs, c + base_slot + S - 1 + ahead, N);
      qx = x16_reverse(x16_nibbles(q, k - c - base_slot + ahead, M));
    }
  }

  // the last antidiagonal's reductions over the group's warps
  __device__ __forceinline__ void combine() {
    const int nb = k & 1;
    if constexpr (W > 1 && W <= 4) {  // a few warps: one broadcast load each, no warp reductions
      int4 v[W];
#pragma unroll
      for (int x = 0; x < W; ++x) v[x] = sh.red[nb][x];
      int best = v[0].x, l = v[0].y, h = v[0].z;
#pragma unroll
      for (int x = 1; x < W; ++x) {
        best = max(best, v[x].x);
        l = min(l, v[x].y);
        h = max(h, v[x].z);
      }
      b2 = (uint32_t)best;
      pl = l;
      ph = h;
      if (need_bs) {
        int s = -1;
#pragma unroll
        for (int x = 0; x < W; ++x)
          if (v[x].x == best) s = max(s, v[x].w);
        pbs = s;
      }
    } else if constexpr (W > 4) {
      const int4 v = lane < W ? sh.red[nb][lane] : make_int4(0, INT_MAX, INT_MIN, -1);
      b2 = (uint32_t)__reduce_max_sync(X16_FULL, v.x);
      pl = __reduce_min_sync(X16_FULL, v.y);
      ph = __reduce_max_sync(X16_FULL, v.z);
      if (need_bs) pbs = __reduce_max_sync(X16_FULL, (uint32_t)v.x == b2 ? v.w : -1);
    }
  }
  // this warp's reductions and edge values of antidiagonal k, for the others
  __device__ __forceinline__ void publish() {
    const int nb = k & 1;
    if (lane == 0) sh.red[nb][warp] = make_int4((int)b2, pl, ph, pbs);
    if (lane == 0 || lane == 31)
      sh.edge[nb][warp][lane & 1] = make_uint2(lane ? En[P - 1] : Fn[0], lane ? Ho[P - 1] : Ho[0]);
    __syncthreads();
  }
  // the group's largest slot whose H equals the best (smallest row)
  __device__ __forceinline__ int best_slot_of(const uint32_t (&H)[P], uint32_t best2) const {
    uint32_t bm = 0;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      uint32_t w = 0;
#pragma unroll
      for (int rq = 0; rq < 4; ++rq)
        w |= x16_halfmask(H[4 * g + rq] + X16_K80 - best2) & (0x10001u << rq);
      bm |= bits8(w) << (8 * g);
    }
    return __reduce_max_sync(X16_FULL, bm ? base_slot + 31 - __clz(bm) : -1);
  }
  // what the antidiagonal k (origin c, live range pl .. ph, H in Hk) means for
  // the best cell, Z-drop's diagonal and the corner
  __device__ __forceinline__ void settle(const uint32_t (&Hk)[P]) {
    if constexpr (LOCAL || ZD) {
      const int gv = (int)(b2 & 0xffffu) - X16_C0 + base;
      if (LOCAL && !ZD && W == 1) {
        if (!track || gv < bv) return;
        pbs = best_slot_of(Hk, b2);
      }
      const int jj = c + pbs, ii = k - jj;
      if (track && (gv > bv || (gv == bv && (ii < bi || (ii == bi && jj < bj))))) {
        bv = gv;
        bi = ii;
        bj = jj;
      }
      if (ZD && (!xrun || b2 > brun2)) dbest = 2 * jj - k;
    }
  }

  // antidiagonal k + 1 in phase PH (0: A, 1: B); Hp: H of k, Hc: H of k - 1 in,
  // of k + 1 out
  template <int PH, bool SLOW>
  __device__ __forceinline__ int step(uint32_t (&Hc)[P], const uint32_t (&Hp)[P]) {
    // ---- codes at the new antidiagonal ------------------------------------------
    uint32_t s2[P];
    if constexpr (UNI) {
      if (PH == 0) {  // reference codes move down one slot
#pragma unroll
        for (int g = 0; g < G; ++g) rw[g] = __funnelshift_r(rw[g], g < G - 1 ? +rw[g < G - 1 ? g + 1 : 0] : +rn, 4);
        rn >>= 4;
      } else {  // query codes move up one slot
#pragma unroll
        for (int g = G - 1; g >= 0; --g) qw[g] = __funnelshift_l(g ? +qw[g ? g - 1 : 0] : +qn, qw[g], 4);
        qn <<= 4;
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        // bit 3 of a nibble: codes differ.  An odd slot's is a byte's sign, so one byte
        // permute spreads a register's two flags; a shift brings the even slots' there
        const uint32_t t1 = (qw[g] ^ rw[g]) + 0x77777777u, t0 = t1 << 4;
        uint32_t n0, n1, n2, n3;
        asm("prmt.b32 %0, %1, 0, 0xaa88;" : "=r"(n0) : "r"(t0));
        asm("prmt.b32 %0, %1, 0, 0xaa88;" : "=r"(n1) : "r"(t1));
        asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(n2) : "r"(t0));
        asm("prmt.b32 %0, %1, 0, 0xbb99;" : "=r"(n3) : "r"(t1));
        s2[4 * g] = (n0 & MI2) | (~n0 & MA2);
        s2[4 * g + 1] = (n1 & MI2) | (~n1 & MA2);
        s2[4 * g + 2] = (n2 & MI2) | (~n2 & MA2);
        s2[4 * g + 3] = (n3 & MI2) | (~n3 & MA2);
      }
    } else {
      if (PH == 0) {
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const uint32_t in = g < G - 1 ? (rw[g < G - 1 ? 4 * g + 4 : 0] & 0xffffu) : rn;
          const uint32_t t = (rw[4 * g] >> 16) | (in << 16);
          rw[4 * g] = rw[4 * g + 1];
          rw[4 * g + 1] = rw[4 * g + 2];
          rw[4 * g + 2] = rw[4 * g + 3];
          rw[4 * g + 3] = t;
        }
        // the query code that enters on k + 2 (phase B)
        const int i = k + 1 - c - base_slot;
        qn = (i >= 1 && i <= M) ? q[i - 1] : 0u;
      } else {
#pragma unroll
        for (int g = G - 1; g >= 0; --g) {
          const uint32_t in = g ? (qw[g ? 4 * g - 1 : 0] >> 16) : qn;
          const uint32_t t = in | (qw[4 * g + 3] << 16);
          qw[4 * g + 3] = qw[4 * g + 2];
          qw[4 * g + 2] = qw[4 * g + 1];
          qw[4 * g + 1] = qw[4 * g];
          qw[4 * g] = t;
        }
        // the reference code that enters on k + 2 (phase A)
        const int j = c + 1 + base_slot + S - 1;
        rn = (j >= 1 && j <= N) ? rs[j - 1] : 0u;
      }
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const uint32_t idx = qw[r] * (uint32_t)A + rw[r];
        const int slo = s_sub[idx & 0xffffu], shi = s_sub[idx >> 16];
        s2[r] = ((uint32_t)slo & 0xffffu) | ((uint32_t)shi << 16);
      }
    }
    // a warp far from the live range (taken from one antidiagonal earlier) has
    // only dead cells
    const bool idle = W > 1 && (base_slot - lane * S > oh + 3 || base_slot - lane * S + 32 * S - 1 < ol - 3) &&
                      ol <= oh;
    // ---- neighbour values across thread boundaries, raw cells of k + 1 -----------
    uint32_t Hr[P], Er[P], Fr[P];
    if (!idle) {
      uint32_t nx = 0, no = 0;
      const int buf = k & 1;
      if (PH == 0) {
        nx = __shfl_down_sync(X16_FULL, Fn[0], 1);
        no = __shfl_down_sync(X16_FULL, Ho[0], 1);
        if ((SLOW || W > 1) && lane == 31) {  // (in a fast block the last thread of one warp is dead)
          const uint2 v = W > 1 && warp < W - 1 ? sh.edge[buf][warp + 1][0] : make_uint2(0u, 0u);
          nx = v.x;
          no = v.y;
        }
      } else {
        nx = __shfl_up_sync(X16_FULL, En[P - 1], 1);
        no = __shfl_up_sync(X16_FULL, Ho[P - 1], 1);
        if ((SLOW || W > 1) && lane == 0) {
          const uint2 v = W > 1 && warp > 0 ? sh.edge[buf][warp - 1][1] : make_uint2(0u, 0u);
          nx = v.x;
          no = v.y;
        }
      }
      uint32_t nib[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        uint32_t acc = 0;
        uint32_t fl[4][4];  // traceback flags: F extended, E extended, F > max(D, E), E > D
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
          // registers in the order 0, 2, 1, 3: the flags of r and r + 2 pack together
          const int rq = (rr & 1) * 2 + (rr >> 1), r = 4 * g + rq;
          uint32_t E, Eo, F, Fo;
          if (PH == 0) {
            E = En[r];
            Eo = Ho[r];
            F = rq < 3 ? Fn[rq < 3 ? r + 1 : 0] : x16_up_g<G>(Fn, g, nx);
            Fo = rq < 3 ? Ho[rq < 3 ? r + 1 : 0] : x16_up_g<G>(Ho, g, no);
          } else {
            E = rq ? En[rq ? r - 1 : 0] : x16_down_g<G>(En, g, nx);
            Eo = rq ? Ho[rq ? r - 1 : 0] : x16_down_g<G>(Ho, g, no);
            F = Fn[r];
            Fo = Ho[r];
          }
          const uint32_t D = __viaddmax_s16x2_relu(Hc[r], s2[r], 0u);
          const uint32_t DE = __vimax_s16x2_relu(D, E);
          Hr[r] = LOCAL ? __vimax3_s16x2_relu(DE, F, Z2) : __vimax_s16x2_relu(DE, F);
          Er[r] = E;
          Fr[r] = F;
          if (TB) {
            // nibble bits c: 3 E > D, 2 F > max(D, E), 1 E extended, 0 F extended.
            // The flag of slot r (bit 15 of its difference) belongs at bit
            // 28 - 4r + c of the word, that of slot r + 4 (bit 31) at 12 - 4r + c.
            // Registers r and r + 2 place a flag 8 bits apart, so one byte permute
            // takes the four sign bits of flag c of both registers as 0x00 / 0xff
            // bytes (255 x flag) in the order of their target bits, and a
            // multiply-add by 2^(4 - 4r + c) on the FMA pipe adds 255 x those bits to
            // a sum.  The sum is 255 x the word; 255 is odd, so one multiply by its
            // inverse mod 2^32 gives the word.
            fl[rq][3] = x16_gt(E, D);
            fl[rq][2] = x16_gt(F, DE);
            fl[rq][1] = x16_gt(E, Eo);
            fl[rq][0] = x16_gt(F, Fo);
            if (rq >= 2) {
#pragma unroll
              for (int cc = 3; cc >= 0; --cc) {
                uint32_t pk;
                asm("prmt.b32 %0, %1, %2, 0xD9FB;" : "=r"(pk) : "r"(fl[rq][cc]), "r"(fl[rq - 2][cc]));
                asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(acc) : "r"(pk), "r"(1u << (4 - 4 * (rq - 2) + cc)), "r"(acc));
              }
            }
          }
        }
        if (TB) nib[g] = acc * 0xfefefeffu;  // 255^-1 mod 2^32
      }
      if (TB) {  // rows start on a sector, so a 16-slot thread's two words are one 8-byte store
        if constexpr (G == 2)
          *reinterpret_cast<uint2 *>(tbp) = make_uint2(nib[0], nib[G - 1]);
        else
          tbp[0] = nib[0];
      }
    }
    if (TB) tbp += ROW;

    // ---- antidiagonal k: its reductions, and what k + 1 takes from them --------------
    combine();
    // nothing alive on k: the sweep ends there (in a fast block pl is then above every ol)
    if ((SLOW || LOCAL || ZD || W > 1) && b2 == 0) return X16_END;
    settle(Hp);
    if (xrun) brun2 = max(brun2, b2);
    if (SLOW && k == M + N) corner = true;
    const int kk = k + 1, cn = c + (PH == 0 ? 1 : 0);
    int low = PH == 0 ? pl - 1 : pl, high = PH == 0 ? ph : ph + 1;  // the candidate slots
    const bool cut = SLOW || LOCAL || ol < low || oh > high;
    if (SLOW) {
      const int jA = max(max(0, kk - M), max(cn + low, (kk + band_lo + 1) >> 1));
      const int jB = min(min(N, kk), min(cn + high, (kk + band_hi) >> 1));
      if (jA > jB) return X16_END;
      low = jA - cn;
      high = jB - cn;
      // (A window moved by whole threads may be left by a range some 20 cells narrower,
      // the widest group's, held to diagonals, by one of two cells less.  Such a pair none
      // of whose antidiagonals has more cells than the window goes on in the int32 sweep,
      // whose window follows the range; others would outgrow that one too)
      if (low < 0 || high >= WIN) {
        const int most = min(min(M, N) + 1, (band_hi - band_lo) / 2 + 1);
        return W == XD_MAX_WARPS && most <= WIN ? X16_OVF : X16_WIDE;
      }
      const int bp = (int)(b2 & 0xffffu), rp = xrun ? (int)(brun2 & 0xffffu) : bp;
      int tmin = rp - X;
      if (ZD) tmin -= max(abs(2 * jA - kk - dbest), abs(2 * jB - kk - dbest));
      if (bp > pceil || tmin < pfloor) return X16_OVF;
      const int a0 = max(jA, 1), b0 = min(jB, kk - 1);
      cells += (uint64_t)max(b0 - a0 + 1, 0);
    }
    // ---- prune k + 1 -----------------------------------------------------------------
    const uint32_t K = CX2 - (xrun ? brun2 : b2);  // 0x8000 - threshold in each half
    uint32_t t2 = 0, am = 0;
    if (cut && !(SLOW || LOCAL || ZD || W > 1) && b2 == 0) return X16_END;
    if (!SLOW) span += ph - pl;  // high - low + 1 = ph - pl + 2 cells
    ol = pl;
    oh = ph;
    if (!idle) {
      if (cut) {
        const int vA = low - base_slot, vB = high - base_slot;
        constexpr uint32_t SFULL = (1u << S) - 1u;
        uint32_t dom = 0;
        if (vB >= 0 && vA < S) dom = (SFULL << max(vA, 0)) & (SFULL >> (S - 1 - min(vB, S - 1))) & SFULL;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const uint32_t d = ((dom >> (8 * g)) & 0xfu) | (((dom >> (8 * g + 4)) & 0xfu) << 16);
#pragma unroll
          for (int rq = 0; rq < 4; ++rq) Hr[4 * g + rq] &= x16_halfmask(d << (15 - rq));
        }
      }
      const int zx = ZD ? 2 * (cn + base_slot) - kk - dbest : 0;
      const uint32_t zp = x16_splat(zx), zn = x16_splat(-zx);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        uint32_t w = 0;
#pragma unroll
        for (int rq = 0; rq < 4; ++rq) {
          const int r = 4 * g + rq;
          uint32_t Kr = K;
          if (ZD) {  // the threshold falls by the distance from the best diagonal, down to 1
            const int a = 2 * (8 * g + rq);
            const uint32_t up = ((uint32_t)a) | ((uint32_t)(a + 8) << 16);
            const uint32_t dn = ((uint32_t)(-a) & 0xffffu) | ((uint32_t)(-(a + 8)) << 16);
            const uint32_t neg = __viaddmax_s16x2(zn, dn, X16_K80);
            Kr = __vminu2(K + __viaddmax_s16x2(zp, up, neg), 0x7fff7fffu);
          }
          const uint32_t m = x16_halfmask(Hr[r] + Kr);  // [H >= threshold] per half
          const uint32_t hm = Hr[r] & m;
          finish_cell(Hc[r], r, hm, m, Er[r], Fr[r]);
          w |= m & (0x10001u << rq);
        }
        am |= bits8(w) << (8 * g);
        t2 = __vimax3_s16x2_relu(t2, Hc[4 * g], Hc[4 * g + 1]);
        t2 = __vimax3_s16x2_relu(t2, Hc[4 * g + 2], Hc[4 * g + 3]);
      }
      t2 = __vimax_s16x2_relu(t2, __byte_perm(t2, t2, 0x1032));
    }
    // ---- reductions of k + 1 (consumed after the next raw update) -----------------------
    if (SLOW || STEP_K) {
      k = kk;
      c = cn;
    }
    b2 = __reduce_max_sync(X16_FULL, t2);
    pl = __reduce_min_sync(X16_FULL, am ? base_slot + __ffs(am) - 1 : INT_MAX);
    ph = __reduce_max_sync(X16_FULL, am ? base_slot + 31 - __clz(am) : INT_MIN);
    if (ZD || (LOCAL && W > 1)) pbs = need_bs ? best_slot_of(Hc, b2) : 0;
    if (SLOW && kk == M + N) {  // the corner is the single cell of antidiagonal M + N
      const int pc = N - cn - base_slot;
      if (pc >= 0 && pc < S) {
        // slot pc: register 4 (pc / 8) + pc % 4, high half when pc % 8 >= 4
        uint32_t hv = 0;
#pragma unroll
        for (int r = 0; r < P; ++r)
          hv |= Hc[r] & (0u - (uint32_t)(4 * (pc >> 3) + (pc & 3) == r));
        const int v = ((pc & 7) < 4) ? (int)(hv & 0xffffu) : (int)(hv >> 16);
        cornerH = v ? v - X16_C0 + base : NEG;
      }
    }
    if constexpr (W > 1) publish();
    return X16_GO;
  }

  // every state value moves by -sft (the base by +sft)
  __device__ __forceinline__ void rebase(int sft) {
    base += sft;
    const uint32_t d2 = x16_splat(-sft);
#pragma unroll
    for (int r = 0; r < P; ++r) {
      Ha[r] = __viaddmax_s16x2_relu(Ha[r], d2, 0u);
      Hb[r] = __viaddmax_s16x2_relu(Hb[r], d2, 0u);
      En[r] = __viaddmax_s16x2_relu(En[r], d2, 0u);
      Fn[r] = __viaddmax_s16x2_relu(Fn[r], d2, 0u);
      Ho[r] = __viaddmax_s16x2_relu(Ho[r], d2, 0u);
    }
  }

  // the window moves up by s slots, whole threads but in the widest group: thread x
  // takes the state of thread x + s / S
  __device__ __forceinline__ void move_array(uint32_t (&v)[P], int s) {
    const int t = s / S;
    const bool in = tid + t >= 0 && tid + t < W * 32;
    if constexpr (ANY_SLOT) {
      __syncthreads();
      sh.move[tid] = make_uint4(v[0], v[1], v[2], v[3]);
      __syncthreads();
      const uint16_t *half = reinterpret_cast<const uint16_t *>(sh.move);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        uint32_t x = 0;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int q = base_slot + r + 4 * hh + s;
          if (q >= 0 && q < WIN) x |= (uint32_t)half[(q & ~7) + 2 * (q & 3) + (q >> 2 & 1)] << (16 * hh);
        }
        v[r] = x;
      }
    } else if constexpr (W == 1) {
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const uint32_t x = __shfl_sync(X16_FULL, v[r], (lane + t) & 31);
        v[r] = in ? x : 0u;
      }
    } else {
      __syncthreads();
      sh.move[tid] = make_uint4(v[0], v[1], v[2], v[3]);
      __syncthreads();
      const uint4 x = in ? sh.move[tid + t] : make_uint4(0u, 0u, 0u, 0u);
      v[0] = x.x;
      v[1] = x.y;
      v[2] = x.z;
      v[3] = x.w;
    }
  }
  __device__ __forceinline__ void move_window(int s) {
    move_array(Ha, s);
    move_array(Hb, s);
    move_array(En, s);
    move_array(Fn, s);
    move_array(Ho, s);
    c += s;
    pl -= s;
    ph -= s;
    if (pbs >= 0) pbs -= s;
    if (ol <= oh) {
      ol -= s;
      oh -= s;
    }
    if constexpr (W > 1) {
      // the next step reads its neighbours' edges and the warps' reductions (the
      // group's values stand for each warp's: they are combined again)
      __syncthreads();
      publish();
    }
  }
};

template <int W, int G, bool LOCAL, bool TB, bool ZD, bool UNI>
// (16-slot threads: at most 168 registers, three blocks of four groups per SM)
__global__ void __launch_bounds__(W == 1 ? 128 : W * 32, W == 1 ? (G == 2 ? 3 : 5) : 1)
    k_sweep16(const FullArgs a, uint32_t *overflow, uint32_t *n_overflow, X16Knobs kn) {
  static_assert(G == 1 || (G == 2 && W == 1), "16 slots per thread in one-warp groups only");
  using SW = Sweep16<W, G, LOCAL, TB, ZD, UNI>;
  constexpr int S = SW::S, P = SW::P, WIN = SW::WIN;
  constexpr int WCODE = W * G;  // the group width the host and the walks know: slots / 256
  constexpr int GROUPS = (W == 1) ? 4 : 1;
  __shared__ X16Shared<W> shm[GROUPS];
  __shared__ int8_t s_sub[MAX_ALPHA * MAX_ALPHA];
  const int A = a.sp.alphabet;
  for (int t = threadIdx.x; t < A * A; t += blockDim.x) s_sub[t] = a.sp.subst[t];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int grp = (W == 1) ? (int)(threadIdx.x >> 5) : 0;
  SW w(shm[grp]);
  X16Shared<W> &sh = shm[grp];
  w.s_sub = s_sub;
  w.A = A;
  w.lane = lane;
  w.warp = (W == 1) ? 0 : (int)(threadIdx.x >> 5);
  w.tid = w.warp * 32 + lane;
  w.base_slot = w.tid * S;
  const int tid = w.tid, base_slot = w.base_slot;
  const int o = a.sp.o, e = a.sp.e;
  w.oe = o + e;
  w.X = a.sp.xdrop;
  w.smax = max(a.sp.smax, 0);
  w.xrun = a.sp.xrun != 0;
  // the largest packed best that leaves every formed value inside 16 bits,
  // and the lowest threshold that keeps every relevant value above the floor
  w.pceil = 0x7fff - 4 * w.smax - 2 * w.oe - 8;
  w.pfloor = 2 * w.smax + 2 * w.oe + 8;
  w.MA2 = x16_splat(a.sp.uni_match);
  w.MI2 = x16_splat(a.sp.uni_mismatch);
  w.NOE2 = x16_splat(-w.oe);
  w.NE2 = x16_splat(-e);
  w.CX2 = x16_splat(0x8000 + w.X);

  auto gsync = [&]() {
    if (W == 1)
      __syncwarp();
    else
      __syncthreads();
  };

  const uint32_t ck_i = blockIdx.x * GROUPS + grp;
  bool first_item = true;
  for (;;) {
    // ---- next pair ------------------------------------------------------------
    uint32_t t0 = 0;
    if (a.ck) {  // a descriptor per group
      t0 = (first_item && ck_i < a.n_ck) ? 0u : a.n_order;
      first_item = false;
    } else if (W == 1) {
      if (lane == 0) t0 = atomicAdd(a.counter, 1u);
      t0 = __shfl_sync(X16_FULL, t0, 0);
    } else {
      if (threadIdx.x == 0) sh.pair = atomicAdd(a.counter, 1u);
      __syncthreads();
      t0 = sh.pair;
      __syncthreads();
    }
    if (t0 >= a.n_order) break;
    const uint32_t p = a.order[t0];
    const int M = (int)a.b.q_len[p], N = (int)a.b.r_len[p];
    w.M = M;
    w.N = N;
    w.q = a.b.q_seq + a.b.q_off[p];
    w.rs = a.b.r_seq + a.b.r_off[p];
    int64_t blo = -(int64_t)M, bhi = N;
    if (a.sp.use_band) band_limits(M, N, a.sp.band, a.sp.band_literal, &blo, &bhi);
    w.band_lo = (int)max(blo, -(int64_t)M);
    w.band_hi = (int)min(bhi, (int64_t)N);

    const XdCkpt *ck = a.ck ? a.ck + ck_i : nullptr;
    const int ckmode = ck ? ck->mode : 0;
    const int seg = ck ? ck->k_start / ck->C : 0;
    if (ckmode == 3) {
      bool skip = ck->flags[0] != 0 || ck->flags[1 + seg] != 0;
      if (!skip && ck->k_start > 0)
        skip = ck->buf[(int64_t)seg * xd_ckpt_stride() + XCK_USED] > WIN;
      if (skip) break;
    }
    uint32_t *tbp = nullptr;
    int32_t *ckp = nullptr;
    if (TB) {
      if (ckmode == 2) {
        ckp = ck->seg_ck;
        tbp = ck->seg_tb;
      } else {
        ckp = reinterpret_cast<int32_t *>(a.tb + a.tbl[p].off);
        tbp = a.tb + a.tbl[p].off + (uint64_t)xd_origin_words(M, N);
      }
    }

    // ---- antidiagonal 0 (or the checkpoint resumed) ----------------------------
    // (0, 0) sits in the middle of the window
    constexpr int MID = W * 16 * S;
    w.base = 0;
    w.c = -MID;
    w.dbest = 0;
    w.bv = w.bi = w.bj = 0;
    w.cells = 0;
    w.cornerH = INT_MIN;
    w.corner = false;
    w.pl = w.ph = MID;
    int dprev = 0;
#pragma unroll
    for (int r = 0; r < P; ++r) w.Ha[r] = w.Hb[r] = w.En[r] = w.Fn[r] = w.Ho[r] = 0u;
    if (base_slot == MID) {  // H(0, 0) = 0
      w.Hb[0] = (uint32_t)X16_C0;
      w.Ho[0] = w.En[0] = w.Fn[0] = (uint32_t)max(X16_C0 - w.oe, 0);
    }
    int status = FILTR_ST_OK;
    int k_first = 1, k_last = M + N;
    int row0 = 0;  // traceback row of antidiagonal k: k - row0
    if (TB && tid == 0 && ckmode == 0) ckp[0] = w.c;
    if (ckmode >= 2) {
      k_first = ck->k_start + 1;
      row0 = k_first;
      k_last = min(ck->k_end, M + N);
      if (ck->k_start > 0) {
        const int32_t *rec = ck->buf + (int64_t)seg * xd_ckpt_stride();
        w.c = rec[XCK_ORIGIN];
        dprev = rec[XCK_DPREV];
        w.base = rec[XCK_BEST];
        w.dbest = rec[XCK_DBEST];
        w.pl = (ck->k_start + rec[XCK_LO]) / 2 - w.c;
        w.ph = (ck->k_start + rec[XCK_HI]) / 2 - w.c;
        const int wwin = rec[XCK_WIN], b0 = w.base;
        auto pk = [&](int v) -> uint32_t {  // real -> packed (minus infinity and far below: 0)
          const int x = v - b0 + X16_C0;
          return (v <= NEG_HALF || x <= 0) ? 0u : (uint32_t)min(x, 0x7fff);
        };
        // records hold eight-slot threads: group g of this thread is record thread tid * G + g
#pragma unroll
        for (int r = 0; r < P; ++r) {
          const int g = r >> 2, rq = r & 3;
          const int32_t *mine = rec + XCK_HDR + (tid * G + g) * 32;
          const bool inl = base_slot + 8 * g + rq < wwin, inh = base_slot + 8 * g + rq + 4 < wwin;
          w.Hb[r] = (inl ? pk(mine[rq]) : 0u) | ((inh ? pk(mine[rq + 4]) : 0u) << 16);
          w.En[r] = (inl ? pk(mine[8 + rq]) : 0u) | ((inh ? pk(mine[8 + rq + 4]) : 0u) << 16);
          w.Fn[r] = (inl ? pk(mine[16 + rq]) : 0u) | ((inh ? pk(mine[16 + rq + 4]) : 0u) << 16);
          w.Ha[r] = (inl ? pk(mine[24 + rq]) : 0u) | ((inh ? pk(mine[24 + rq + 4]) : 0u) << 16);
          // records hold what a neighbour's E and F are (see finish_cell)
          w.Ho[r] = __viaddmax_s16x2_relu(w.Hb[r], w.NOE2, 0u);
          w.En[r] = __vimax_s16x2_relu(w.En[r], w.Ho[r]);
          w.Fn[r] = __vimax_s16x2_relu(w.Fn[r], w.Ho[r]);
        }
        if (ckmode == 3) {
          w.bv = rec[XCK_BV];
          w.bi = rec[XCK_BI];
          w.bj = rec[XCK_BJ];
          w.cells = (uint64_t)(uint32_t)rec[XCK_CELLS_LO] | ((uint64_t)(uint32_t)rec[XCK_CELLS_HI] << 32);
        }
      }
    }
    const bool first_b = dprev == 1;  // resumed after a phase A step: a phase B step comes first
    if (first_b) {  // H of k_first - 1 belongs in Ha, which that step reads
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const uint32_t x = w.Ha[r];
        w.Ha[r] = w.Hb[r];
        w.Hb[r] = x;
      }
    }
    w.k = k_first - 1;
    w.b2 = x16_splat(X16_C0);  // best(k_first - 1) is the base
    w.brun2 = w.b2;
    w.ol = -(1 << 29);  // the antidiagonal before is not known: the first step masks its range
    w.oh = 1 << 29;
    w.pbs = (w.k + w.dbest) / 2 - w.c;  // a step settles on it again
    // the best cell is the result of local alignments; Z-drop needs each
    // antidiagonal's best diagonal.  A global X-drop pair reports its best
    // cell only when it is dropped, which it then takes from the int32 rerun,
    // so its sweep keeps neither.
    w.track = (LOCAL || ZD) && ckmode != 2;
    w.need_bs = ZD || w.track;
    w.Z2 = 0u;
    bool resumed = true;  // the state's best cell and diagonal are already settled
    w.tbp = TB ? tbp + (int64_t)(k_first - row0) * SW::ROW + G * tid : nullptr;
    if (W > 1) w.move_window(0);  // publish the edges and reductions
    w.load_codes(w.k, w.c);
    int stop = X16_GO;
    uint32_t qx = 0, rx = 0;
    bool ahead = false;  // qx, rx hold the next block's codes
    const bool keep_track = w.track;

    while (stop == X16_GO && w.k < k_last) {
      // ---- a block of 16 antidiagonals (or what is left) ----------------------------
      w.combine();
      if (w.b2 == 0) {
        stop = X16_END;
        break;
      }
      if (kn.rebase > 0) {  // keep the packed range centred on the best
        const int sft = (int)(w.b2 & 0xffffu) - X16_C0;
        if (sft > kn.rebase || sft < -kn.rebase) {
          w.rebase(sft);
          w.b2 = x16_splat(X16_C0);
          w.brun2 = __viaddmax_s16x2_relu(w.brun2, x16_splat(-sft), 0u);
          if (W > 1) w.move_window(0);  // publish the shifted values
        }
      }
      if (LOCAL) w.Z2 = x16_splat(min(max(X16_C0 - w.base, 0), 0x7fff));
      const bool phase_b = resumed && first_b;
      // room on each side (a block moves an end by 8 slots), and the new codes
      // (in one-warp groups the first and last thread stay dead besides: a fast
      // step does not clear the edge values that wrap around to them)
      constexpr int ROOM = X16_BLOCK / 2 + 1 + (W == 1 ? S : 1);
      int block = X16_BLOCK;
      if (w.pl < ROOM || w.ph > WIN - 1 - ROOM) {
        const int mid = (w.pl + w.ph) >> 1;
        int s = SW::ANY_SLOT ? mid - WIN / 2 : (mid - WIN / 2) / S * S;
        if (SW::ANY_SLOT && w.ph - w.pl >= WIN - 2 * ROOM) {
          // less room than a block takes: two antidiagonals at a time (columns [a1, b1] and
          // up to b2 at most), in a window that holds them and the live range, if one does
          block = 2;
          const int l = w.c + w.pl, h = w.c + w.ph, k1 = w.k + 1, k2 = k1 + 1, d = phase_b ? 0 : 1;
          const int a1 = max(max(max(0, k1 - M), (k1 + w.band_lo + 1) >> 1), l);
          const int b1 = min(min(min(N, k1), (k1 + w.band_hi) >> 1), h + 1);
          const int b2 = phase_b ? b1 : min(min(min(N, k2), (k2 + w.band_hi) >> 1), b1 + 1);
          const int most = min(l, a1 - d);  // the origin
          const int least = max(h + 1, b2 + 1 - d) - WIN;
          s = max(min(w.c, most), min(least, most)) - w.c;
        }
        if (s != 0) {
          w.move_window(s);
          w.load_codes(w.k, w.c);
          ahead = false;
        }
      }
      const int kb = w.k + 1;
      if (UNI) {
        if (ahead) {
          w.qn = qx;
          w.rn = rx;
        } else {
          w.load_next(w.qn, w.rn, 0);
          if (phase_b) w.rn = 0;  // a lone phase B step takes a query code only
        }
        ahead = !phase_b && block == X16_BLOCK;
        if (ahead) w.load_next(qx, rx, X16_BLOCK / 2);
      } else if (phase_b) {
        const int i = kb - w.c - base_slot;
        w.qn = (i >= 1 && i <= M) ? w.q[i - 1] : 0u;
      } else if (!ahead) {
        const int j = w.c + 1 + base_slot + S - 1;
        w.rn = (j >= 1 && j <= N) ? w.rs[j - 1] : 0u;
        ahead = true;
      }
      if (TB) {  // the block's window origins
        const int x = phase_b ? 0 : lane;
        if (w.warp == 0 && lane < (phase_b ? 1 : block) && kb + x <= k_last)
          ckp[kb - row0 + x] = phase_b ? w.c : w.c + 1 + (x >> 1);
      }
      const int bp = (int)(w.b2 & 0xffffu), rp = w.xrun ? max((int)(w.brun2 & 0xffffu), bp) : bp;
      const int dlo = 2 * (w.c + w.pl) - w.k - X16_BLOCK, dhi = 2 * (w.c + w.ph) - w.k + X16_BLOCK;
      const int kend = w.k + X16_BLOCK;
      const bool fast = !phase_b && kend <= k_last && kend < M + N && !resumed && w.pl >= ROOM &&
                        w.ph <= WIN - 1 - ROOM && kb - dhi >= 2 && kb + dlo >= 2 &&
                        (int64_t)kend + dhi <= 2 * (int64_t)N && (int64_t)kend - dlo <= 2 * (int64_t)M &&
                        dlo >= w.band_lo && dhi <= w.band_hi && bp + 9 * w.smax <= w.pceil &&
                        rp - w.X - (ZD ? max(dhi, w.dbest) - min(dlo, w.dbest) : 0) - X16_BLOCK * w.oe >= w.pfloor;
      if (fast) {
        w.span = 0;
        int x = 0;
#pragma unroll 1
        for (; x < X16_BLOCK; x += 2) {
          stop = w.template step<0, false>(w.Ha, w.Hb);
          if (stop != X16_GO) break;
          stop = w.template step<1, false>(w.Hb, w.Ha);
          if (stop != X16_GO) {
            ++x;
            break;
          }
        }
        w.cells += (uint64_t)(uint32_t)(w.span + 2 * x);
        if (!SW::STEP_K) {
          w.k += x;
          w.c += (x + 1) >> 1;
        }
      } else {
        int x = phase_b ? 1 : 0;
        const int xe = phase_b ? 2 : block;
#pragma unroll 1
        for (; x < xe && w.k < k_last; ++x) {
          if (resumed) w.track = false;
          if ((x & 1) == 0)
            stop = w.template step<0, true>(w.Ha, w.Hb);
          else
            stop = w.template step<1, true>(w.Hb, w.Ha);
          if (resumed) {
            w.track = keep_track;
            resumed = false;
          }
          if (stop != X16_GO) break;
        }
        if (phase_b) ahead = false;
      }
    }
    // H of the last antidiagonal: Ha after a phase A step, Hb after a phase B step
    const bool in_a = (((w.k - k_first) & 1) == 0) != first_b;
    bool ended = stop == X16_END;
    if (stop == X16_WIDE) status = FILTR_ST_TOO_WIDE;
    if (stop == X16_OVF) status = X16_OVERFLOW;
    if (stop == X16_GO) {  // the last antidiagonal's reductions
      w.combine();
      if (w.b2 == 0) {
        ended = true;
      } else {
        if (w.k >= k_first) {
          uint32_t hl[P];
#pragma unroll
          for (int r = 0; r < P; ++r) {
            const uint32_t x = w.Ha[r], y = w.Hb[r];
            hl[r] = in_a ? x : y;
          }
          w.settle(hl);
        }
        if (w.xrun) w.brun2 = max(w.brun2, w.b2);
        if (w.k == M + N) w.corner = true;
      }
    }
    const bool corner = w.corner;
    if (status == FILTR_ST_OK && stop == X16_GO && k_last == M + N) ended = true;
    // a dropped global pair without its best cell: the int32 sweep finds it
    if (!LOCAL && !w.track && ckmode != 2 && status == FILTR_ST_OK && ended && !corner) status = X16_OVERFLOW;
    if (ckmode == 3 && status == FILTR_ST_TOO_WIDE && WCODE < XD_MAX_WARPS) break;
    if (ckmode >= 2 && status == X16_OVERFLOW) {  // the whole pair goes to the int32 sweep
      if (tid == 0 && ckmode == 3) ck->flags[0] = 3;
      break;
    }

    // the corner value lives in one thread; broadcast it
    int cornerH = w.cornerH;
    if (!LOCAL) {
      int ch = __reduce_max_sync(X16_FULL, cornerH);
      if (W > 1) {
        __syncthreads();
        if (lane == 0) sh.tmp[0][w.warp] = ch;
        __syncthreads();
        ch = INT_MIN;
        for (int x = 0; x < W; ++x) ch = max(ch, sh.tmp[0][x]);
      }
      cornerH = ch;
    }
    if (ckmode == 3 && !ended && status == FILTR_ST_OK) {
      // segment done, sweep not finished: store the window state after k_end,
      // moved down by whole eight-slot threads so that it starts at the window's
      // first slots (a narrower group may take it up)
      int32_t *rec = ck->buf + (int64_t)(ck->k_end / ck->C) * xd_ckpt_stride();
      int used = 0, first = INT_MAX;
      uint32_t h1[P], h2[P];
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const uint32_t x = w.Ha[r], y = w.Hb[r];
        h1[r] = in_a ? x : y;
        h2[r] = in_a ? y : x;
        const int sl = base_slot + 8 * (r >> 2) + (r & 3);  // slot of the low half
        const uint32_t any = h1[r] | h2[r] | w.En[r] | w.Fn[r];
        if (any & 0xffffu) used = max(used, sl + 1), first = min(first, sl);
        if (any >> 16) used = max(used, sl + 5), first = min(first, sl + 4);
      }
      used = __reduce_max_sync(X16_FULL, used);
      first = __reduce_min_sync(X16_FULL, first);
      if (W > 1) {
        __syncthreads();
        if (lane == 0) {
          sh.tmp[0][w.warp] = used;
          sh.tmp[1][w.warp] = first;
        }
        __syncthreads();
        for (int x = 0; x < W; ++x) {
          used = max(used, sh.tmp[0][x]);
          first = min(first, sh.tmp[1][x]);
        }
      }
      const int drop = first == INT_MAX ? 0 : first >> 3;  // eight-slot threads
      const int bs = w.base;
      auto rv = [&](uint32_t x, int hh) -> int32_t {  // packed half -> real (0: minus infinity)
        const int v = hh ? (int)(x >> 16) : (int)(x & 0xffffu);
        return v ? v - X16_C0 + bs : NEG;
      };
      // eight-slot record threads: group g of this thread is record thread tid * G + g - drop
#pragma unroll
      for (int r = 0; r < P; ++r) {
        const int at = tid * G + (r >> 2) - drop;
        if (at < 0) continue;
        int32_t *mine = rec + XCK_HDR + at * 32;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int s = (r & 3) + 4 * hh;
          mine[s] = rv(h1[r], hh);
          mine[8 + s] = rv(w.En[r], hh);
          mine[16 + s] = rv(w.Fn[r], hh);
          mine[24 + s] = rv(h2[r], hh);
        }
      }
      if (tid == 0) {
        rec[XCK_ORIGIN] = w.c + 8 * drop;
        rec[XCK_DPREV] = in_a ? 1 : 0;  // phase A moved the origin
        rec[XCK_BEST] = (w.xrun ? (int)(w.brun2 & 0xffffu) : (int)(w.b2 & 0xffffu)) - X16_C0 + w.base;
        rec[XCK_LO] = 2 * (w.c + w.pl) - w.k;
        rec[XCK_HI] = 2 * (w.c + w.ph) - w.k;
        rec[XCK_DBEST] = w.dbest;
        rec[XCK_USED] = used - 8 * drop;
        rec[XCK_WIN] = WIN - 8 * drop;
        rec[XCK_BV] = w.bv;
        rec[XCK_BI] = w.bi;
        rec[XCK_BJ] = w.bj;
        rec[XCK_CELLS_LO] = (int32_t)(uint32_t)w.cells;
        rec[XCK_CELLS_HI] = (int32_t)(uint32_t)(w.cells >> 32);
        ck->flags[1 + seg] = WCODE;
      }
      gsync();
      continue;
    }
    if (tid == 0 && ckmode != 2) {
      if (ckmode == 3) {
        ck->flags[0] = 1;
        if (status != FILTR_ST_TOO_WIDE) ck->flags[1 + seg] = WCODE;
      }
      int score = 0, ei = 0, ej = 0;
      if (status == FILTR_ST_TOO_WIDE) {
        const uint32_t slot = atomicAdd(n_overflow, 1u);
        overflow[slot] = p;
      } else if (status == X16_OVERFLOW) {
        const uint32_t slot = atomicAdd(a.n_ovf16, 1u);
        a.ovf16[slot] = p;
        status = FILTR_ST_TOO_WIDE;  // until the int32 rerun writes the result
      } else if (LOCAL) {
        if (w.bv > 0) {
          score = w.bv;
          ei = w.bi;
          ej = w.bj;
        } else {
          status = FILTR_ST_EMPTY;
        }
      } else if (corner) {
        score = cornerH;
        ei = M;
        ej = N;
      } else {
        status = FILTR_ST_DROPPED;
        score = w.bv;
        ei = w.bi;
        ej = w.bj;
      }
      filtr_result res;
      res.score = score;
      res.q_end = ei;
      res.r_end = ej;
      res.q_begin = (LOCAL && status == FILTR_ST_OK) ? -1 : 0;
      res.r_begin = res.q_begin;
      res.status = status;
      res.cigar_len = 0;
      res.reserved = 0;
      res.cigar_off = 0;
      res.cells = w.cells;
      a.out[p] = res;
      FwdOut f;
      f.score = score;
      f.end_i = ei;
      f.end_j = ej;
      f.status = status;
      a.fwd[p] = f;
    }
    gsync();
  }
}
// Group widths: W = 1 (256 slots) runs one warp per pair (8 slots per thread,
// four pairs per 128-thread block).  W = 2 (512 slots) runs one warp of 16-slot
// threads: bookkeeping done once per warp and no block barriers.  (Two warps of
// 8-slot threads have half the cell work each, but exchanging edges and
// reductions every antidiagonal costs more: the megabase pair's forward took
// 670 ms that way, 601 ms on one warp.)  The traceback rows and the checkpoint
// records are those of 8-slot threads: thread t of the one-warp group writes
// words 2t and 2t + 1.  W >= 4 runs W warps of 8-slot threads; those instances take
// 168 to 193 registers (half the blocks per SM of the sweep with a sliding origin; at
// W = 32, held to 64, they spill 284 to 516 bytes) and gain for their fewer instructions.
// Whole calls, the sliding origin and this: W = 1, 10,000 long reads 244 -> 134 ms; W = 2,
// 1,500 Z-drop reads 17.7 -> 10.9; W = 4, 1,000 reads of 4-8 kbp with X = 1500 26.1 -> 18.6;
// W = 8, X = 3500 48.1 -> 35.8; W = 16, 400 reads, X = 7000 44.6 -> 29.3; W = 32, 200 protein
// pairs of 6-9 thousand, X = 7500 70.7 -> 41.4.
template <int KW, int G, bool LOCAL, bool TB, bool ZD>
cudaError_t x16_launch(const FullArgs &a, int grid, uint32_t *ovf, uint32_t *novf, X16Knobs kn,
                       cudaStream_t s) {
  if (a.sp.uni)
    k_sweep16<KW, G, LOCAL, TB, ZD, true><<<grid, KW == 1 ? 128 : KW * 32, 0, s>>>(a, ovf, novf, kn);
  else
    k_sweep16<KW, G, LOCAL, TB, ZD, false><<<grid, KW == 1 ? 128 : KW * 32, 0, s>>>(a, ovf, novf, kn);
  return cudaGetLastError();
}

template <int KW, int G, bool ZD>
cudaError_t x16_dispatch(const FullArgs &a, int grid, uint32_t *ovf, uint32_t *novf, X16Knobs kn,
                         cudaStream_t s) {
  const bool L = a.sp.mode == FILTR_LOCAL, T = a.sp.traceback != 0;
  if (L) return T ? x16_launch<KW, G, true, true, ZD>(a, grid, ovf, novf, kn, s)
                  : x16_launch<KW, G, true, false, ZD>(a, grid, ovf, novf, kn, s);
  return T ? x16_launch<KW, G, false, true, ZD>(a, grid, ovf, novf, kn, s)
           : x16_launch<KW, G, false, false, ZD>(a, grid, ovf, novf, kn, s);
}

template <int KW, int G, bool LOCAL, bool TB, bool ZD>
int x16_occ() {
  int nb = 0, nb2 = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_sweep16<KW, G, LOCAL, TB, ZD, true>, KW == 1 ? 128 : KW * 32, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb2, k_sweep16<KW, G, LOCAL, TB, ZD, false>, KW == 1 ? 128 : KW * 32,
                                                0);
  return std::min(nb, nb2);
}

template <int KW, int G, bool ZD>
int x16_occ_w(const ScoreParams &sp) {
  const bool L = sp.mode == FILTR_LOCAL, T = sp.traceback != 0;
  if (L) return T ? x16_occ<KW, G, true, true, ZD>() : x16_occ<KW, G, true, false, ZD>();
  return T ? x16_occ<KW, G, false, true, ZD>() : x16_occ<KW, G, false, false, ZD>();
}

template <bool ZD>
cudaError_t x16_launch_any(const FullArgs &a, int W, int grid, uint32_t *ovf, uint32_t *novf, X16Knobs kn,
                           cudaStream_t s) {
  switch (W) {
    case 1: return x16_dispatch<1, 1, ZD>(a, grid, ovf, novf, kn, s);
    case 2: return x16_dispatch<1, 2, ZD>(a, grid, ovf, novf, kn, s);
    case 4: return x16_dispatch<4, 1, ZD>(a, grid, ovf, novf, kn, s);
    case 8: return x16_dispatch<8, 1, ZD>(a, grid, ovf, novf, kn, s);
    case 16: return x16_dispatch<16, 1, ZD>(a, grid, ovf, novf, kn, s);
    case 32: return x16_dispatch<32, 1, ZD>(a, grid, ovf, novf, kn, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool ZD>
int x16_occ_any(int W, const ScoreParams &sp) {
  switch (W) {
    case 1: return x16_occ_w<1, 1, ZD>(sp);
    case 2: return x16_occ_w<1, 2, ZD>(sp);
    case 4: return x16_occ_w<4, 1, ZD>(sp);
    case 8: return x16_occ_w<8, 1, ZD>(sp);
    case 16: return x16_occ_w<16, 1, ZD>(sp);
    case 32: return x16_occ_w<32, 1, ZD>(sp);
    default: return 0;
  }
}

}  // namespace
}  // namespace filtr
