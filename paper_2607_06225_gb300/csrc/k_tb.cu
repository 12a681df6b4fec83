// k_tb.cu -- traceback walk, CIGAR offset scan and CIGAR compaction.
//
// The walk follows the 4-bit choices the forward kernels stored (one nibble per
// cell, see tb_push4 in filtr_internal.h) from
// the end cell back to the start, tracking the current value so that a local
// walk stops on the first H of 0 (Smith-Waterman) and emitting run-length BAM
// ops in reverse into a per-pair staging area.  Global walks that reach row 0
// or column 0 finish with the forced gap.  A scan then places every pair's
// CIGAR in pair order and a warp per pair copies it forward into the caller's
// buffer.
#include <climits>

#include "filtr_internal.h"
#include "k_xdrop_layout.h"

namespace filtr {
namespace {

constexpr int OP_I = 1, OP_D = 2, OP_EQ = 7, OP_X = 8;

struct FullGeom {
  int R, HS, M, N;
  bool band;
  int64_t lo, hi;
  int64_t base;   // first word of strip `s`
  int s;          // current strip (or one past the last)
  int64_t jlo;    // first column of strip s
  int64_t nsteps; // steps of strip s
};

__device__ __forceinline__ void geom_seek(FullGeom &g, int s) {
  while (g.s != s) {  // move `base` strip by strip
    int64_t jl, jh;
    if (g.s < s) {
      strip_cols((int64_t)g.s * g.HS, g.HS, g.M, g.N, g.band, g.lo, g.hi, &jl, &jh);
      g.base += strip_tb_words(jl, jh, g.R);
      ++g.s;
      strip_cols((int64_t)g.s * g.HS, g.HS, g.M, g.N, g.band, g.lo, g.hi, &jl, &jh);
    } else {
      --g.s;
      strip_cols((int64_t)g.s * g.HS, g.HS, g.M, g.N, g.band, g.lo, g.hi, &jl, &jh);
      g.base -= strip_tb_words(jl, jh, g.R);
    }
    g.jlo = jl;
    g.nsteps = jh >= jl ? (jh - jl + 1) + 31 : 0;
  }
}

// A cursor past the last strip of an M x N int32 tile (strips of 32 * R rows):
// base = the words of every strip, so the first seek moves it down to the strip
// that holds the row asked for.
__device__ __forceinline__ void geom_init(FullGeom &g, int R, int M, int N, const ScoreParams &sp) {
  g.R = R;
  g.HS = 32 * R;
  g.M = M;
  g.N = N;
  g.band = sp.use_band != 0;
  band_limits(M, N, sp.band, sp.band_literal, &g.lo, &g.hi);
  if (!g.band) {
    g.lo = -(int64_t)M - 1;
    g.hi = (int64_t)N + 1;
  }
  const int nstrips = (M + g.HS - 1) / g.HS;
  g.base = 0;
  g.s = nstrips;
  g.jlo = 1;
  g.nsteps = 0;
  for (int s = 0; s < nstrips; ++s) {
    int64_t jl, jh;
    strip_cols((int64_t)s * g.HS, g.HS, M, N, g.band, g.lo, g.hi, &jl, &jh);
    g.base += strip_tb_words(jl, jh, g.R);
  }
}

// Choice bits of cell (i, j) of an int32 tile (banded or not).  Successive calls
// on one cursor should ask for rows near each other.
__device__ __forceinline__ uint32_t full_bits(const uint32_t *tb, FullGeom &g, int i, int j) {
  const int s = (i - 1) / g.HS;
  geom_seek(g, s);
  const int rho = (i - 1) - s * g.HS;
  const int l = rho / g.R, k = rho - l * g.R;
  const int64_t t = (int64_t)j - g.jlo + l;
  if (t < 0 || t >= g.nsteps) return 0;  // never taken on a consistent traceback
  const int wps = (g.R + 7) / 8;
  const uint32_t w = __ldg(tb + g.base + (t * wps + (k >> 3)) * 32 + l);
  return tb_nibble(w, k);
}

// The int16x2 tiled kernel's layout (unbanded): every strip has N + 63 steps
// of 2 * ceil(R/16) words per lane; the high half of a lane's rows runs one step behind.
struct PackGeom {
  int R;
  int64_t strip_words;
};

__device__ __forceinline__ uint32_t pack_bits(const uint32_t *tb, const PackGeom &g, int i, int j) {
  const int HS = 32 * g.R, P = g.R >> 1;
  const int s = (i - 1) / HS;
  const int rho = (i - 1) - s * HS;
  const int l = rho / g.R, kk = rho - l * g.R;
  const int h = kk >= P ? 1 : 0, k = kk - h * P;
  const int64_t t = (int64_t)j - 1 + 2 * l + h;
  const int G = (P + 7) / 8, wps = 2 * G;
  const uint32_t w = __ldg(tb + s * g.strip_words + (t * wps + h * G + (k >> 3)) * 32 + l);
  const int c = k & 7;
  return (((w >> c) & 1u) << 3) | (((w >> (8 + c)) & 1u) << 2) | (((w >> (16 + c)) & 1u) << 1) |
         ((w >> (24 + c)) & 1u);
}

struct Emitter {
  uint32_t *st;
  uint32_t n;
  int cur;
  uint32_t run;
  __device__ void put(int op, uint32_t len) {
    if (op == cur) {
      run += len;
    } else {
      if (cur >= 0) st[n++] = (run << 4) | (uint32_t)cur;
      cur = op;
      run = len;
    }
  }
  __device__ void flush() {
    if (cur >= 0) st[n++] = (run << 4) | (uint32_t)cur;
    cur = -1;
  }
};

// One thread walks pair p (any layout).
__device__ __forceinline__ void walk_thread(const WalkArgs &a, const BatchDev &b,
                                            filtr_result *out, uint32_t p) {
  const FwdOut f = a.fwd[p];
  const TbLayout L = a.tbl[p];
  if (f.status != FILTR_ST_OK && f.status != FILTR_ST_DROPPED) {
    out[p].cigar_len = 0;
    return;
  }
  const int M = (int)b.q_len[p], N = (int)b.r_len[p];
  const uint8_t *q = b.q_seq + b.q_off[p];
  const uint8_t *r = b.r_seq + b.r_off[p];
  const bool local = a.sp.mode == FILTR_LOCAL;
  const int A = a.sp.alphabet, e = a.sp.e, oe = a.sp.o + a.sp.e;
  const uint32_t *tb = a.tb + L.off;

  FullGeom g;
  XdGeom xg;
  PackGeom pg{L.R, (int64_t)pack_strip_tb_words(1, N, L.R)};
  if (L.family == FAM_FULL && L.valid) {
    geom_init(g, L.R, M, N, a.sp);
  } else if (L.family == FAM_XDROP && L.valid) {
    xd_geom_init(xg, tb, M, N, L);
  }

  Emitter em{a.stage + a.stage_off[p], 0, -1, 0};
  int i = f.end_i, j = f.end_j, v = f.score, state = 0;
  for (;;) {
    if (state == 0) {
      if (i == 0 && j == 0) break;
      if (local && v == 0) break;
      if (i == 0) {
        em.put(OP_D, (uint32_t)j);
        j = 0;
        break;
      }
      if (j == 0) {
        em.put(OP_I, (uint32_t)i);
        i = 0;
        break;
      }
      const uint32_t nib = (L.family == FAM_FULL)   ? full_bits(tb, g, i, j)
                                 : (L.family == FAM_PACK) ? pack_bits(tb, pg, i, j)
                                                          : xd_bits(xg, i, j);
      if (nib & TB_PF) {
        state = 2;
      } else if (nib & TB_PE) {
        state = 1;
      } else {
        const int qc = q[i - 1], rc = r[j - 1];
        em.put(qc == rc ? OP_EQ : OP_X, 1);
        v -= a.sp.subst[qc * A + rc];
        --i;
        --j;
      }
    } else if (state == 1) {
      if (j == 0) {
        state = 0;
        continue;
      }
      const uint32_t nib = (L.family == FAM_FULL)   ? full_bits(tb, g, i, j)
                                 : (L.family == FAM_PACK) ? pack_bits(tb, pg, i, j)
                                                          : xd_bits(xg, i, j);
      em.put(OP_D, 1);
      if (nib & TB_EEXT) {
        v += e;
      } else {
        v += oe;
        state = a.sp.mid ? 3 : 0;
      }
      --j;
    } else if (state == 2) {
      if (i == 0) {
        state = 0;
        continue;
      }
      const uint32_t nib = (L.family == FAM_FULL)   ? full_bits(tb, g, i, j)
                                 : (L.family == FAM_PACK) ? pack_bits(tb, pg, i, j)
                                                          : xd_bits(xg, i, j);
      em.put(OP_I, 1);
      if (nib & TB_FEXT) {
        v += e;
      } else {
        v += oe;
        state = a.sp.mid ? 3 : 0;
      }
      --i;
    } else {  // state 3 (M/I/D): the gap opened from M here, a diagonal step
      if (i == 0 && j == 0) break;
      const int qc = q[i - 1], rc = r[j - 1];
      em.put(qc == rc ? OP_EQ : OP_X, 1);
      v -= a.sp.subst[qc * A + rc];
      --i;
      --j;
      state = 0;
    }
  }
  em.flush();
  filtr_result *res = out + p;
  res->q_begin = i;
  res->r_begin = j;
  res->cigar_len = em.n;
}

__global__ void k_walk(const WalkArgs a) {
  const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  const GraphDesc *gd = a.gd;  // captured pipeline: batch, outputs and count from here
  if (gd && gd->abort) return;
  if (t >= (gd ? gd->n : a.n_order)) return;
  walk_thread(a, gd ? gd->b : a.b, gd ? gd->out : a.out, a.order[t]);
}

// ---- warp walks ----------------------------------------------------------------
// The walk is serial, and one thread per pair spends it waiting on a dependent
// load per step.  A warp keeps a band of choice bits on chip instead: 32 rows
// (iw - 31 .. iw) by the eight diagonals d0 - 4 .. d0 + 3 around the path, lane x
// loading the eight cells of row iw - x.  While the path crosses these rows the
// next 32 are already being loaded, around the diagonal the path entered this
// window on (and for the antidiagonal layout, whose words are found through the
// window origins, the origins of the rows after those).  A path that drifts off
// the band is loaded again around where it is.
//
// The state of the walk is the same in every lane.  A run of diagonal steps (matches and
// mismatches, H taken from the diagonal) is taken in one go: lane d looks at the
// cell d steps down the diagonal, a ballot finds where the run ends (a gap, row or
// column 0, the band's edge, or for local alignments the first cell of value 0,
// found by a warp scan of the scores), and another tells '=' from 'X'.  A gap's
// extension bits are looked at the same way, along the row or the column.
//
// Measured against windows of 32 antidiagonals loaded when the path enters them
// (antidiagonal layout) and three cached lines of 32 cells (tiles), walked by lane
// 0 but for the diagonal runs: see the figures at launch_walk.

struct WalkCore {
  const uint8_t *q, *r;
  const int8_t *subst;
  int A, e, oe;
  bool local, mid;  // mid: a gap that opened leaves through a diagonal step (state 3)
  int i, j, v, state;
  uint32_t *st;     // staged ops
  uint32_t n, run;  // ops staged; length of the op being grown
  int cur;
  __device__ __forceinline__ void put(int op, uint32_t len) {
    if (op == cur) {
      run += len;
    } else {
      flush();
      cur = op;
      run = len;
    }
  }
  __device__ __forceinline__ void flush() {
    if (cur >= 0) {
      if ((threadIdx.x & 31) == 0) st[n] = (run << 4) | (uint32_t)cur;
      ++n;
    }
    cur = -1;
  }
  __device__ __forceinline__ void store(filtr_result *res) {  // the finished walk
    flush();
    if ((threadIdx.x & 31) == 0) {
      res->q_begin = i;
      res->r_begin = j;
      res->cigar_len = n;
    }
  }
};

__device__ __forceinline__ WalkCore walk_core(const WalkArgs &a, const BatchDev &b, uint32_t p, const int8_t *subst) {
  WalkCore w;
  w.q = b.q_seq + b.q_off[p];
  w.r = b.r_seq + b.r_off[p];
  w.subst = subst;
  w.A = a.sp.alphabet;
  w.e = a.sp.e;
  w.oe = a.sp.o + a.sp.e;
  w.local = a.sp.mode == FILTR_LOCAL;
  w.mid = a.sp.mid != 0;
  w.st = a.stage + a.stage_off[p];
  w.n = w.run = 0;
  w.cur = -1;
  w.state = 0;
  return w;
}

constexpr int WB = 8;       // diagonals of the band
constexpr int WB_MID = 4;   // the path's diagonal when the band is loaded around it
struct WalkBand {
  uint8_t nb[32][WB];       // choice bits: row iw - x, diagonal d0 - WB_MID + y
  int32_t c[96];            // antidiagonal layout: origins of kc, kc - 1, ...
};

// Loaders keep the raw words of one window in registers between issue() and
// commit().
//
// Tiled layouts: a word of each cell of the lane's row.
struct TileLoader {
  const uint32_t *tb;
  bool pk, fb;
  PackGeom pg;
  FullGeom g;    // banded int32 tiles: this lane's strip cursor
  int R, M, N;
  int s, row0;   // this lane's strip and its first row (0-based)
  uint32_t raw[WB];
  int sub;       // the cells' place in their words
  __device__ __forceinline__ void start(WalkBand &, int, int) {}
  __device__ __forceinline__ void ahead(WalkBand &, int, int) {}
  __device__ __forceinline__ void issue(WalkBand &, int iw, int d0) {
    const int i = iw - (int)(threadIdx.x & 31), j0 = i + d0 - WB_MID;
#pragma unroll
    for (int y = 0; y < WB; ++y) raw[y] = 0;
    if (i < 1) return;
    const int HS = 32 * R;
    while (i <= row0) row0 -= HS, --s;  // the rows move a window at a time
    while (i > row0 + HS) row0 += HS, ++s;
    const int rho = i - 1 - row0, l = rho * ((1 << 20) / R + 1) >> 20, k = rho - l * R;  // rho / R, rho < 1024
    int64_t at;
    int stride, steps, t;
    if (pk) {
      const int P = R >> 1, h = k >= P ? 1 : 0, kk = k - h * P, G = (P + 7) >> 3;
      t = j0 - 1 + 2 * l + h;
      at = (int64_t)s * pg.strip_words + (h * G + (kk >> 3)) * 32 + l;
      stride = 64 * G;
      steps = N + 63;
      sub = kk & 7;
    } else {
      int64_t base;
      int jlo = 1;
      steps = N + 31;
      if (fb) {
        geom_seek(g, s);
        base = g.base;
        jlo = (int)g.jlo;
        steps = (int)g.nsteps;
      } else {
        base = (int64_t)s * strip_tb_words(1, N, R);
      }
      t = j0 - jlo + l;
      at = base + (k >> 3) * 32 + l;
      stride = (R + 7) / 8 * 32;
      sub = 4 * (7 - (k & 7));
    }
    const uint32_t *w = tb + at + (int64_t)t * stride;
    if (j0 >= 1 && j0 + WB - 1 <= N && t >= 0 && t + WB - 1 < steps) {
#pragma unroll
      for (int y = 0; y < WB; ++y) raw[y] = __ldg(w + y * stride);
    } else {
#pragma unroll
      for (int y = 0; y < WB; ++y)
        if (j0 + y >= 1 && j0 + y <= N && t + y >= 0 && t + y < steps) raw[y] = __ldg(w + y * stride);
    }
  }
  __device__ __forceinline__ void commit(WalkBand &C) {
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int y = 0; y < WB; ++y) {
      const uint32_t x = raw[y] >> sub;
      const uint32_t nib = pk ? ((x & 1u) << 3) | ((x >> 8 & 1u) << 2) | ((x >> 16 & 1u) << 1) | (x >> 24 & 1u)
                              : x & 15u;
      if (y < 4)
        lo |= nib << (8 * y);
      else
        hi |= nib << (8 * (y - 4));
    }
    __syncwarp();  // the last window's readers are done
    *reinterpret_cast<uint2 *>(C.nb[threadIdx.x & 31]) = make_uint2(lo, hi);
    __syncwarp();
  }
};

// Where antidiagonal k's window origin and traceback row live (antidiagonals stay
// below 2^31).  run(k): row k's words, with those of the rows around it in the
// range (lo, hi] at multiples of wpk.
struct XdRows {  // one pair's own layout
  const int32_t *ck;
  const uint32_t *tb;
  int wpk;
  int lo, hi;
  __device__ __forceinline__ int origin(int k) const { return __ldg(ck + k); }
  __device__ __forceinline__ const uint32_t *run(int k) { return tb + (int64_t)k * wpk; }
};
struct XdSegRows {  // recomputed segments, segment s = (k - 1) / C, from antidiagonal k0 + 1 on
  const XdCkpt *seg;     // by segment: where its rows are
  const int32_t *width;  // by segment: group width it was computed at
  const int32_t *ck;     // origins of k0 + 1, k0 + 2, ...
  int C, k0;
  int wpk, lo, hi;       // the segment looked up last
  const uint32_t *base;
  __device__ __forceinline__ int origin(int k) const { return __ldg(ck + (k - 1 - k0)); }
  __device__ __forceinline__ const uint32_t *run(int k) {
    if (k <= lo || k > hi) {
      const int s = (k - 1) / C;
      wpk = xd_words_per_k(__ldg(width + s), 8);
      base = seg[s].seg_tb;
      lo = s * C;
      hi = lo + C;
    }
    return base + (int64_t)(k - 1 - lo) * wpk;
  }
};

// Antidiagonal layout: the word of cell (i, j) sits in the row of antidiagonal
// i + j, at the slot the row's origin tells.  The origins of a window's 70
// antidiagonals (and eight on each side, for a band loaded a few diagonals off)
// are loaded one window earlier than its words.
template <class Rows>
struct XdLoader {
  Rows rows;
  int k_min, k_max;  // antidiagonals that have a row: k_min < k <= k_max
  int cn[3];         // origins on their way: kn, kn - 1, ... (lane + 32 z)
  int kn, kc;        // top of cn; top of the band's c
  uint32_t raw[WB];
  uint32_t sub;      // 4 bits per cell: its slot within its word
  __device__ __forceinline__ void load_origins(int iw, int d0) {
    kn = 2 * iw + d0 + (WB - 1 - WB_MID) + 8;
#pragma unroll
    for (int z = 0; z < 3; ++z) {
      const int k = kn - (int)(threadIdx.x & 31) - 32 * z;
      cn[z] = k > k_min && k <= k_max ? rows.origin(k) : 0;
    }
  }
  __device__ __forceinline__ void store_origins(WalkBand &C) {
    __syncwarp();
#pragma unroll
    for (int z = 0; z < 3; ++z) C.c[(threadIdx.x & 31) + 32 * z] = cn[z];
    kc = kn;
    __syncwarp();
  }
  // the first window of a band at (iw, d0): its origins, waited for
  __device__ __forceinline__ void start(WalkBand &C, int iw, int d0) {
    load_origins(iw, d0);
    store_origins(C);
  }
  // the window after the one about to be issued at (iw, d0)
  __device__ __forceinline__ void ahead(WalkBand &C, int iw, int d0) { load_origins(iw, d0); }
  __device__ __forceinline__ void issue(WalkBand &C, int iw, int d0) {
    const int i = iw - (int)(threadIdx.x & 31), j0 = i + d0 - WB_MID, k0 = i + j0, x0 = kc - k0;
    sub = 0;
    // (the bounds on x0 always hold: a band is issued at most 3 diagonals off its origins)
    if (i >= 1 && j0 >= 1 && k0 > k_min && k0 + WB - 1 <= k_max && x0 >= WB - 1 && x0 < 96) {
      const uint32_t *row = rows.run(k0);
      const bool one = k0 > rows.lo && k0 + WB - 1 <= rows.hi;
#pragma unroll
      for (int y = 0; y < WB; ++y) {
        if (!one && y) row = rows.run(k0 + y);
        const int p = j0 + y - C.c[x0 - y];
        raw[y] = (unsigned)p < 8u * (unsigned)rows.wpk ? __ldg(row + (p >> 3)) : 0u;
        sub |= (uint32_t)(p & 7) << (4 * y);
        row += rows.wpk;
      }
    } else {
#pragma unroll
      for (int y = 0; y < WB; ++y) {
        const int j = j0 + y, k = k0 + y, x = x0 - y;
        raw[y] = 0;
        if (i >= 1 && j >= 1 && k > k_min && k <= k_max && x >= 0 && x < 96) {
          const uint32_t *row = rows.run(k);
          const int p = j - C.c[x];
          if ((unsigned)p < 8u * (unsigned)rows.wpk) raw[y] = __ldg(row + (p >> 3));
          sub |= (uint32_t)(p & 7) << (4 * y);
        }
      }
    }
  }
  __device__ __forceinline__ void commit(WalkBand &C) {
    uint32_t lo = 0, hi = 0;
#pragma unroll
    for (int y = 0; y < WB; ++y) {
      const uint32_t nib = raw[y] >> (28 - 4 * (sub >> (4 * y) & 7u)) & 15u;
      if (y < 4)
        lo |= nib << (8 * y);
      else
        hi |= nib << (8 * (y - 4));
    }
    __syncwarp();  // the last window's readers are done
    *reinterpret_cast<uint2 *>(C.nb[threadIdx.x & 31]) = make_uint2(lo, hi);
    __syncwarp();
  }
};
template <class L>
struct WalkAhead {  // a window's origins must be stored before its words are issued
  static __device__ __forceinline__ void next(L &ld, WalkBand &C, int iw, int d0) { ld.issue(C, iw, d0); }
};
template <class Rows>
struct WalkAhead<XdLoader<Rows>> {
  static __device__ __forceinline__ void next(XdLoader<Rows> &ld, WalkBand &C, int iw, int d0) {
    ld.store_origins(C);
    ld.issue(C, iw, d0);
    ld.ahead(C, iw - 32, d0);
  }
};

// Walks until the alignment's start is reached (true), or until the current cell
// is on antidiagonal k_stop or before (false, state kept).
template <class L>
__device__ __forceinline__ bool walk_band(WalkCore &w, L &ld, WalkBand &C, int k_stop) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int iw = 0, d0 = 0, dn = 0;  // this window; the diagonal the next is issued around
  bool open = false;
  for (;;) {
    if (w.state == 0) {
      if ((w.i == 0 && w.j == 0) || (w.local && w.v == 0)) return true;
      if (w.i == 0) {
        w.put(OP_D, (uint32_t)w.j);
        w.j = 0;
        return true;
      }
      if (w.j == 0) {
        w.put(OP_I, (uint32_t)w.i);
        w.i = 0;
        return true;
      }
    }
    if (w.i + w.j <= k_stop) return false;
    if (w.state == 1 && w.j == 0) {
      w.state = 0;
      continue;
    }
    if (w.state == 2 && w.i == 0) {
      w.state = 0;
      continue;
    }
    if (w.state == 3) {  // the gap opened from M here, so this cell is a diagonal step
      if (w.i == 0 && w.j == 0) return true;
      const int qc = w.q[w.i - 1], rc = w.r[w.j - 1];
      w.put(qc == rc ? OP_EQ : OP_X, 1);
      w.v -= w.subst[qc * w.A + rc];
      --w.i;
      --w.j;
      w.state = 0;
      continue;
    }
    // ---- the window that holds (i, j) ---------------------------------------------
    int x0 = iw - w.i, y0 = w.j - w.i - d0 + WB_MID;
    if (!open || x0 >= 32 || y0 < 0 || y0 >= WB) {
      const int d = w.j - w.i, yn = d - dn + WB_MID;
      if (open && x0 == 32 && yn >= 1 && yn < WB - 1) {  // the next one, on its way since this one was entered
        iw -= 32;
        d0 = dn;
      } else {
        iw = w.i;
        d0 = d;
        ld.start(C, iw, d0);
        ld.issue(C, iw, d0);
        ld.ahead(C, iw - 32, d);
        open = true;
      }
      ld.commit(C);
      dn = d;
      WalkAhead<L>::next(ld, C, iw - 32, d);
      if (lane < 2) {  // the residues of the rows after those
        const uint8_t *s = lane ? w.r + w.j : w.q + w.i;
        if ((lane ? w.j : w.i) > 192) asm volatile("prefetch.global.L1 [%0];" ::"l"(s - 192));
      }
      x0 = iw - w.i;
      y0 = d - d0 + WB_MID;
    }
    if (w.state == 0) {  // a run down the diagonal
      const int ii = w.i - lane, jj = w.j - lane;
      bool ok = ii >= 1 && jj >= 1 && ii + jj > k_stop && x0 + lane < 32;
      uint32_t nib = 0;
      int qc = 0, rc = 1, sc = 0;
      if (ok) {
        nib = C.nb[x0 + lane][y0];
        ok = (nib & (TB_PE | TB_PF)) == 0u;
        qc = __ldg(w.q + ii - 1);
        rc = __ldg(w.r + jj - 1);
      }
      int dv = 0;
      if (w.local) {
        if (ok) sc = w.subst[qc * w.A + rc];
        int pre = sc;  // inclusive scan of the scores down the diagonal
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(FULL, pre, o);
          if (lane >= o) pre += t;
        }
        if (w.v - (pre - sc) == 0) ok = false;  // the value at cell d
        dv = pre;
      }
      const unsigned okm = __ballot_sync(FULL, ok);
      const int n = okm == FULL ? 32 : __ffs(~okm) - 1;
      if (n > 0) {
        const unsigned eqm = __ballot_sync(FULL, qc == rc);
        if (w.local) w.v -= __shfl_sync(FULL, dv, n - 1);
        int d = 0;
        while (d < n) {
          const unsigned rest = eqm >> d;
          const bool eq = (rest & 1u) != 0u;
          const unsigned stop = eq ? ~rest : rest;
          const int len = min(stop ? __ffs(stop) - 1 : 32 - d, n - d);
          w.put(eq ? OP_EQ : OP_X, (uint32_t)len);
          d += len;
        }
        w.i -= n;
        w.j -= n;
        continue;
      }
      nib = __shfl_sync(FULL, nib, 0);
      w.state = nib & TB_PF ? 2 : 1;
    }
    // ---- a gap: lane t looks at its t-th residue's extension bit --------------------
    const bool down = w.state == 2;  // along the column (query residues), else the row
    const int ii = down ? w.i - lane : w.i, jj = down ? w.j : w.j - lane;
    const int x = down ? x0 + lane : x0, y = down ? y0 + lane : y0 - lane;
    const bool in = ii >= 1 && jj >= 1 && ii + jj > k_stop && x < 32 && y >= 0 && y < WB;
    const bool ext = in && (C.nb[in ? x : 0][in ? y : 0] & (down ? TB_FEXT : TB_EEXT)) != 0u;
    const unsigned extm = __ballot_sync(FULL, ext), inm = __ballot_sync(FULL, in);
    const int n = extm == FULL ? 32 : __ffs(~extm) - 1;    // residues that extend
    const bool opens = n < 32 && (inm >> n & 1u) != 0u;   // and then one that opens the gap
    const int len = n + (opens ? 1 : 0);
    if (len > 0) w.put(down ? OP_I : OP_D, (uint32_t)len);
    w.v += n * w.e + (opens ? w.oe : 0);
    if (down)
      w.i -= len;
    else
      w.j -= len;
    if (opens) w.state = w.mid ? 3 : 0;
  }
}

__device__ __forceinline__ void load_subst(int8_t *s_sub, const ScoreParams &sp) {
  for (int x = threadIdx.x; x < sp.alphabet * sp.alphabet; x += blockDim.x) s_sub[x] = sp.subst[x];
  __syncthreads();
}

// One warp per pair of a batched X-drop call (4 pairs per 128-thread block).
__global__ void __launch_bounds__(128) k_walk_xdw(const WalkArgs a) {
  __shared__ WalkBand band[4];
  __shared__ int8_t s_sub[MAX_ALPHA * MAX_ALPHA];
  load_subst(s_sub, a.sp);
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t t = blockIdx.x * 4 + wib;
  if (t >= a.n_order) return;
  const uint32_t p = a.order[t];
  const FwdOut f = a.fwd[p];
  const TbLayout L = a.tbl[p];
  if (f.status != FILTR_ST_OK && f.status != FILTR_ST_DROPPED) {
    if (lane == 0) a.out[p].cigar_len = 0;
    return;
  }
  const int M = (int)a.b.q_len[p], N = (int)a.b.r_len[p];
  const uint32_t *base = a.tb + L.off;
  WalkCore w = walk_core(a, a.b, p, s_sub);
  w.i = f.end_i;
  w.j = f.end_j;
  w.v = f.score;
  XdLoader<XdRows> ld;
  ld.rows = XdRows{reinterpret_cast<const int32_t *>(base), base + xd_origin_words(M, N),
                   xd_words_per_k(L.warps, L.R), INT_MIN, INT_MAX};
  ld.k_min = 0;
  ld.k_max = w.i + w.j;
  walk_band(w, ld, band[wib], -1);
  w.store(a.out + p);
}

// One warp per pair over the tiled layouts.
__global__ void __launch_bounds__(128) k_walk_tw(const WalkArgs a) {
  __shared__ WalkBand band[4];
  __shared__ int8_t s_sub[MAX_ALPHA * MAX_ALPHA];
  load_subst(s_sub, a.sp);
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t t = blockIdx.x * 4 + wib;
  const GraphDesc *gd = a.gd;  // captured pipeline: batch, outputs and count from here
  if (gd && gd->abort) return;
  if (t >= (gd ? gd->n : a.n_order)) return;
  const BatchDev b = gd ? gd->b : a.b;
  filtr_result *const out = gd ? gd->out : a.out;
  const uint32_t p = a.order[t];
  const TbLayout L = a.tbl[p];
  const bool pk = L.family == FAM_PACK;
  if (!L.valid || !(pk || L.family == FAM_FULL)) {
    if (lane == 0) walk_thread(a, b, out, p);  // empty pairs
    return;
  }
  const FwdOut f = a.fwd[p];
  if (f.status != FILTR_ST_OK && f.status != FILTR_ST_DROPPED) {
    if (lane == 0) out[p].cigar_len = 0;
    return;
  }
  WalkCore w = walk_core(a, b, p, s_sub);
  w.i = f.end_i;
  w.j = f.end_j;
  w.v = f.score;
  TileLoader ld;
  ld.tb = a.tb + L.off;
  ld.pk = pk;
  ld.fb = !pk && a.sp.use_band;
  ld.R = L.R;
  ld.M = (int)b.q_len[p];
  ld.N = (int)b.r_len[p];
  ld.s = 0;
  ld.row0 = 0;
  ld.pg = PackGeom{L.R, (int64_t)pack_strip_tb_words(1, ld.N, L.R)};
  if (ld.fb) geom_init(ld.g, L.R, ld.M, ld.N, a.sp);
  walk_band(w, ld, band[wib], -1);
  w.store(out + p);
}

// Resumable walk over recomputed segments (antidiagonals above k0) of a
// checkpointed X-drop traceback; one warp.  Stops when the walk reaches k0 (earlier
// segments, recomputed next, go on from the saved state) or when the alignment's
// start is reached.
__global__ void k_walk_segments(const WalkArgs a, const XdSegRows rows, WalkState *ws) {
  __shared__ WalkBand band;
  __shared__ int8_t s_sub[MAX_ALPHA * MAX_ALPHA];
  load_subst(s_sub, a.sp);
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const WalkState st = *ws;
  if (st.done) return;
  const uint32_t p = a.order[0];
  WalkCore w = walk_core(a, a.b, p, s_sub);
  w.i = st.i;
  w.j = st.j;
  w.v = st.v;
  w.state = st.state;
  w.n = st.n;
  w.cur = st.cur;
  w.run = st.run;
  XdLoader<XdSegRows> ld;
  ld.rows = rows;
  ld.k_min = rows.k0;
  ld.k_max = w.i + w.j;
  // (a walk in a gap stops on k0 as well; 0 is the start itself)
  const bool done = walk_band(w, ld, band, rows.k0 > 0 ? rows.k0 : -1);
  __syncwarp();
  if (done) w.store(a.out + p);
  if (threadIdx.x == 0) {
    WalkState o;
    o.i = w.i;
    o.j = w.j;
    o.v = w.v;
    o.state = w.state;
    o.done = done ? 1 : 0;
    o.n = w.n;
    o.cur = w.cur;
    o.run = w.run;
    *ws = o;
  }
}

// Exclusive scan of cigar_len (pair order) into offs; *total = sum.  One CTA.
__global__ void k_scan(const filtr_result *out, uint32_t n, uint64_t *offs, uint64_t *total,
                       const GraphDesc *gd) {
  __shared__ uint64_t part[1024];
  __shared__ uint64_t carry;
  if (gd) {  // captured pipeline (uniform over the block)
    if (gd->abort) return;
    out = gd->out;
    n = gd->n;
  }
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  constexpr int PER = 8;
  for (uint64_t base = 0; base < n; base += (uint64_t)blockDim.x * PER) {
    uint64_t v[PER];
    uint64_t sum = 0;
    const uint64_t b0 = base + (uint64_t)threadIdx.x * PER;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      v[k] = (b0 + k < n) ? out[b0 + k].cigar_len : 0;
      sum += v[k];
    }
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
      uint64_t add = (threadIdx.x >= (unsigned)off) ? part[threadIdx.x - off] : 0;
      __syncthreads();
      part[threadIdx.x] += add;
      __syncthreads();
    }
    uint64_t run = carry + part[threadIdx.x] - sum;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      if (b0 + k < n) offs[b0 + k] = run;
      run += v[k];
    }
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry += part[threadIdx.x];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

// One warp per pair: reverse the staged ops into the caller's buffer.
__global__ void k_compact(const WalkArgs a, uint32_t n, const uint64_t *offs, uint32_t *cigar,
                          uint64_t cap, filtr_result *out) {
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (a.gd) {  // captured pipeline
    if (a.gd->abort) return;
    n = a.gd->n;
    cigar = a.gd->cigar;
    cap = a.gd->cap;
    out = a.gd->out;
  }
  if (w >= n) return;
  const uint32_t len = out[w].cigar_len;
  const uint64_t off = offs[w];
  if (lane == 0) out[w].cigar_off = off;
  if (len == 0 || cigar == nullptr || off + len > cap) return;
  const uint32_t *st = a.stage + a.stage_off[w];
  for (uint32_t x = lane; x < len; x += 32) cigar[off + x] = st[len - 1 - x];
}

}  // namespace

constexpr uint32_t WALK_WARP_PAIRS = 16384;

cudaError_t launch_walk(const WalkArgs &a, cudaStream_t s) {
  if (a.n_order == 0) return cudaSuccess;
  // A warp per pair keeps more loads in flight for each pair but issues the
  // serial walk as a whole warp's instructions.  Up to about one warp per resident
  // slot of the device (and some) it is the faster form; with many more pairs a
  // thread per pair (32 pairs per instruction stream) is: 2.5 ms against 3.4 ms
  // for 100,000 protein pairs.  The band windows of walk_band took the walk of 64
  // protein pairs from 0.17 to 0.10 ms, of 512 banded reads from 6.2 (a thread
  // per pair: about 27) to 2.1, of an 80 kbp banded pair from 21.3 to 7.4, of a
  // megabase X-drop pair from 144 to 54 and of 10,000 long reads from 17.2 to 14.5.
  if (a.n_order <= WALK_WARP_PAIRS)
    k_walk_tw<<<(a.n_order + 3) / 4, 128, 0, s>>>(a);
  else
    k_walk<<<(a.n_order + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}


cudaError_t launch_walk_xd(const WalkArgs &a, cudaStream_t s) {
  if (a.n_order == 0) return cudaSuccess;
  k_walk_xdw<<<(a.n_order + 3) / 4, 128, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_walk_segments(const WalkArgs &a, const XdCkpt *seg, const int32_t *width, const int32_t *ck,
                                 int C, int k0, WalkState *st, cudaStream_t s) {
  k_walk_segments<<<1, 32, 0, s>>>(a, XdSegRows{seg, width, ck, C, k0, 0, 0, 0, nullptr}, st);
  return cudaGetLastError();
}

cudaError_t launch_scan_offsets(const filtr_result *out, uint32_t n, uint64_t *offs,
                                uint64_t *total, cudaStream_t s, const GraphDesc *gd) {
  k_scan<<<1, 1024, 0, s>>>(out, n, offs, total, gd);
  return cudaGetLastError();
}

cudaError_t launch_compact(const WalkArgs &a, uint32_t n, const uint64_t *offs, uint32_t *cigar,
                           uint64_t cap, filtr_result *out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t threads = (uint64_t)n * 32;
  k_compact<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(a, n, offs, cigar, cap, out);
  return cudaGetLastError();
}

}  // namespace filtr
