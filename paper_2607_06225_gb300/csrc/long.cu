// long.cu -- filtr_align_long: one long pair with every SM on it.
//
// X-drop pairs (and pairs with an empty side) run as a one-pair batch of the
// antidiagonal kernel with a 4-warp first window (reruns widen it), or as a
// segmented sweep; the antidiagonal order is inherently sequential, so one group
// is what the pair can use.  Full-matrix and banded pairs run a warp per row
// strip across the device (k_split.cuh), then the ordinary traceback walk.
#include <algorithm>
#include <cstring>
#include <vector>

#include "../../include/filtr_testing.h"
#include "filtr_ctx.h"
#include "k_split.cuh"
#include "k_xdrop_layout.h"
#include "plan.h"

namespace filtr {

// X-drop pairs with more antidiagonals than this run as a segmented sweep, each
// segment at the narrowest group width that holds its live region
constexpr int64_t XD_SEGMENTED_SWEEP = 1 << 16;
namespace {

struct Carve {
  char *base;
  size_t cap, used = 0;
  template <class T>
  T *take(size_t count) {
    used = (used + 255) / 256 * 256;
    T *p = reinterpret_cast<T *>(base + used);
    used += count * sizeof(T);
    return p;
  }
};

filtr_status validate_seq(Ctx *c, const uint8_t *q, uint32_t M, const uint8_t *r, uint32_t N,
                          int alphabet, cudaStream_t st) {
  uint32_t *d_bad = reinterpret_cast<uint32_t *>(c->d_small);
  cudaError_t e = cudaMemsetAsync(d_bad, 0, 4, st);
  if (e == cudaSuccess) e = launch_validate(q, M, alphabet, d_bad, st);
  if (e == cudaSuccess) e = launch_validate(r, N, alphabet, d_bad, st);
  if (!c->ensure_host(64)) return FILTR_ERR_NOMEM;
  uint32_t *h = reinterpret_cast<uint32_t *>(c->h_stage);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, d_bad, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "validating residues");
  if (*h) {
    set_error("%u residue codes are >= the alphabet size %d", *h, alphabet);
    return FILTR_ERR_INVALID;
  }
  return FILTR_OK;
}

// a warp per row strip of the int32 tile (k_split.cuh); withhold != 0 is the timeout test
filtr_status run_long(Ctx *c, const ScoreParams &sp, const uint8_t *q, uint32_t M, const uint8_t *r,
                      uint32_t N, filtr_result *out, uint32_t *cigar, uint64_t cap, cudaStream_t st,
                      int withhold, unsigned long long timeout_ns, bool sync = true, int R = 8) {
  const int HS = 32 * R;
  int64_t widest = N;
  if (sp.use_band) {
    int64_t lo, hi;
    band_limits(M, N, sp.band, sp.band_literal, &lo, &hi);
    widest = std::max<int64_t>(1, std::min<int64_t>(N, hi - lo + HS));
    // A banded strip starts when the one above is a strip's height further, so the
    // pair's time is the steps down its rows: strips of 4 rows per lane take 159
    // cheaper steps (0.27 us) for 128 rows where strips of 8 take 287 of 0.32 us for 256:
    // forward sweep of an 80 kbp pair with a 7 kbp wide band 31.3 -> 29.1 ms, its walk
    // over more strips 7.2 -> 7.7.  Not where a wide band keeps more than a warp per
    // scheduler busy, nor where the traceback (up to twice as much) does not fit.
    if (R == 8 && widest / 128 + 6 <= 4 * (int64_t)c->sms) {
      const uint64_t need = split_space(1, ((uint64_t)M + 127) / 128, (uint64_t)widest + 1).bytes +
                            (sp.traceback ? 4 * (full_tb_words(M, N, 4, sp) + M + N) : 0) + 8192;
      if (need <= c->ws_bytes)
        return run_long(c, sp, q, M, r, N, out, cigar, cap, st, withhold, timeout_ns, sync, 4);
    }
  }
  const uint32_t nstrips = (uint32_t)((M + (uint64_t)HS - 1) / HS);
  const uint64_t tb_words = sp.traceback ? full_tb_words(M, N, R, sp) : 0;
  // a banded strip starts HS columns after the one above, so only about
  // widest / HS of them ever run at once; more warps would only wait
  const int64_t in_flight = sp.use_band ? widest / HS + 6 : (int64_t)nstrips;
  const int grid = (int)std::max<int64_t>(
      withhold ? 2 : 1,
      std::min<int64_t>((int64_t)c->sms * c->split_blocks_per_sm(false, R, sp),
                        (std::min<int64_t>(in_flight, nstrips) + FULL_WARPS - 1) / FULL_WARPS));
  const uint64_t stride = (uint64_t)widest + 1;
  const SplitSpace space = split_space(1, nstrips, stride);

  Carve cv{c->ws, c->ws_bytes};
  char *d_split = cv.take<char>(space.bytes);
  FwdOut *d_fwd = cv.take<FwdOut>(1);
  uint32_t *d_one = cv.take<uint32_t>(16);  // order, lengths, offsets of the one-pair batch
  TbLayout *d_tbl = cv.take<TbLayout>(1);
  uint64_t *d_misc = cv.take<uint64_t>(8);   // stage_off, offsets, total
  uint32_t *d_stage = sp.traceback ? cv.take<uint32_t>((size_t)M + N + 1) : nullptr;
  uint32_t *d_tb = cv.take<uint32_t>(tb_words);
  if (cv.used > c->ws_bytes) {
    set_error("the long pair needs %zu workspace bytes (traceback %llu); the context has %zu -- "
              "use a band, X-drop, or score only",
              cv.used, (unsigned long long)tb_words * 4, c->ws_bytes);
    return FILTR_ERR_NOMEM;
  }
  // host-side constants for the one-pair batch used by the walk
  if (!c->ensure_host(4096)) return FILTR_ERR_NOMEM;
  char *h = reinterpret_cast<char *>(c->h_stage);
  uint32_t one[16] = {0, M, N};            // order[0] = 0, q_len = M, r_len = N
  TbLayout L{};
  L.off = 0;
  L.family = FAM_FULL;
  L.R = (uint8_t)R;
  L.warps = 1;
  L.valid = sp.traceback ? 1 : 0;
  uint64_t misc[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // stage_off, q_off, r_off
  memcpy(h, one, sizeof one);
  memcpy(h + 64, &L, sizeof L);
  memcpy(h + 128, misc, sizeof misc);
  cudaError_t e = cudaMemcpyAsync(d_one, h, sizeof one, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_tbl, h + 64, sizeof L, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_misc, h + 128, sizeof misc, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return cuda_fail(e, "long-pair setup");

  const uint64_t *d_off = d_misc + 1;
  const BatchDev b{q, r, d_off, d_off + 1, d_one + 1, d_one + 2};
  SplitLaunch sl{};
  sl.packed = false;
  sl.R = R;
  sl.count = 1;
  sl.max_strips = nstrips;
  sl.grid = grid;
  c->last_strip_rows = HS;
  sl.a.f.b = b;
  sl.a.f.sp = sp;
  sl.a.f.order = d_one;
  sl.a.f.out = out;
  sl.a.f.fwd = d_fwd;
  sl.a.f.tb = d_tb;
  sl.a.f.tbl = d_tbl;
  sl.a.timeout_ns = timeout_ns;
  sl.a.withhold = withhold;
  split_bind(&sl.a, d_split, space, (uint32_t)stride);
  const int *err = sl.a.err;
  c->span_begin(Ctx::PH_FORWARD, st);
  e = launch_split(sl, st);
  c->span_end(st);
  if (e != cudaSuccess) return cuda_fail(e, "long-pair kernel launch");
  uint32_t launches = 3;
  if (sp.traceback && !withhold) {
    WalkArgs wa;
    wa.b = b;
    wa.sp = sp;
    wa.order = d_one;
    wa.n_order = 1;
    wa.out = out;
    wa.fwd = d_fwd;
    wa.tb = d_tb;
    wa.tbl = d_tbl;
    wa.stage = d_stage;
    wa.stage_off = d_misc;
    c->span_begin(Ctx::PH_WALK, st);
    e = launch_walk(wa, st);
    c->span_end(st);
    if (e == cudaSuccess) e = launch_scan_offsets(out, 1, d_misc + 3, d_misc + 4, st);
    if (e == cudaSuccess) e = launch_compact(wa, 1, d_misc + 3, cigar, cap, out, st);
    launches += 3;
    if (e != cudaSuccess) return cuda_fail(e, "long-pair traceback");
  }
  c->last_launches = launches;
  c->last_cells_estimate = band_cells(M, N, sp);
  c->last_cells_packed = 0;
  c->last_waves = 1;
  if (!sync) return FILTR_OK;  // the result's status reports a timeout
  // the wait flag (and the CIGAR length) decide the status: synchronise once
  int *h_err = reinterpret_cast<int *>(h + 1024);
  filtr_result *h_res = reinterpret_cast<filtr_result *>(h + 1088);
  e = cudaMemcpyAsync(h_err, err, 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h_res, out, sizeof(filtr_result), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "long-pair completion");
  if (*h_err) {
    set_error("a strip wait ran out after %llu ns", (unsigned long long)timeout_ns);
    return FILTR_ERR_TIMEOUT;
  }
  if (sp.traceback && h_res->cigar_len > cap) {
    set_error("the CIGAR needs %u ops, cigar_cap is %llu", h_res->cigar_len, (unsigned long long)cap);
    return FILTR_ERR_CIGAR_CAP;
  }
  return FILTR_OK;
}

// X-drop with checkpointed traceback (a one-pair antidiagonal sweep).
filtr_status run_xdrop_ckpt(Ctx *c, const ScoreParams &sp, const filtr_params *params,
                            const uint8_t *q, uint32_t M, const uint8_t *r, uint32_t N,
                            filtr_result *out, uint32_t *cigar, uint64_t cap, cudaStream_t st,
                            int C) {
  const int64_t K = (int64_t)M + N;
  const int64_t nseg = (K + C - 1) / C;
  static const int kLadder[] = {1, 2, 4, 8, 16, XD_MAX_WARPS};
  Carve cv{c->ws, c->ws_bytes};
  int32_t *ck_buf = cv.take<int32_t>((size_t)(nseg + 1) * xd_ckpt_stride());
  XdCkpt *d_ck = cv.take<XdCkpt>(2 * nseg + 1);
  int32_t *d_flags = cv.take<int32_t>(nseg + 1);
  WalkState *d_ws = cv.take<WalkState>(1);
  FwdOut *d_fwd = cv.take<FwdOut>(1);
  uint32_t *d_one = cv.take<uint32_t>(16);   // order, lengths
  TbLayout *d_tbl = cv.take<TbLayout>(1);
  uint64_t *d_misc = cv.take<uint64_t>(8);   // stage_off, offsets, CIGAR offset
  uint32_t *d_ovf = cv.take<uint32_t>(4);
  // the CIGAR staging at the workspace's end, and what lies between: the pool that
  // the segments are recomputed into
  uint32_t *pool = cv.take<uint32_t>(0);
  const uint64_t stage_words = sp.traceback ? (uint64_t)M + N + 1 : 0;
  if (cv.used + stage_words * 4 > c->ws_bytes) {
    set_error("checkpointed traceback needs %llu workspace bytes; the context has %zu",
              (unsigned long long)(cv.used + stage_words * 4), c->ws_bytes);
    return FILTR_ERR_NOMEM;
  }
  const uint64_t pool_words = (c->ws_bytes - cv.used) / 4 - stage_words;
  uint32_t *d_stage = pool + pool_words;
  // host staging: the one-pair batch, the segment descriptors, the flags
  const size_t desc_off = 4096;
  const size_t flags_off = desc_off + (size_t)(2 * nseg + 1) * sizeof(XdCkpt);
  if (!c->ensure_host(flags_off + (size_t)(nseg + 1) * 4 + 64)) return FILTR_ERR_NOMEM;
  char *h = reinterpret_cast<char *>(c->h_stage);
  uint32_t one[16] = {0, M, N};  // order, q_len, r_len
  TbLayout L{};
  uint64_t misc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  memcpy(h, one, sizeof one);
  memcpy(h + 64, &L, sizeof L);
  memcpy(h + 128, misc, sizeof misc);
  XdCkpt *hk = reinterpret_cast<XdCkpt *>(h + desc_off);
  for (int64_t sgi = 0; sgi < nseg; ++sgi)
    hk[sgi] = XdCkpt{3, C, ck_buf, (int)(sgi * C), (int)std::min<int64_t>((sgi + 1) * C, K), nullptr, nullptr,
                     d_flags};
  cudaError_t e = cudaMemcpyAsync(d_one, h, sizeof one, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_tbl, h + 64, sizeof L, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_misc, h + 128, sizeof misc, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(d_ck, hk, nseg * sizeof(XdCkpt), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_flags, 0, (nseg + 1) * 4, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(d_ovf, 0, 16, st);
  if (e != cudaSuccess) return cuda_fail(e, "checkpoint setup");
  const uint64_t *d_off = d_misc + 1;
  BatchDev b{q, r, d_off, d_off + 1, d_one + 1, d_one + 2};
  FullArgs fa;
  fa.b = b;
  fa.sp = sp;
  fa.sp.traceback = 0;  // the forward sweep keeps checkpoints only
  fa.order = d_one;
  fa.n_order = 1;
  fa.counter = nullptr;  // unused with checkpoints
  fa.out = out;
  fa.fwd = d_fwd;
  fa.tb = nullptr;
  fa.tbl = d_tbl;
  fa.strip_buf = nullptr;
  fa.strip_stride = 0;
  fa.max_n = 0;
  fa.max_m = 0;
  fa.x16_rebase = c->xd16_mode == 2 ? 0 : X16_REBASE;
  // forward: every segment is offered to each width in turn; the narrowest
  // window that holds it does the work, the other launches return at once
  uint32_t launches = 0;
  c->span_begin(Ctx::PH_FORWARD, st);
  for (int64_t sgi = 0; sgi < nseg && e == cudaSuccess; ++sgi) {
    fa.ck = d_ck + sgi;
    for (int W : kLadder) {
      e = launch_xdrop(fa, W, 1, d_ovf, d_ovf + 1, st);
      ++launches;
      if (e != cudaSuccess) break;
    }
  }
  c->span_end(st);
  FwdOut *hf = reinterpret_cast<FwdOut *>(h + 256);
  int32_t *hflags = reinterpret_cast<int32_t *>(h + flags_off);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hf, d_fwd, sizeof(FwdOut), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hflags, d_flags, (nseg + 1) * 4, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "checkpointed forward sweep");
  const FwdOut f = *hf;
  c->last_launches = launches;
  c->last_strip_rows = 0;
  if (hflags[0] == 3) {  // the packed sweep left its 16-bit range: the whole pair in int32
    ScoreParams s32 = sp;
    s32.xd16 = 0;
    const filtr_status rc = run_xdrop_ckpt(c, s32, params, q, M, r, N, out, cigar, cap, st, C);
    c->last_xd16 = 1;
    c->last_xd16_rerun = 1;
    return rc;
  }
  c->last_xd16 = sp.xd16 ? 1u : 0u;
  c->last_xd16_rerun = 0;
  if (!sp.traceback || (f.status != FILTR_ST_OK && f.status != FILTR_ST_DROPPED)) return FILTR_OK;
  // The forward sweep is one chain, each antidiagonal waiting for the last; the
  // segments of the path, given their checkpoints, are not.  So the forward goes
  // without traceback (a megabase pair: 475 ms instead of 579), and the segments are
  // recomputed with it side by side, a launch per width, and walked: all at once
  // where the pool holds them, else in groups, from the path's end backwards.
  const int64_t ke = (int64_t)f.end_i + f.end_j, n_path = (ke + C - 1) / C;
  XdCkpt *by_width = hk + nseg;
  struct SegGroup {  // segments [s0, s1)
    int64_t s0, s1;
    int64_t first[7];       // its descriptors of each width
    const int32_t *ck;      // origins of its antidiagonals
  };
  std::vector<SegGroup> groups;
  int64_t nb = 0;
  for (int64_t s1 = n_path; s1 > 0;) {
    int64_t s0 = s1;
    uint64_t words = 0;  // rows
    for (; s0 > 0 && !(c->ckpt_recompute && s0 < s1); --s0) {
      const int W = hflags[s0];  // of segment s0 - 1
      if (W <= 0) {
        set_error("checkpointed sweep: segment %lld has no width", (long long)s0 - 1);
        return FILTR_ERR_CUDA;
      }
      const uint64_t w = (uint64_t)C * xd_words_per_k(W, 8);
      if (words + w + (uint64_t)(s1 - s0 + 1) * C > pool_words) break;
      words += w;
    }
    if (s0 == s1) {
      set_error("checkpointed traceback: the workspace of %zu bytes does not hold one segment", c->ws_bytes);
      return FILTR_ERR_NOMEM;
    }
    SegGroup g{s0, s1, {}, reinterpret_cast<int32_t *>(pool + words)};
    uint64_t at = 0;
    for (int64_t s = s0; s < s1; ++s) {
      hk[s] = XdCkpt{2, C, ck_buf, (int)(s * C), (int)std::min<int64_t>((s + 1) * C, ke), pool + at,
                     reinterpret_cast<int32_t *>(pool + words) + (s - s0) * C, d_flags};
      at += (uint64_t)C * xd_words_per_k(hflags[1 + s], 8);
    }
    for (int wi = 0; wi < 6; ++wi) {
      g.first[wi] = nb;
      for (int64_t s = s0; s < s1; ++s)
        if (hflags[1 + s] == kLadder[wi]) by_width[nb++] = hk[s];
    }
    g.first[6] = nb;
    groups.push_back(g);
    s1 = s0;
  }
  if (groups.empty()) groups.push_back(SegGroup{0, 0, {}, nullptr});  // the path is the origin alone
  WalkState *hw = reinterpret_cast<WalkState *>(h + 512);
  *hw = WalkState{f.end_i, f.end_j, f.score, 0, 0, -1, 0, 0};
  e = cudaMemcpyAsync(d_ws, hw, sizeof(WalkState), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && nb)
    e = cudaMemcpyAsync(d_ck, hk, (nseg + nb) * sizeof(XdCkpt), cudaMemcpyHostToDevice, st);
  FullArgs ra = fa;
  ra.sp = sp;  // traceback on
  ra.out = reinterpret_cast<filtr_result *>(c->d_small + 3072);  // mode 2 writes no result
  WalkArgs wa;
  wa.b = b;
  wa.sp = sp;
  wa.order = d_one;
  wa.n_order = 1;
  wa.out = out;
  wa.fwd = d_fwd;
  wa.tb = nullptr;
  wa.tbl = d_tbl;
  wa.stage = d_stage;
  wa.stage_off = d_misc;
  for (const SegGroup &g : groups) {
    c->span_begin(Ctx::PH_FORWARD, st);
    for (int wi = 5; wi >= 0 && e == cudaSuccess; --wi) {
      if (g.first[wi + 1] == g.first[wi]) continue;
      ra.ck = d_ck + nseg + g.first[wi];
      ra.n_ck = (uint32_t)(g.first[wi + 1] - g.first[wi]);
      const int per = xd_pairs_per_cta(kLadder[wi], ra.sp);
      e = launch_xdrop(ra, kLadder[wi], (int)((ra.n_ck + per - 1) / per), d_ovf, d_ovf + 1, st);
      ++launches;
    }
    c->span_end(st);
    c->span_begin(Ctx::PH_WALK, st);
    if (e == cudaSuccess) e = launch_walk_segments(wa, d_ck, d_flags + 1, g.ck, C, (int)(g.s0 * C), d_ws, st);
    ++launches;
    c->span_end(st);
    if (e != cudaSuccess) return cuda_fail(e, "recomputing and walking segments");
  }
  uint64_t *d_offs = d_misc + 4;
  e = cudaMemsetAsync(d_offs, 0, 8, st);
  if (e == cudaSuccess) e = launch_compact(wa, 1, d_offs, cigar, cap, out, st);
  filtr_result *hr = reinterpret_cast<filtr_result *>(h + 1024);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hr, out, sizeof(filtr_result), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "checkpointed traceback");
  c->last_launches = launches + 1;
  c->last_waves = (int)groups.size();
  if (hr->cigar_len > cap) {
    set_error("the CIGAR needs %u ops, cigar_cap is %llu", hr->cigar_len, (unsigned long long)cap);
    return FILTR_ERR_CIGAR_CAP;
  }
  return FILTR_OK;
}

}  // namespace

// One long full-matrix / banded pair on the whole GPU without waiting for it
// (the serving loop's path for large requests).
filtr_status long_pair_async(Ctx *c, const ScoreParams &sp, const filtr_params *params,
                             const uint8_t *q, uint32_t M, const uint8_t *r, uint32_t N,
                             filtr_result *out, uint32_t *cigar, uint64_t cap, cudaStream_t st) {
  if (c->done_ev) cudaEventSynchronize(c->done_ev);
  c->ev_used = 0;
  c->spans.clear();
  const filtr_status rc =
      run_long(c, sp, q, M, r, N, out, cigar, cap, st, 0, SPLIT_TIMEOUT_NS, false);
  if (!c->done_ev) cudaEventCreateWithFlags(&c->done_ev, cudaEventDisableTiming);
  if (c->done_ev) cudaEventRecord(c->done_ev, st);
  return rc;
}

}  // namespace filtr

using namespace filtr;

extern "C" {

filtr_status filtr_align_long(filtr_ctx *ctx, const filtr_params *params, const uint8_t *q,
                              uint32_t M, const uint8_t *r, uint32_t N, filtr_result *out,
                              uint32_t *cigar, uint64_t cigar_cap, void *stream) {
  ScoreParams sp;
  filtr_status rc = to_score_params(params, &sp);
  if (rc != FILTR_OK) return rc;
  if (sp.mid) {
    set_error("filtr_align_long: the M/I/D form runs only in filtr_align_batch");
    return FILTR_ERR_UNSUPPORTED;
  }
  if (!ctx || !out || (M && !q) || (N && !r) || (sp.traceback && cigar_cap && !cigar)) {
    set_error("filtr_align_long: NULL argument");
    return FILTR_ERR_INVALID;
  }
  if (M >= (1u << 30) || N >= (1u << 30)) {
    set_error("sequence longer than 2^30");
    return FILTR_ERR_UNSUPPORTED;
  }
  Ctx *c = reinterpret_cast<Ctx *>(ctx);
  cudaStream_t st = (cudaStream_t)stream;
  cudaSetDevice(c->device);
  if (c->done_ev) cudaEventSynchronize(c->done_ev);
  c->ev_used = 0;
  c->spans.clear();
  if (!score_range_ok(sp, M, N)) {
    set_error("scores could exceed 2^28 (2^26 for local alignments) for these lengths and penalties");
    return FILTR_ERR_UNSUPPORTED;
  }
  rc = validate_seq(c, q, M, r, N, sp.alphabet, st);
  if (rc != FILTR_OK) return rc;
  sp.xd16 = (c->xd16_mode != 1 && xd16_eligible(sp)) ? 1 : 0;
  if (sp.use_xdrop && M && N &&
      (c->ckpt_interval > 0 || (int64_t)M + N > XD_SEGMENTED_SWEEP ||
       4 * xd_tb_words(M, N, 32, 8) > c->ws_bytes / 2)) {  // the widest traceback would not fit
    const int C = c->ckpt_interval > 0 ? c->ckpt_interval : 4096;
    rc = run_xdrop_ckpt(c, sp, params, q, M, r, N, out, cigar, cigar_cap, st, C);
    if (!c->done_ev) cudaEventCreateWithFlags(&c->done_ev, cudaEventDisableTiming);
    if (c->done_ev) cudaEventRecord(c->done_ev, st);
    return rc;
  }
  if (sp.use_xdrop || M == 0 || N == 0 || (uint64_t)M * N < (1ull << 22) || M <= 512) {
    // a one-pair batch: lengths and offsets from the small device buffer
    uint64_t *d_off = reinterpret_cast<uint64_t *>(c->d_small + 1024);
    uint32_t *d_len = reinterpret_cast<uint32_t *>(c->d_small + 1088);
    if (!c->ensure_host(4096)) return FILTR_ERR_NOMEM;
    char *h = reinterpret_cast<char *>(c->h_stage);
    uint64_t offs[2] = {0, 0};
    uint32_t lens[2] = {M, N};
    memcpy(h + 2048, offs, sizeof offs);
    memcpy(h + 2112, lens, sizeof lens);
    cudaError_t e = cudaMemcpyAsync(d_off, h + 2048, sizeof offs, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_len, h + 2112, sizeof lens, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the staging is reused by the batch call
    if (e != cudaSuccess) return cuda_fail(e, "one-pair setup");
    BatchDev b{q ? q : reinterpret_cast<const uint8_t *>(c->d_small),
               r ? r : reinterpret_cast<const uint8_t *>(c->d_small), d_off, d_off + 1, d_len, d_len + 1};
    const int w0 = c->xdrop_warps0;
    c->xdrop_warps0 = 4;
    rc = align_batch_impl(c, params, 1, b, out, cigar, cigar_cap, st, false, lens, lens + 1, true);
    c->xdrop_warps0 = w0;
    return rc;
  }
  rc = run_long(c, sp, q, M, r, N, out, cigar, cigar_cap, st, 0, SPLIT_TIMEOUT_NS);
  if (!c->done_ev) cudaEventCreateWithFlags(&c->done_ev, cudaEventDisableTiming);
  if (c->done_ev) cudaEventRecord(c->done_ev, st);
  return rc;
}

filtr_status filtr_test_set_checkpoint(filtr_ctx *ctx, int32_t interval) {
  if (!ctx || interval < 0) {
    set_error("filtr_test_set_checkpoint: bad arguments");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->ckpt_interval = interval;
  return FILTR_OK;
}

filtr_status filtr_test_set_first_width(filtr_ctx *ctx, int32_t warps) {
  if (!ctx || (warps != 0 && warps != 1 && warps != 2 && warps != 4 && warps != 8 && warps != 16 &&
               warps != 32)) {
    set_error("filtr_test_set_first_width: bad arguments");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->xdrop_warps0 = warps;
  return FILTR_OK;
}

filtr_status filtr_test_set_device_plan(filtr_ctx *ctx, int32_t mode) {
  if (!ctx || mode < 0 || mode > 2) {
    set_error("filtr_test_set_device_plan: bad arguments");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->dev_plan_mode = mode;
  return FILTR_OK;
}

filtr_status filtr_test_set_split(filtr_ctx *ctx, int32_t mode) {
  if (!ctx || mode < 0 || mode > 2) {
    set_error("filtr_test_set_split: bad arguments");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->split_mode = mode;
  return FILTR_OK;
}

filtr_status filtr_test_set_strip_wait(filtr_ctx *ctx, int32_t withhold, uint64_t timeout_ns) {
  if (!ctx) {
    set_error("filtr_test_set_strip_wait: ctx is NULL");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->strip_withhold = withhold != 0;
  reinterpret_cast<Ctx *>(ctx)->strip_timeout_ns = timeout_ns;
  return FILTR_OK;
}

filtr_status filtr_test_last_strip_rows(filtr_ctx *ctx, int32_t *rows) {
  if (!ctx || !rows) {
    set_error("filtr_test_last_strip_rows: NULL argument");
    return FILTR_ERR_INVALID;
  }
  *rows = reinterpret_cast<Ctx *>(ctx)->last_strip_rows;
  return FILTR_OK;
}

filtr_status filtr_test_set_packed_sweep(filtr_ctx *ctx, int32_t mode) {
  if (!ctx || mode < 0 || mode > 2) {
    set_error("filtr_test_set_packed_sweep: bad arguments");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->xd16_mode = mode;
  return FILTR_OK;
}

filtr_status filtr_test_force_recompute(filtr_ctx *ctx, int32_t on) {
  if (!ctx) {
    set_error("filtr_test_force_recompute: ctx is NULL");
    return FILTR_ERR_INVALID;
  }
  reinterpret_cast<Ctx *>(ctx)->ckpt_recompute = on != 0;
  return FILTR_OK;
}

filtr_status filtr_test_long_timeout(filtr_ctx *ctx, const filtr_params *params, const uint8_t *q,
                                     uint32_t M, const uint8_t *r, uint32_t N,
                                     uint64_t timeout_ns) {
  ScoreParams sp;
  filtr_status rc = to_score_params(params, &sp);
  if (rc != FILTR_OK) return rc;
  if (!ctx || !q || !r || M <= 512 || N == 0) {
    set_error("filtr_test_long_timeout: needs M > 512 and device sequences");
    return FILTR_ERR_INVALID;
  }
  Ctx *c = reinterpret_cast<Ctx *>(ctx);
  cudaSetDevice(c->device);
  if (c->done_ev) cudaEventSynchronize(c->done_ev);
  sp.traceback = 0;
  filtr_result *d_out = reinterpret_cast<filtr_result *>(c->d_small + 2048);
  rc = run_long(c, sp, q, M, r, N, d_out, nullptr, 0, c->own_stream, 1, timeout_ns);
  return rc;
}

}  // extern "C"
