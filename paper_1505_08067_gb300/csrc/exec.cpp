// See exec.h.
#include "exec.h"

#include "umma_stage.h"

#include <algorithm>

namespace gbfft {

// Blocks of a line launch: tiles of 2^tile_log elements.
static int lines_grid(const PassDesc& d, int tile_log) {
  const int64_t outer = d.tiles_inner > 0 ? d.tiles / d.tiles_inner : 0;
  const int64_t n = (outer * d.count_inner) << d.logL, tile = int64_t(1) << tile_log;
  return (int)std::min<int64_t>((n + tile - 1) >> tile_log, 0x7fffffff);
}

cudaError_t bind_launches(const PlanSpec& s, const Caps& caps, const cf* tables, int* status,
                          PassLaunch* launches) {
  for (int i = 0; i < s.passes.size(); ++i) {
    const PassSpec& p = s.passes[i];
    PassLaunch l{};
    if (p.kind == PASS_TRANSPOSE) l.grid = caps.sm_count;  // SMs: the transpose sizes its grid
    if (p.kind == PASS_FFT) {
      l.d = pass_desc(p, 0, s.batch, s.batch);
      l.d.tw = tables;
      l.d.epi_hi = (p.epi == 1 || p.epi == 2) ? tables + p.epi_hi_off : nullptr;
      l.d.epi_lo = (p.epi == 1 || p.epi == 2) ? tables + p.epi_lo_off : nullptr;
      l.d.status = status;
      l.d.h = p.conv ? static_cast<const cf*>(s.filter[p.h_dim]) : nullptr;
      l.R = p.R;
      l.lmap = p.lmap;
      l.smap = p.smap;
      l.grid = p.grid;
      l.block = p.block;
      l.smem = p.smem;
      if (p.tc_prec) {
        l.fn = resolve_tc_pass(p.logL, p.tc_prec, p.variant, p.io16);
        if (!l.fn) return cudaErrorInvalidDeviceFunction;
        l.specialised = true;
      } else {
        l.fn = resolve_kernel(l.R, l.lmap, l.smap, l.d, s.generic_only, &l.specialised);
        const bool rows = p.lmap == MAP_ROWS;
        if (p.line_off >= 0 &&
            (p.conv ? (rows ? resolve_conv_lines(p.logL, &l) : resolve_conv_cols(p.logL, &l))
                    : (rows ? resolve_lines(p.logL, &l) : resolve_cols(p.logL, &l))))
          l.grid = lines_grid(l.d, l.lines);
      }
      cudaError_t e = prepare_launch(l);
      if (e != cudaSuccess) return e;
      if (p.tc_prec) {
        // persistent grid: the DFT-matrix fragments a block builds once serve
        // many tiles
        int per_sm = 0;
        e = occupancy(l, &per_sm);
        if (e != cudaSuccess) return e;
        if (p.variant != 1) {
          // the occupancy query reports one block per SM for this kernel
          // where its registers and shared memory allow more (measured):
          // count from the kernel's attributes, within the SM's tensor memory
          int own = 0;
          e = resident_blocks(l.fn, l.block, l.smem, umma_tmem_cols(p.logL), &own);
          if (e != cudaSuccess) return e;
          per_sm = std::max(per_sm, own);
        }
        l.ctas_per_sm = per_sm;
        const int64_t g = (int64_t)std::max(per_sm, 1) * caps.sm_count;
        l.grid = (int)std::min<int64_t>(g, l.grid);
        l.persistent_grid = l.grid;
        launches[i] = l;
        continue;
      }
      // the library's choice for contiguous FP32 transforms of 2^12 is the
      // register kernel (0.320 against 0.335 ms per 2^27 elements for the
      // staged one, the choice the autotuner makes in every measured run);
      // variant 2 still asks for the staged kernel
      const bool reg4096 = p.variant == 0 && !p.conv && !p.tc_prec && p.logL == 12 &&
                           p.lmap == MAP_ROWS && p.smap == MAP_ROWS;
      const bool want_staged =
          ((p.variant == 0 && !reg4096) || p.variant == 2 || p.variant == 4) && !l.lines;
      l.has_staged = want_staged && resolve_staged(l.d, l.lmap, l.smap, s.generic_only, &l.staged);
      l.staged.tmap = p.variant != 4;
      if (l.has_staged) {
        e = prepare_staged(l.staged, l.d.tiles, caps.sm_count);
        if (e != cudaSuccess) return e;
      }
      if (p.variant == 3 && l.specialised) {
        int per_sm = 0;
        e = occupancy(l, &per_sm);
        if (e != cudaSuccess) return e;
        const int64_t g = (int64_t)std::max(per_sm, 1) * caps.sm_count;
        l.grid = (int)std::min<int64_t>(g, l.grid);
        l.persistent_grid = l.grid;
        l.d.l2_prefetch = 1;
      }
    }
    launches[i] = l;
  }
  if (s.tc_cols) {
    // the column forms of the two row passes (pass 1 and 3 of the five)
    const int n = s.passes.size(), logN = s.passes[1].logL + s.passes[3].logL;
    for (int h = 0; h < 2; ++h) {
      const PassSpec& p = s.passes[1 + 2 * h];
      PassLaunch l = launches[1 + 2 * h];
      l.fn = h ? resolve_umma_cols2(p.logL, p.tc_prec, p.io16)
               : resolve_umma_cols1(p.logL, p.tc_prec, p.io16);
      if (!l.fn) return cudaErrorInvalidDeviceFunction;
      cudaError_t e = prepare_launch(l);
      if (e != cudaSuccess) return e;
      int per_sm = 0;
      e = resident_blocks(l.fn, l.block, l.smem, umma_tmem_cols(p.logL), &per_sm);
      if (e != cudaSuccess) return e;
      l.ctas_per_sm = per_sm;
      l.persistent_grid = std::max(per_sm, 1) * caps.sm_count;
      l.d.epi_logN = logN;
      if (tc_columns_fused(p.tc_prec, p.io16)) {  // else both passes swap, as in the six steps
        l.d.conj_in = h == 0 && s.direction == FFT_INVERSE;
        l.d.conj_out = h == 1 && s.direction == FFT_INVERSE;
      }
      launches[n + h] = l;
    }
  }
  return cudaSuccess;
}

// The two column launches of a six-step plan for nb transforms, with the
// twiddle transpose between them where the first does not multiply.
static cudaError_t enqueue_tc_cols(const PlanSpec& s, const PassLaunch* launches, const void* in,
                                   void* out, void* work, void* work2, int64_t nb,
                                   cudaStream_t st) {
  const bool fused = tc_columns_fused(s.passes[1].tc_prec, s.passes[1].io16);
  for (int h = 0; h < 2; ++h) {
    if (h && !fused) {
      const PassSpec& t = s.passes[2];
      const cudaError_t e = launch_transpose(work, work2, nb, t.tr_rows, t.tr_cols, t.tr_logN,
                                             t.tr_sign, t.io16, launches[2].grid, st);
      if (e != cudaSuccess) return e;
    }
    PassLaunch l = launches[s.passes.size() + h];
    const PassSpec& p = s.passes[1 + 2 * h];
    const int logN = l.d.epi_logN, le = logN - p.logL;
    l.d.tiles = nb << (logN - 12);  // tiles of 4096 elements
    l.d.count_inner = nb << le;
    l.grid = (int)std::min<int64_t>(l.persistent_grid, l.d.tiles);
    if (h == 0)
      encode_tc_cols_map(l.d, in, nb << p.logL, le, elem_bytes(s.precision), 1 << (12 - p.logL),
                         std::min(1 << p.logL, 256));
    const cudaError_t e = launch_pass(l, !h ? in : fused ? work : work2, h ? out : work, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t bind_joined(const PlanSpec& s, const Caps& caps, const cf* tables, int* status,
                        unsigned* counters, JoinedLaunch* j) {
  const int l0 = s.passes[0].logL, l1 = s.passes[1].logL;
  const bool inv = s.direction == FFT_INVERSE;
  const cudaError_t e = s.dims == 2 ? prepare_joined_frames(l1, l0, s.join_tile_log, inv,
                                                            caps.sm_count, j)
                                    : prepare_joined(l0 + l1, s.join_apart, inv,
                                                     caps.sm_count, j);
  if (e != cudaSuccess) return e;
  j->d.tw1 = tables + s.join_tw1;
  j->d.tw2 = tables + s.join_tw2;
  j->d.o.lag = s.join_lag;
  j->d.o.ring = s.join_ring;
  j->d.ctr = counters;
  j->d.status = status;
  j->d.polls = kJoinPolls;
  return cudaSuccess;
}

cudaError_t enqueue_tables(const PlanSpec& s, cf* tables, cudaStream_t st) {
  TwiddleList list{};
  static_assert(decltype(s.tables)::capacity() <= 40, "every table fits the list");
  for (const TwSegment& t : s.tables)
    list.t[list.n++] = TwiddleTable{t.off, t.count, t.den, t.mult, t.mode, t.r};
  return launch_twiddle_list(tables, list, st);
}

static cudaError_t enqueue_range(const PlanSpec& s, const PassLaunch* launches, const void* in,
                                 void* out, void* work, int64_t b0, int64_t nb, cudaStream_t st,
                                 int64_t work2_off, const JoinedLaunch* joined);

cudaError_t enqueue_passes(const PlanSpec& s, const PassLaunch* launches, const void* in,
                           void* out, void* work, int64_t b0, int64_t nb, cudaStream_t st,
                           int64_t work2_off, const JoinedLaunch* joined) {
  if (work2_off < 0) work2_off = s.work2_off;
  if (nb <= 0) return cudaSuccess;
  if (s.chunk_batch <= 0 || nb <= s.chunk_batch)
    return enqueue_range(s, launches, in, out, work, b0, nb, st, work2_off, joined);
  // sub-batches in stream order, each reusing the workspace from its start
  const int64_t E = s.dims == 1 ? s.n[0] : s.n[0] * s.n[1];
  const int64_t eb = elem_bytes(s.precision);
  for (int64_t c = 0; c < nb; c += s.chunk_batch) {
    const int64_t n = std::min(s.chunk_batch, nb - c);
    cudaError_t e = enqueue_range(s, launches, static_cast<const char*>(in) + c * E * eb,
                                  static_cast<char*>(out) + c * E * eb, work, b0 + c, n, st,
                                  work2_off, joined);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

static cudaError_t enqueue_range(const PlanSpec& s, const PassLaunch* launches, const void* in,
                                 void* out, void* work, int64_t b0, int64_t nb, cudaStream_t st,
                                 int64_t work2_off, const JoinedLaunch* joined) {
  if (nb <= 0) return cudaSuccess;
  const int64_t E = s.dims == 1 ? s.n[0] : s.n[0] * s.n[1];
  if (joined && joined->fn && (work || joined->frames)) {
    // the output of one transform is written while the input of a later one is
    // still read: in place or apart, not partly overlapping
    const uintptr_t a = (uintptr_t)in, b = (uintptr_t)out, bytes = (uintptr_t)(nb * E) * 8;
    if (joined->second || a == b || a + bytes <= b || b + bytes <= a)
      return launch_joined(*joined, nb, in, out, work, st);
  }
  // the second workspace buffer of six-step plans
  void* work2 = work ? static_cast<char*>(work) + work2_off * elem_bytes(s.precision) : nullptr;
  if (s.tc_cols && work) return enqueue_tc_cols(s, launches, in, out, work, work2, nb, st);
  auto buf = [&](int b) -> void* {
    return b == BUF_IN ? const_cast<void*>(in) : b == BUF_OUT ? out : b == BUF_WORK2 ? work2 : work;
  };
  for (int i = 0; i < s.passes.size(); ++i) {
    const PassSpec& p = s.passes[i];
    const void* src = buf(p.src);
    void* dst = buf(p.dst);
    cudaError_t e;
    if (p.kind == PASS_COPY) {
      e = launch_copy(src, dst, nb * E, 1, 1, st);
    } else if (p.kind == PASS_TRANSPOSE) {
      e = launch_transpose(src, dst, nb, p.tr_rows, p.tr_cols, p.tr_logN, p.tr_sign, p.io16,
                           launches[i].grid, st);
    } else {
      PassLaunch l = launches[i];
      if (b0 != 0 || nb != s.batch) {
        PassDesc d = pass_desc(p, b0, nb, s.batch);
        d.tw = l.d.tw;
        d.epi_hi = l.d.epi_hi;
        d.epi_lo = l.d.epi_lo;
        d.status = l.d.status;
        d.h = l.d.h;
        l.d = d;
        if (!l.lines)
          l.fn = p.tc_prec ? resolve_tc_pass(p.logL, p.tc_prec, p.variant, p.io16)
                         : resolve_kernel(l.R, l.lmap, l.smap, l.d, s.generic_only, &l.specialised);
        e = prepare_launch(l);
        if (e != cudaSuccess) return e;
        d.l2_prefetch = launches[i].d.l2_prefetch;
        l.d.l2_prefetch = d.l2_prefetch;
        l.grid = l.lines ? lines_grid(d, l.lines)
                         : (int)std::min<int64_t>(d.tiles, l.persistent_grid ? l.persistent_grid
                                                                              : 0x7fffffff);
      }
      if (l.d.tiles == 0) continue;
      if (l.has_staged && ((uintptr_t)src & 15) == 0) {
        StagedLaunch sl = l.staged;
        sl.grid = (int)std::min<int64_t>(sl.max_grid > 0 ? sl.max_grid : sl.grid, l.d.tiles);
        e = launch_staged(sl, l.d, src, dst, st);
      } else {
        e = launch_pass(l, src, dst, st);
      }
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gbfft
