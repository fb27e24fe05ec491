// Test infrastructure: replays the joined two-pass kernel (fft_join.h) on the
// CPU, tile by tile in ticket order and thread by thread, with every access
// checked: global and workspace offsets inside their buffers, shared slots
// inside the tile and written in the phase before they are read, no slot
// written twice in a phase, every output written once, workspace elements read
// only after the transform's own first pass wrote them.  Also checks the tile
// order: what a ticket waits for is complete once the tickets before it are.
// It never stands in for the GPU.
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "fft_join.h"

using namespace gbfft;

namespace {

struct Ctx {
  const cf *in, *tw1, *tw2, *h;
  int64_t h_len;
  cf *out, *work;
  int64_t in_len, out_len, work_len;
  std::vector<uint8_t> out_hits;
  std::vector<int64_t> work_owner;  // transform whose first pass wrote the element
  int64_t b;                        // transform being replayed
  int tw1_len, tw2_len;
  const cf* sm;
  int smem_len, conflicts;
  std::vector<int64_t> phase_of;
  int64_t phase, errors;
  std::string first;
};
Ctx g;

void err(const char* what, int64_t i) {
  if (g.errors++ == 0) {
    char b[160];
    snprintf(b, sizeof b, "%s (index %lld)", what, (long long)i);
    g.first = b;
  }
}

struct CheckMem {
  static cf ldin(const cf* p, int off) {
    const int64_t i = p - g.in + off;
    if (i < 0 || i >= g.in_len) { err("input load out of bounds", i); return mk(0, 0); }
    return g.in[i];
  }
  static cf ldw(const cf* p, int off) {
    const int64_t i = p - g.work + off;
    if (i < 0 || i >= g.work_len) { err("workspace load out of bounds", i); return mk(0, 0); }
    if (g.work_owner[i] != g.b) err("workspace element of another transform", i);
    return g.work[i];
  }
  static void stw(cf* p, int off, cf v) {
    const int64_t i = p - g.work + off;
    if (i < 0 || i >= g.work_len) { err("workspace store out of bounds", i); return; }
    if (g.work_owner[i] == g.b) err("workspace element written twice", i);
    g.work_owner[i] = g.b;
    g.work[i] = v;
  }
  static void stout(cf* p, int off, cf v) {
    const int64_t i = p - g.out + off;
    if (i < 0 || i >= g.out_len) { err("output store out of bounds", i); return; }
    if (g.out_hits[i]++) err("output element written twice", i);
    g.out[i] = v;
  }
  static int at(const cf* s, int i) {
    i += (int)(s - g.sm);
    if (i < 0 || i >= g.smem_len) { err("shared slot out of bounds", i); return 0; }
    return i;
  }
  static cf lds(const cf* s, int i) {
    i = at(s, i);
    if (g.phase_of[i] != g.phase) err("shared slot read that the last phase did not write", i);
    return g.sm[i];
  }
  static void sts(cf* s, int i, cf v) {
    i = at(s, i);
    if (g.phase_of[i] == g.phase) err("shared slot written twice in a phase", i);
    g.phase_of[i] = g.phase;
    const_cast<cf*>(g.sm)[i] = v;
  }
  static cf ldtw(const cf* p) {
    const bool one = p >= g.tw1 && p < g.tw1 + g.tw1_len, two = p >= g.tw2 && p < g.tw2 + g.tw2_len;
    if (p >= g.h && p < g.h + g.h_len) return *p;
    if (!one && !two) { err("twiddle load out of bounds", 0); return mk(1, 0); }
    return *p;
  }
  static cf rotor(int64_t m, int logN) {
    if (m < 0 || m >= int64_t(1) << logN) err("rotor exponent out of range", m);
    const double a = -2.0 * M_PI * (double)m / (double)(int64_t(1) << logN);
    return mk((float)cos(a), (float)sin(a));
  }
};

std::vector<cf> roots(int n) {
  std::vector<cf> t(n);
  for (int j = 0; j < n; ++j) t[j] = mk((float)cos(2 * M_PI * j / n), (float)-sin(2 * M_PI * j / n));
  return t;
}

template <class SH, int KIND, class First, class Store>
void tile(cf* sm, cf* st, const cf* tw, int col0, int logN, First first, Store store) {
  using B = JoinBody<SH, KIND, CheckMem>;
  std::vector<cf> regs((size_t)SH::kThreads * kJoinR);
  auto v = [&](int t) -> cf (&)[kJoinR] { return *reinterpret_cast<cf(*)[kJoinR]>(&regs[(size_t)t * kJoinR]); };
  auto each = [&](auto f) { for (int t = 0; t < SH::kThreads; ++t) f(v(t), t); };
  ++g.phase;
  if (KIND == JOIN_FIRST)
    for (int lane = 0; lane < 32; ++lane) B::steps(st, col0, logN, lane);
  each([&](cf (&r)[kJoinR], int t) { first(r, t); B::dft0(r); B::template put<0>(r, sm, t); });
  if constexpr (SH::kNst == 3) {  // rows and columns of frames: no steps to keep
    each([&](cf (&r)[kJoinR], int t) { B::template get<1>(r, sm, t); B::template turn<1, false>(r, tw, 0, 0, t); });
    ++g.phase;
    each([&](cf (&r)[kJoinR], int t) { B::template put<1>(r, sm, t); });
  }
  each([&](cf (&r)[kJoinR], int t) {
    B::template get<SH::kLast>(r, sm, t);
    B::template turn<SH::kLast, KIND == JOIN_FIRST>(r, tw, col0, logN, t);  // pass 1 carries the four-step twiddle
    store(r, t);
  });
}

template <int LOGN, int TL, bool INV>
int64_t run(int64_t nb, int64_t lag, int ring, const cf* in, cf* out) {
  using PR = JoinPair<LOGN, TL>;
  using B1 = JoinBody<typename PR::P1, JOIN_FIRST, CheckMem>;
  using B2 = JoinBody<typename PR::P2, JOIN_COLS, CheckMem>;
  g = Ctx{};
  std::vector<cf> t1 = roots(PR::kN1), t2 = roots(PR::kN2), work((size_t)ring * PR::kN),
                  sm(std::max(B1::kSlots, B2::kSlots) + PR::kSteps);
  g.in = in;
  g.out = out;
  g.in_len = g.out_len = nb * PR::kN;
  g.work = work.data();
  g.work_len = (int64_t)work.size();
  g.out_hits.assign(g.out_len, 0);
  g.work_owner.assign(g.work_len, -1);
  g.tw1 = t1.data();
  g.tw2 = t2.data();
  g.tw1_len = PR::kN1;
  g.tw2_len = PR::kN2;
  g.sm = sm.data();
  g.smem_len = (int)sm.size();
  g.phase_of.assign(sm.size(), -1);
  cf* st = sm.data() + std::max(B1::kSlots, B2::kSlots);
  JoinOrder o{nb, LOGN - PR::kTileLog, ring, std::min<int64_t>(lag, nb * PR::kTiles)};
  std::vector<uint32_t> done(2 * ring, 0);
  for (int64_t t = 0; t < join_tickets(o); ++t) {
    const JoinTicket k = join_ticket(o, t);
    const JoinDep dep = join_dep(o, k);
    if (k.b < 0 || k.b >= nb || k.tile < 0 || k.tile >= PR::kTiles) { err("ticket out of range", t); break; }
    if (done[dep.pass * ring + dep.slot] < dep.count) err("a ticket waits for a later one", t);
    const int slot = (int)(k.b % ring);
    cf* w = work.data() + (int64_t)slot * PR::kN;
    g.b = k.b;
    if (k.pass == 0) {
      const int col0 = k.tile * PR::kG1;
      tile<typename PR::P1, JOIN_FIRST>(
          sm.data(), st, g.tw1, col0, LOGN,
          [&](cf (&v)[kJoinR], int i) { B1::template first<INV, false>(v, in + k.b * PR::kN + col0, PR::kN2, i); },
          [&](cf (&v)[kJoinR], int i) { B1::template store_block<PR::kG2>(v, w + col0 * PR::kG2, st, PR::kN2, i); });
    } else {
      tile<typename PR::P2, JOIN_COLS>(
          sm.data(), st, g.tw2, 0, 0,
          [&](cf (&v)[kJoinR], int i) { B2::template first<false, true>(v, w + k.tile * PR::kTile, PR::kG2, i); },
          [&](cf (&v)[kJoinR], int i) { B2::template store_cols<INV>(v, out + k.b * PR::kN + k.tile * PR::kG2, PR::kN1, i); });
    }
    ++done[k.pass * ring + slot];
  }
  for (int64_t i = 0; i < g.out_len; ++i)
    if (g.out_hits[i] != 1) { err("output element not written exactly once", i); break; }
  return g.errors;
}

template <int TL, int LOGL, bool INV>
void rows(const cf* in, cf* out, int64_t total, int64_t t, cf* sm) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_ROWS, CheckMem>;
  const int64_t valid = (total >> LOGL) - t * B::G;
  tile<SH, JOIN_ROWS>(
      sm, sm, g.tw1, 0, 0,
      [&](cf (&v)[kJoinR], int i) { B::template first_rows<INV>(v, in + (t << TL), valid, i); },
      [&](cf (&v)[kJoinR], int i) { B::store_rows(v, out + (t << TL), valid, i); });
}
template <int TL, int LOGL, bool INV>
void cols(cf* mid, cf* out, int64_t total, int64_t t, int lc, cf* sm) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_COLS, CheckMem>;
  tile<SH, JOIN_COLS>(
      sm, sm, g.tw2, 0, 0,
      [&](cf (&v)[kJoinR], int i) { B::first_frame(v, mid, t * B::G, total >> LOGL, lc, i); },
      [&](cf (&v)[kJoinR], int i) { B::template store_frame<INV>(v, out, t * B::G, total >> LOGL, lc, i); });
}

// Frames: the row pass writes `mid` (the output buffer on the GPU, kept apart
// here so that reads and writes of it can be checked on their own).
template <int TL, bool INV>
int64_t run_frames(int64_t batch, int lr, int lc, const cf* in, cf* out) {
  g = Ctx{};
  const int64_t total = batch << (lr + lc);
  std::vector<cf> t1 = roots(1 << lc), t2 = roots(1 << lr), mid(total), sm(1 << 15);
  const int tpt_log = std::max(0, lr + lc - TL);
  const int64_t nb = (total + (int64_t(1) << (TL + tpt_log)) - 1) >> (TL + tpt_log);
  int64_t lag, ring;
  join_plan(nb, tpt_log, 6, lag, ring);
  JoinOrder o{nb, tpt_log, (int)ring, lag};
  g.in = in;
  g.out = out;
  g.work = mid.data();
  g.in_len = g.out_len = g.work_len = total;
  g.out_hits.assign(total, 0);
  g.work_owner.assign(total, -1);
  g.b = 0;
  g.tw1 = t1.data();
  g.tw2 = t2.data();
  g.tw1_len = 1 << lc;
  g.tw2_len = 1 << lr;
  g.sm = sm.data();
  g.smem_len = (int)sm.size();
  g.phase_of.assign(sm.size(), -1);
  std::vector<uint32_t> done(2 * ring, 0);
  for (int64_t t = 0; t < join_tickets(o); ++t) {
    const JoinTicket k = join_ticket(o, t);
    const JoinDep dep = join_dep(o, k);
    if (k.b < 0 || k.b >= nb || k.tile < 0 || k.tile >> tpt_log) { err("ticket out of range", t); break; }
    if (done[dep.pass * ring + dep.slot] < dep.count) err("a ticket waits for a later one", t);
    const int64_t at = (k.b << tpt_log) + k.tile;
    switch (k.pass ? 100 + lr : lc) {
#define GB_R(L) case L: rows<TL, L, INV>(in, mid.data(), total, at, sm.data()); break;
#define GB_C(L) case 100 + L: cols<TL, L, INV>(mid.data(), out, total, at, lc, sm.data()); break;
      GB_R(4) GB_R(5) GB_R(6) GB_R(7) GB_R(8) GB_R(9) GB_R(10)
      GB_C(4) GB_C(5) GB_C(6) GB_C(7) GB_C(8)
      default:
        if constexpr (TL == 13) switch (k.pass ? 100 + lr : lc) { GB_C(9) GB_C(10) GB_C(11) default: break; }
#undef GB_R
#undef GB_C
    }
    ++done[k.pass * ring + (int)(k.b % ring)];
  }
  for (int64_t i = 0; i < total; ++i)
    if (g.out_hits[i] != 1 || g.work_owner[i] != 0) { err("element not written exactly once", i); break; }
  return g.errors;
}

// ---------------------------------------------------- fast convolution --
// Lines or columns of frames, tile by tile: the stages, the filter, the stages
// in reverse order.
template <int TL, int LOGL, int KIND>
void conv(const cf* in, cf* out, int64_t total, int lc, const cf* h, int64_t lines, float scale) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using RS = typename JoinReverse<SH>::S;
  using B = JoinBody<SH, KIND, CheckMem>;
  using BR = JoinBody<RS, KIND, CheckMem>;
  std::vector<cf> sm(std::max(B::kSlots, BR::kSlots));
  g.sm = sm.data();
  g.smem_len = (int)sm.size();
  g.phase_of.assign(sm.size(), -1);
  const int64_t n = total >> LOGL;
  for (int64_t t = 0; t * B::G < n; ++t) {
    std::vector<cf> keep((size_t)SH::kThreads * kJoinR);
    auto k = [&](int i) -> cf (&)[kJoinR] { return *reinterpret_cast<cf(*)[kJoinR]>(&keep[(size_t)i * kJoinR]); };
    auto copy = [](cf (&d)[kJoinR], const cf (&s)[kJoinR]) { for (int j = 0; j < kJoinR; ++j) d[j] = s[j]; };
    tile<SH, KIND>(
        sm.data(), sm.data(), g.tw1, 0, 0,
        [&](cf (&v)[kJoinR], int i) {
          if constexpr (KIND == JOIN_ROWS) B::template first_rows<false>(v, in + (t << TL), n - t * B::G, i);
          else B::first_frame(v, g.work, t * B::G, n, lc, i);
        },
        [&](cf (&v)[kJoinR], int i) { B::filter(v, h, lines, t * B::G, scale, i); copy(k(i), v); });
    tile<RS, KIND>(
        sm.data(), sm.data(), g.tw1, 0, 0, [&](cf (&v)[kJoinR], int i) { copy(v, k(i)); },
        [&](cf (&v)[kJoinR], int i) {
          if constexpr (KIND == JOIN_ROWS) BR::template store_rows<true>(v, g.work + (t << TL), n - t * B::G, i);
          else BR::template store_frame<true>(v, out, t * B::G, n, lc, i);
        });
  }
}

template <int KIND>
bool conv_len(int logl, const cf* in, cf* out, int64_t total, int lc, const cf* h, int64_t lines, float scale) {
  switch (logl) {
#define GB_CV(TL, L) case L: conv<TL, L, KIND>(in, out, total, lc, h, lines, scale); return true;
    GB_CV(12, 3) GB_CV(12, 4) GB_CV(12, 5) GB_CV(12, 6) GB_CV(12, 7) GB_CV(12, 8)
    default: break;
  }
  if constexpr (KIND == JOIN_ROWS) {
    switch (logl) { GB_CV(12, 9) GB_CV(12, 10) GB_CV(12, 11) default: break; }
  } else {
    switch (logl) { GB_CV(13, 9) GB_CV(13, 10) GB_CV(13, 11) default: break; }
  }
#undef GB_CV
  return false;
}

}  // namespace

extern "C" int64_t join_run(int logn, int tile_log, int64_t nb, int inverse, int64_t lag, int ring, const float* in,
                            float* out, char* msg, size_t len) {
  const cf* x = reinterpret_cast<const cf*>(in);
  cf* y = reinterpret_cast<cf*>(out);
  int64_t e = -1;
  switch (logn * 100 + tile_log) {
#define GB_RUN(L, TL) \
  case L * 100 + TL:  \
    e = inverse ? run<L, TL, true>(nb, lag, ring, x, y) : run<L, TL, false>(nb, lag, ring, x, y); break;
    GB_RUN(15, 12) GB_RUN(16, 12) GB_RUN(17, 12) GB_RUN(17, 13) GB_RUN(18, 12) GB_RUN(18, 13)
    GB_RUN(19, 13) GB_RUN(20, 13) GB_RUN(20, 14)
#undef GB_RUN
    default: break;
  }
  snprintf(msg, len, "%s", g.first.c_str());
  return e;
}

extern "C" int64_t join_run_frames(int64_t batch, int lr, int lc, int inverse, const float* in,
                                   float* out, char* msg, size_t len) {
  const cf* x = reinterpret_cast<const cf*>(in);
  cf* y = reinterpret_cast<cf*>(out);
  if (!join_frame(lr, lc, int64_t(1) << 40)) return -1;
  const int64_t e = join_frame_tile_log(lr) == 12
                        ? (inverse ? run_frames<12, true>(batch, lr, lc, x, y) : run_frames<12, false>(batch, lr, lc, x, y))
                        : (inverse ? run_frames<13, true>(batch, lr, lc, x, y) : run_frames<13, false>(batch, lr, lc, x, y));
  snprintf(msg, len, "%s", g.first.c_str());
  return e;
}

// cols = 0: batch lines of 2^logl; else the columns of 2^logl rows of frames of
// `cols` columns.  Filters as fft_filter_t lays them out.
extern "C" int64_t conv_run(int64_t batch, int logl, int cols, int64_t lines, float scale,
                            const float* h, const float* in, float* out, char* msg, size_t len) {
  const cf* x = reinterpret_cast<const cf*>(in);
  cf* y = reinterpret_cast<cf*>(out);
  const int64_t total = (batch << logl) * (cols ? cols : 1);
  int lc = 0;
  while (1 << lc < cols) ++lc;
  g = Ctx{};
  std::vector<cf> t1 = roots(1 << logl);
  g.in = x;
  g.out = y;
  g.in_len = g.out_len = g.work_len = total;
  g.tw1 = t1.data();
  g.tw1_len = 1 << logl;
  g.tw2 = nullptr;
  g.h = reinterpret_cast<const cf*>(h);
  g.h_len = lines << logl;
  g.out_hits.assign(total, 0);
  bool ok;
  if (cols) {  // columns read and write the output buffer: the input is put there first
    std::vector<cf> mid(x, x + total);
    g.work = mid.data();
    g.work_owner.assign(total, 0);
    ok = conv_len<JOIN_COLS>(logl, x, y, total, lc, g.h, lines, scale);
    for (int64_t i = 0; i < total; ++i)
      if (g.out_hits[i] != 1) { err("output element not written exactly once", i); break; }
  } else {
    g.work = y;
    g.work_owner.assign(total, -1);
    ok = conv_len<JOIN_ROWS>(logl, x, y, total, 0, g.h, lines, scale);
    for (int64_t i = 0; i < total; ++i)
      if (g.work_owner[i] != 0) { err("output element not written", i); break; }
  }
  if (!ok) err("no such length", logl);
  snprintf(msg, len, "%s", g.first.c_str());
  return g.errors;
}
