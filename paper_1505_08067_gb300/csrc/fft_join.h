// Per-thread phases of the joined two-pass kernel (joined.cu): both passes of
// a four-step transform (Sec. 3.3) as column passes over tiles of 8192
// elements, 32 per thread.
//
// One exchange instead of two: a pass of 256 / 512 / 1024 points is two stages
// (16 x 16, 32 x 16, 32 x 32), so its tile crosses shared memory once, and one
// stage fewer is twiddled.  (2048 points: 16 x 16 x 8.)  A stage's twiddles
// w^{ik}, i < r, are products of at most log2 r table values w^{k 2^m}, each
// FP64-generated and rounded once, which is closer to the exact value than the
// powers of a single root, and costs as many multiplies.
//
// N = N1 N2, x[n1 N2 + n2], X[k2 N1 + k1]:
//   pass 1  a tile holds G1 = 8192 / N1 adjacent columns n2; the output is
//           multiplied by w_N^{n2 k1} and written to the workspace in blocks of
//           G2 = 8192 / N2 values k1: element (n2, k1) at
//             (k1 / G2) (N2 G2) + n2 G2 + (k1 mod G2);
//   pass 2  a tile holds G2 adjacent k1 -- one contiguous block of the
//           workspace -- and writes G2 adjacent outputs per row k2.
// The workspace layout is private to the two passes: the second reads whole
// contiguous tiles, the first writes runs of G2 elements per column and, with
// 16 lanes along k1 and two adjacent columns per warp, whole 128-byte lines.
//
// w_N^{n2 k1} with k1 = jb + i Ns (last stage: butterfly jb, output i) is
// w_N^{n2 jb} w_N^{n2 Ns i}.  The first factor is the same for every output of
// a butterfly, so it multiplies the butterfly's inputs instead, where it is
// folded into their twiddles (the chain starts from it); the second depends on
// the column and i only: G1 * r values per tile, computed once per tile and
// kept in shared memory.
#pragma once
#include "fft_core.h"
#include "fft_stage.h"

namespace gbfft {

constexpr int kJoinR = 32;  // elements per thread

// cos / sin of odd multiples of pi/16 (32-point roots), rounded to FP32.
#define GB_C16 0.98078528040323044f
#define GB_S16 0.19509032201612826f
#define GB_C316 0.83146961230254524f
#define GB_S316 0.55557023301960222f

// a * w32^m, w32 = exp(-2 pi i / 32); m is a compile-time constant once unrolled.
GB_HD cf mul_w32(cf a, int m) {
  m &= 31;
  if ((m & 1) == 0) return mul_w16(a, m >> 1);
  switch (m) {
    case 1: return cmul(a, mk(GB_C16, -GB_S16));
    case 3: return cmul(a, mk(GB_C316, -GB_S316));
    case 5: return cmul(a, mk(GB_S316, -GB_C316));
    case 7: return cmul(a, mk(GB_S16, -GB_C16));
    case 9: return cmul(a, mk(-GB_S16, -GB_C16));
    case 11: return cmul(a, mk(-GB_S316, -GB_C316));
    case 13: return cmul(a, mk(-GB_C316, -GB_S316));
    case 15: return cmul(a, mk(-GB_C16, -GB_S16));
    case 17: return cmul(a, mk(-GB_C16, GB_S16));
    case 19: return cmul(a, mk(-GB_C316, GB_S316));
    case 21: return cmul(a, mk(-GB_S316, GB_C316));
    case 23: return cmul(a, mk(-GB_S16, GB_C16));
    case 25: return cmul(a, mk(GB_S16, GB_C16));
    case 27: return cmul(a, mk(GB_S316, GB_C316));
    case 29: return cmul(a, mk(GB_C316, GB_S316));
    default: return cmul(a, mk(GB_C16, GB_S16));  // 31
  }
}

// Forward DFT of length 32 = 8 x 4 in registers, natural order in and out
// (n = 4 n1 + n2, k = k1 + 8 k2).
GB_HD void dft32(cf* v) {
  cf t[32];
GB_UNROLL
  for (int n2 = 0; n2 < 4; ++n2) {
    cf y[8];
GB_UNROLL
    for (int n1 = 0; n1 < 8; ++n1) y[n1] = v[4 * n1 + n2];
    dft_pq<2, 4>(y);
GB_UNROLL
    for (int k1 = 0; k1 < 8; ++k1) t[4 * k1 + n2] = mul_w32(y[k1], n2 * k1);
  }
GB_UNROLL
  for (int k1 = 0; k1 < 8; ++k1) {
    dft_small<4, 1>(t + 4 * k1);
GB_UNROLL
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 8 * k2] = t[4 * k1 + k2];
  }
}

template <int RR>
GB_HD void join_dft(cf* v) {
  if constexpr (RR == 32) dft32(v);
  else dft_radix<RR>(v);
}

// A pass of 2^LOGL points in tiles of 2^TL elements: log2 radices RA, RB (and
// RC) of its stages.
template <int TL, int LOGL, int RA, int RB, int RC = 0>
struct JoinShape {
  static_assert(RA + RB + RC == LOGL, "the radices multiply to the length");
  static constexpr int kLogL = LOGL, kL = 1 << LOGL, kTileLog = TL, kTile = 1 << TL;
  static constexpr int kThreads = kTile / kJoinR;
  static constexpr int kG = kTile / kL;  // transforms per tile
  static constexpr int kNst = RC ? 3 : 2;
  static constexpr int kRA = RA;
  GB_HDC static constexpr int rlog(int s) { return s == 0 ? RA : s == 1 ? RB : RC; }
  GB_HDC static constexpr int radix(int s) { return 1 << rlog(s); }
  GB_HDC static constexpr int ns(int s) { return s == 0 ? 1 : s == 1 ? 1 << RA : 1 << (RA + RB); }
  static constexpr int kLast = kNst - 1;
  // Shared-memory layouts.  By column (ROWL = false): adjacent columns
  // adjacent, G slots of padding after every 2^RA rows where G < 16.  By
  // transform (ROWL = true): a padding slot after every 2^RA elements and a
  // pitch of max(1, 16 / G) mod 16.  With the thread maps below the 16 lanes
  // of a half warp (64-bit accesses) then always touch 16 distinct slots mod 16.
  static constexpr int kColPad = kG < 16 ? kG : 0;
  static constexpr int kPitch0 = kL + (kL >> RA);
  static constexpr int kPitch = kPitch0 + (((kG < 16 ? 16 / kG : 1) - kPitch0) & 15);
  static constexpr int kSlotsCol = kL * kG + (kL >> RA) * kColPad;
  static constexpr int kSlotsRow = kG * kPitch;
};

// Which butterfly (transform c of the tile, butterfly jb) the index
// u = q * 256 + thread id is: adjacent lanes along the columns, or 16 lanes along
// jb and the columns next.
enum { JMAP_COLS = 0, JMAP_BLOCK = 1 };

// ROWL: the shared layout.  Mem: the memory policy (the device's, or the CPU
// replay's): ldin / ldw (input, workspace), stw / stout, lds / sts, ldtw, rotor.
template <class SH, bool ROWL, class Mem>
struct JoinBody {
  static constexpr int G = SH::kG, L = SH::kL, R = kJoinR, T = SH::kThreads;
  static constexpr int kSlots = ROWL ? SH::kSlotsRow : SH::kSlotsCol;

  template <int MAP>
  GB_HD static void coords(int u, int& c, int& jb) {
    if (MAP == JMAP_COLS) {
      c = u % G;
      jb = u / G;
    } else {
      c = (u >> 4) % G;
      jb = (u & 15) | (u / (16 * G)) << 4;
    }
  }
  GB_HD static int slot(int pos, int c) {
    if (ROWL) return c * SH::kPitch + pos + (pos >> SH::kRA);
    return pos * G + c + (pos >> SH::kRA) * SH::kColPad;
  }
  // Thread map of stage s: the loads' (columns) at first, the stores' at
  // last; a middle stage's lanes follow the shared layout.
  GB_HDC static constexpr int map_of(int s) {
    return s == 0 || !ROWL ? JMAP_COLS : JMAP_BLOCK;
  }

  // Stage 0: element a of column c at base + a*e + c; WORK: from the workspace.
  template <bool INV, bool WORK>
  GB_HD static void first(cf (&v)[R], const cf* base, int e, int tid) {
    constexpr int RR = SH::radix(0), NB = R / RR;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<JMAP_COLS>(q * T + tid, c, jb);
      const cf* p = base + (int64_t)jb * e + c;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf x = WORK ? Mem::ldw(p, i * (L / RR) * e) : Mem::ldin(p, i * (L / RR) * e);
        v[q * RR + i] = INV ? mk(x.y, x.x) : x;
      }
    }
  }
  GB_HD static void dft0(cf (&v)[R]) {
    constexpr int RR = SH::radix(0);
GB_UNROLL
    for (int q = 0; q < R / RR; ++q) join_dft<RR>(v + q * RR);
  }

  // Outputs of stage S to shared memory, natural (Stockham) order.
  template <int S>
  GB_HD static void put(const cf (&v)[R], cf* sm, int tid) {
    constexpr int RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<map_of(S)>(q * T + tid, c, jb);
      const int k = jb & (Ns - 1);
      const int base = (jb - k) * RR + k;
GB_UNROLL
      for (int i = 0; i < RR; ++i) Mem::sts(sm, slot(base + i * Ns, c), v[q * RR + i]);
    }
  }

  // Stage S's inputs from shared memory.
  template <int S>
  GB_HD static void get(cf (&v)[R], const cf* sm, int tid) {
    constexpr int RR = SH::radix(S), NB = R / RR;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<map_of(S)>(q * T + tid, c, jb);
GB_UNROLL
      for (int i = 0; i < RR; ++i) v[q * RR + i] = Mem::lds(sm, slot(jb + i * (L / RR), c));
    }
  }

  // Stage S: twiddles and DFT.  tw: w_L^j, j < L.  TW4: the four-step
  // twiddle's factor w_N^{col jb}, N = 2^logN, folded into the inputs' twiddles
  // (col0: the tile's first column).
  template <int S, bool TW4>
  GB_HD static void turn(cf (&v)[R], const cf* tw, int col0, int logN, int tid) {
    constexpr int RR = SH::radix(S), RL = SH::rlog(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<map_of(S)>(q * T + tid, c, jb);
      const int k = (jb & (Ns - 1)) * (L / (Ns * RR));
      cf w[RR];
      if (TW4) {
        w[0] = Mem::rotor((int64_t)(col0 + c) * jb, logN);
        v[q * RR] = cmul(v[q * RR], w[0]);
      }
GB_UNROLL
      for (int m = 0; m < RL; ++m) {
        const cf r = Mem::ldtw(tw + (k << m));
        w[1 << m] = TW4 ? cmul(w[0], r) : r;
GB_UNROLL
        for (int j = 1; j < (1 << m); ++j) w[(1 << m) + j] = cmul(w[j], r);
      }
GB_UNROLL
      for (int i = 1; i < RR; ++i) v[q * RR + i] = cmul(v[q * RR + i], w[i]);
      join_dft<RR>(v + q * RR);
    }
  }

  // The second factor of the four-step twiddle, w_N^{col Ns i} of the last
  // stage, for every column of the tile: st[i * G + c].
  // Computed by one warp.
  static constexpr int kSteps = G * SH::radix(SH::kLast);
  GB_HD static void steps(cf* st, int col0, int logN, int lane) {
    for (int x = lane; x < kSteps; x += 32) {
      const int i = x / G, c = x - i * G;
      Mem::sts(st, x, Mem::rotor((int64_t)(col0 + c) * (i * SH::ns(SH::kLast)), logN));
    }
  }

  // Pass 1: outputs times the steps to the workspace in blocks of G2 rows
  // k1; wb: the workspace at this tile's first column (n2 = 0 of the block
  // layout plus col0 * G2), cols: N2.
  template <int G2>
  GB_HD static void store_block(const cf (&v)[R], cf* wb, const cf* st, int cols, int tid) {
    constexpr int S = SH::kLast, RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<map_of(S)>(q * T + tid, c, jb);
      cf* p = wb + (jb / G2) * (cols * G2) + c * G2 + jb % G2;
GB_UNROLL
      for (int i = 0; i < RR; ++i)
        Mem::stw(p, (i * Ns / G2) * (cols * G2) + i * Ns % G2,
                 cmul(v[q * RR + i], Mem::lds(st, i * G + c)));
    }
  }

  // Last stage's outputs, row a of column c at base + a*e + c.
  template <bool INV>
  GB_HD static void store_cols(const cf (&v)[R], cf* base, int e, int tid) {
    constexpr int S = SH::kLast, RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<map_of(S)>(q * T + tid, c, jb);
      cf* p = base + (int64_t)jb * e + c;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf x = v[q * RR + i];
        Mem::stout(p, i * Ns * e, INV ? mk(x.y, x.x) : x);
      }
    }
  }
};

// A two-pass transform of N = 2^LOGN points: the shapes of its passes.
template <class S1, class S2>
struct JoinPairOf {
  using P1 = S1;
  using P2 = S2;
  static_assert(S1::kTileLog == S2::kTileLog, "one block size for both passes");
  static constexpr int kLogN = S1::kLogL + S2::kLogL;
  static constexpr int kN = 1 << kLogN, kN1 = S1::kL, kN2 = S2::kL;
  static constexpr int kG1 = S1::kG, kG2 = S2::kG;
  static constexpr int kThreads = S1::kThreads, kTileLog = S1::kTileLog, kTile = S1::kTile;
  static constexpr int kTiles = kN / kTile;  // tiles of one transform, per pass
  // shared-memory elements: the larger tile, then the first pass's steps
  static constexpr int kSlots = S1::kSlotsRow > S2::kSlotsCol ? S1::kSlotsRow : S2::kSlotsCol;
  static constexpr int kTileSlots = kSlots;
  static constexpr int kSteps = S1::kG << S1::rlog(S1::kLast);
};
template <int TL> using Join128 = JoinShape<TL, 7, 4, 3>;
template <int TL> using Join256 = JoinShape<TL, 8, 4, 4>;
template <int TL> using Join512 = JoinShape<TL, 9, 5, 4>;
template <int TL> using Join1024 = JoinShape<TL, 10, 5, 5>;
template <int LOGN> struct JoinPair;
template <> struct JoinPair<15> : JoinPairOf<Join128<12>, Join256<12>> {};
template <> struct JoinPair<16> : JoinPairOf<Join256<12>, Join256<12>> {};
template <> struct JoinPair<17> : JoinPairOf<Join256<13>, Join512<13>> {};
template <> struct JoinPair<18> : JoinPairOf<Join512<13>, Join512<13>> {};
template <> struct JoinPair<19> : JoinPairOf<Join512<13>, Join1024<13>> {};
template <> struct JoinPair<20> : JoinPairOf<Join1024<14>, Join1024<14>> {};
constexpr int kJoinMinLog = 15, kJoinMaxLog = 20;
// log2 of the tile, and of the blocks per SM it allows (512 threads of 32
// elements in all).
GB_HD constexpr int join_tile_log(int logn) { return logn <= 16 ? 12 : logn <= 19 ? 13 : 14; }
GB_HD constexpr int join_blocks_log(int tile_log) { return 14 - tile_log; }
// Fewest elements a plan joins its passes for.
constexpr int64_t kJoinMinElems = int64_t(1) << 21;

// ------------------------------------------------------------- the order --
// Tiles are handed out in one order to whichever block asks next (a counter),
// so a tile only ever waits for tiles handed out before it, which running
// blocks hold: no wait depends on blocks that have not started.
//
// Transform b's second pass follows its first by `lag` transforms; in between,
// first-pass tiles of later transforms keep every block busy while the last
// tiles of b's first pass finish.  The workspace is a ring of `ring` >= lag + 1
// transforms, so what the second pass reads was written a few tens of MB
// earlier and is still in L2, and the next user of the slot overwrites it
// there: the intermediate need not reach HBM.
struct JoinOrder {
  int64_t nb;  // transforms
  int32_t tpt_log;  // log2 tiles per transform and pass
  int32_t lag, ring;
};
struct JoinTicket {
  int pass;     // 0 or 1
  int64_t b;    // transform
  int32_t tile;
};
GB_HD int64_t join_tickets(const JoinOrder& o) { return (2 * o.nb) << o.tpt_log; }
GB_HD JoinTicket join_ticket(const JoinOrder& o, int64_t t) {
  JoinTicket k;
  const int64_t lead = (int64_t)o.lag << o.tpt_log;
  const int32_t mask = (1 << o.tpt_log) - 1;
  if (t < lead) {  // the first `lag` transforms' first passes
    k.pass = 0;
    k.b = t >> o.tpt_log;
    k.tile = (int32_t)t & mask;
    return k;
  }
  t -= lead;
  const int64_t mid = (2 * (o.nb - o.lag)) << o.tpt_log;
  if (t < mid) {  // second pass of b, first pass of b + lag, tile by tile
    const int64_t b = t >> (o.tpt_log + 1);
    k.pass = (t & 1) ? 0 : 1;
    k.b = k.pass ? b : b + o.lag;
    k.tile = (int32_t)(t >> 1) & mask;
    return k;
  }
  t -= mid;
  k.pass = 1;
  k.b = o.nb - o.lag + (t >> o.tpt_log);
  k.tile = (int32_t)t & mask;
  return k;
}
// What ticket k waits for: `count` finished tiles of ring slot `slot` in pass
// `pass` (counted over the slot's users so far); count 0: nothing.
struct JoinDep {
  int pass, slot;
  uint32_t count;
};
GB_HD JoinDep join_dep(const JoinOrder& o, const JoinTicket& k) {
  JoinDep d;
  const int64_t use = k.b / o.ring;
  d.slot = (int)(k.b - use * o.ring);
  d.pass = k.pass ? 0 : 1;  // its own first pass, or the slot's previous second pass
  d.count = (uint32_t)((k.pass ? use + 1 : use) << o.tpt_log);
  return d;
}

}  // namespace gbfft
