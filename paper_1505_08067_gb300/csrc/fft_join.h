// Per-thread phases of the joined kernels (joined.cuh): the two passes of a
// four-step transform (Sec. 3.3), or the row and column passes of 2D frames
// (Sec. 3.1), over tiles of 4096 .. 16384 elements, 32 per thread.
//
// One exchange instead of two: a pass of up to 1024 points is two stages
// (16 x 16, 32 x 16, 32 x 32), so its tile crosses shared memory once, and one
// stage fewer is twiddled (2048 .. 8192 points: three).  A stage's twiddles
// w^{ik}, i < r, are products of at most log2 r table values w^{k 2^m}, each
// FP64-generated and rounded once, which is closer to the exact value than the
// powers of a single root, and costs as many multiplies.
//
// Four-step transforms.  N = N1 N2, x[n1 N2 + n2], X[k2 N1 + k1]:
//   pass 1  a tile of 2^TL elements (4096 .. 16384) holds G1 = 2^TL / N1 adjacent
//           columns n2; the output is
//           multiplied by w_N^{n2 k1} and written to the workspace in blocks of
//           G2 = 2^TL / N2 values k1: element (n2, k1) at
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
};

// The same length with the stages in reverse order.
template <class SH> struct JoinReverse;
template <int TL, int LOGL, int RA, int RB, int RC>
struct JoinReverse<JoinShape<TL, LOGL, RA, RB, RC>> {
  using S = JoinShape<TL, LOGL, RC ? RC : RB, RC ? RB : RA, RC ? RA : 0>;
};

// What a tile's pass is: the first of a four-step transform (columns in, blocks
// of the workspace out), columns in and out, or contiguous rows in and out.
enum { JOIN_FIRST = 0, JOIN_COLS = 1, JOIN_ROWS = 2 };

// Mem: the memory policy (the device's, or the CPU replay's): ldin / ldw
// (input, intermediate), stw / stout, lds / sts, ldtw, rotor.
template <class SH, int KIND, class Mem>
struct JoinBody {
  static constexpr int G = SH::kG, L = SH::kL, R = kJoinR, T = SH::kThreads, TILE = SH::kTile;
  GB_HDC static constexpr int jbs(int s) { return L >> SH::rlog(s); }  // butterflies of stage s

  // Shared-memory layouts.  Column passes: adjacent columns adjacent, G slots
  // of padding after every 2^RA rows where G < 16.  The others: transform by
  // transform, a padding slot after every 2^RA elements and a pitch mod 16 of
  // 16 / G (first passes, whose loads put G lanes across the transforms) or of
  // the lanes along a transform (rows).  The 16 lanes of a half warp (64-bit
  // accesses) then touch 16 distinct slots mod 16 (rows of 32: two share one).
  static constexpr int kColPad = G < 16 ? G : 0;
  static constexpr int kMinJb = jbs(0) < jbs(SH::kLast) ? jbs(0) : jbs(SH::kLast);
  static constexpr int kPitch0 = L + (L >> SH::kRA);
  static constexpr int kPitchMod =
      KIND == JOIN_ROWS ? (kMinJb < 16 ? kMinJb : 0) : (G < 16 ? 16 / G : 1);
  static constexpr int kPitch = kPitch0 + ((kPitchMod - kPitch0) & 15);
  static constexpr int kSlots =
      KIND == JOIN_COLS ? L * G + (L >> SH::kRA) * kColPad : G * kPitch;
  GB_HD static int slot(int pos, int c) {
    if (KIND != JOIN_COLS) return c * kPitch + pos + (pos >> SH::kRA);
    return pos * G + c + (pos >> SH::kRA) * kColPad;
  }

  // Which butterfly (transform c of the tile, butterfly jb) of stage S the index
  // u = q T + thread id is: adjacent lanes across the columns where memory is
  // read or written by columns, along jb for rows; the last stage of a first
  // pass has 16 lanes along jb and the columns next.
  template <int S>
  GB_HD static void coords(int u, int& c, int& jb) {
    if (KIND == JOIN_ROWS) {
      jb = u % jbs(S);
      c = u / jbs(S);
    } else if (KIND == JOIN_COLS || S == 0) {
      c = u % G;
      jb = u / G;
    } else {
      c = (u >> 4) % G;
      jb = (u & 15) | (u / (16 * G)) << 4;
    }
  }

  // Stage 0 of a column pass: element a of column c at base + a*e + c; WORK:
  // from the workspace.
  template <bool INV, bool WORK>
  GB_HD static void first(cf (&v)[R], const cf* base, int e, int tid) {
    constexpr int RR = SH::radix(0), NB = R / RR;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<0>(q * T + tid, c, jb);
      const cf* p = base + (int64_t)jb * e + c;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf x = WORK ? Mem::ldw(p, i * (L / RR) * e) : Mem::ldin(p, i * (L / RR) * e);
        v[q * RR + i] = INV ? mk(x.y, x.x) : x;
      }
    }
  }
  // Stage 0 of a row pass: the tile's first `valid` rows, consecutive at base;
  // zeros for the rest.
  template <bool INV>
  GB_HD static void first_rows(cf (&v)[R], const cf* base, int64_t valid, int tid) {
    constexpr int RR = SH::radix(0), NB = R / RR;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<0>(q * T + tid, c, jb);
      const cf* p = base + c * L + jb;
      const bool ok = c < valid;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf x = ok ? Mem::ldin(p, i * (L / RR)) : mk(0.f, 0.f);
        v[q * RR + i] = INV ? mk(x.y, x.x) : x;
      }
    }
  }
  // Column `col` of all frames of L rows of 2^lc elements: its first element.
  GB_HD static int64_t frame_col(int64_t col, int lc) {
    return ((col >> lc) << (SH::kLogL + lc)) + (col & ((int64_t(1) << lc) - 1));
  }
  // Fast convolution, between its two rounds: after the forward stages this
  // thread holds the spectrum at positions jb + i Ns of its last-stage
  // butterflies, which are the inputs of its first-stage butterflies in the
  // reversed schedule (Ns = L / radix).  Multiplies them by scale * H and swaps
  // real and imaginary parts for the inverse.  Rows: line u's filter at
  // h + (u mod lines) L (first: the tile's first line); columns: column u's in
  // column u mod lines of a frame of rows of `lines` elements; lines = 1: one
  // filter for all.
  GB_HD static void filter(cf (&v)[R], const cf* h, int64_t lines, int64_t first, float scale,
                           int tid) {
    constexpr int S = SH::kLast, RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
    if (first >= lines) first %= lines;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<S>(q * T + tid, c, jb);
      int64_t u = lines > 1 ? first + c : 0;
      if (u >= lines) u %= lines;  // seldom: first is below lines
      const int64_t e = KIND == JOIN_COLS && lines > 1 ? lines : 1;
      const cf* p = h + (KIND == JOIN_COLS ? u : u * L) + jb * e;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf z = cmul(v[q * RR + i], Mem::ldtw(p + i * Ns * e));
        v[q * RR + i] = mk(z.y * scale, z.x * scale);
      }
    }
  }

  // Stage 0 of a frame's column pass: columns col0 .. col0 + G - 1 of all the
  // frames in buf, of which there are `cols`; zeros beyond.
  GB_HD static void first_frame(cf (&v)[R], const cf* buf, int64_t col0, int64_t cols, int lc,
                                int tid) {
    constexpr int RR = SH::radix(0), NB = R / RR;
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<0>(q * T + tid, c, jb);
      const cf* p = buf + frame_col(col0 + c, lc) + (jb << lc);
      const bool ok = col0 + c < cols;
GB_UNROLL
      for (int i = 0; i < RR; ++i)
        v[q * RR + i] = ok ? Mem::ldw(p, (i * (L / RR)) << lc) : mk(0.f, 0.f);
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
      coords<S>(q * T + tid, c, jb);
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
      coords<S>(q * T + tid, c, jb);
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
      coords<S>(q * T + tid, c, jb);
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
  // stage, for every column of the tile: st[i * G + c], by `lanes` threads.
  static constexpr int kSteps = G * SH::radix(SH::kLast);
  GB_HD static void steps(cf* st, int col0, int logN, int lane, int lanes = 32) {
    for (int x = lane; x < kSteps; x += lanes) {
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
      coords<S>(q * T + tid, c, jb);
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
      coords<S>(q * T + tid, c, jb);
      cf* p = base + (int64_t)jb * e + c;
GB_UNROLL
      for (int i = 0; i < RR; ++i) {
        const cf x = v[q * RR + i];
        Mem::stout(p, i * Ns * e, INV ? mk(x.y, x.x) : x);
      }
    }
  }
  // Last stage of a row pass / of a frame's column pass.
  template <bool INV = false>
  GB_HD static void store_rows(const cf (&v)[R], cf* base, int64_t valid, int tid) {
    constexpr int S = SH::kLast, RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<S>(q * T + tid, c, jb);
      cf* p = base + c * L + jb;
      if (c < valid) {
GB_UNROLL
        for (int i = 0; i < RR; ++i) {
          const cf x = v[q * RR + i];
          Mem::stw(p, i * Ns, INV ? mk(x.y, x.x) : x);
        }
      }
    }
  }
  template <bool INV>
  GB_HD static void store_frame(const cf (&v)[R], cf* buf, int64_t col0, int64_t cols, int lc,
                                int tid) {
    constexpr int S = SH::kLast, RR = SH::radix(S), NB = R / RR, Ns = SH::ns(S);
GB_UNROLL
    for (int q = 0; q < NB; ++q) {
      int c, jb;
      coords<S>(q * T + tid, c, jb);
      cf* p = buf + frame_col(col0 + c, lc) + (jb << lc);
      if (col0 + c < cols) {
GB_UNROLL
        for (int i = 0; i < RR; ++i) {
          const cf x = v[q * RR + i];
          Mem::stout(p, (i * Ns) << lc, INV ? mk(x.y, x.x) : x);
        }
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
  static constexpr int kSteps = S1::kG << S1::rlog(S1::kLast);
};
template <int TL> using Join128 = JoinShape<TL, 7, 4, 3>;
template <int TL> using Join256 = JoinShape<TL, 8, 4, 4>;
template <int TL> using Join512 = JoinShape<TL, 9, 5, 4>;
template <int TL> using Join1024 = JoinShape<TL, 10, 5, 5>;
// Lengths of row and column passes (2^4 .. 2^10 rows, 2^4 .. 2^11 columns in joined
// frames; 2^3 .. 2^11 in lines.cu and conv_lines.cu).
template <int TL, int LOGL> struct JoinLen;
template <int TL> struct JoinLen<TL, 3> { using S = JoinShape<TL, 3, 1, 2>; };
template <int TL> struct JoinLen<TL, 4> { using S = JoinShape<TL, 4, 2, 2>; };
template <int TL> struct JoinLen<TL, 5> { using S = JoinShape<TL, 5, 3, 2>; };
template <int TL> struct JoinLen<TL, 6> { using S = JoinShape<TL, 6, 3, 3>; };
template <int TL> struct JoinLen<TL, 7> { using S = Join128<TL>; };
template <int TL> struct JoinLen<TL, 8> { using S = Join256<TL>; };
template <int TL> struct JoinLen<TL, 9> { using S = Join512<TL>; };
template <int TL> struct JoinLen<TL, 10> { using S = Join1024<TL>; };
template <int TL> struct JoinLen<TL, 11> { using S = JoinShape<TL, 11, 4, 4, 3>; };
// TL: log2 of the tile (join_tile_log).
template <int LOGN, int TL> struct JoinPair;
template <int TL> struct JoinPair<15, TL> : JoinPairOf<Join128<TL>, Join256<TL>> {};
template <int TL> struct JoinPair<16, TL> : JoinPairOf<Join256<TL>, Join256<TL>> {};
template <int TL> struct JoinPair<17, TL> : JoinPairOf<Join256<TL>, Join512<TL>> {};
template <int TL> struct JoinPair<18, TL> : JoinPairOf<Join512<TL>, Join512<TL>> {};
template <int TL> struct JoinPair<19, TL> : JoinPairOf<Join512<TL>, Join1024<TL>> {};
template <int TL> struct JoinPair<20, TL> : JoinPairOf<Join1024<TL>, Join1024<TL>> {};
constexpr int kJoinMinLog = 15, kJoinMaxLog = 20;
// Tiles of a transform of 2^logn points.  Joined, with work for several tiles per
// block: the smallest whose row segments are 128 bytes wide (64 in one of the two
// passes of 2^17 .. 2^19).  Apart, on fewer elements: smaller, over more SMs
// (2^22 elements: 2^17 20.0 us against 24.1 for twice the tile, 2^18 21.7 and
// 24.6, 2^20 26.1 and 30.4).
GB_HD constexpr int join_tile_log(int logn, bool apart) {
  return apart ? (logn <= 18 ? 12 : 13) : logn <= 16 ? 12 : logn <= 19 ? 13 : 14;
}
// log2 of the blocks per SM (512 threads of 32 elements in all).
GB_HD constexpr int join_blocks_log(int tile_log) { return 14 - tile_log; }
// Such transforms run with the passes of this file: joined, or (join_apart) in
// a launch each.  While the whole batch fits L2, so does the intermediate in any
// order, and two launches that start early have no dispatching warp, no waits
// and more registers.  Measured, the two-launch kernels before (launched early
// too), apart, and joined: 2^15 x 1 5.7, 4.2, 8.3 us; 2^18 x 1 10.6, 5.4, 8.9;
// 2^20 x 1 11.4, 8.2, 17.0; 2^18 x 16 34.0, 21.7, 28.2; 2^17 x 64 52.9, 37.4, 45.0;
// 2^17 x 97 84.2, 63.0, 61.9; 2^17 x 128 110, 88, 78; 2^20 x 12 81, 75, 72.
GB_HD constexpr bool join_transform(int logn) { return logn >= kJoinMinLog && logn <= kJoinMaxLog; }
GB_HD constexpr bool join_apart(int64_t elems) { return elems < int64_t(3) << 22; }

// Frames: rows of 2^lc, columns of 2^lr, `elems` elements in all.  Below 2^23.6
// elements the intermediate fits L2 in any order, and a launch per pass (lines.cu)
// is up to twice as fast (1024 x 1024: 17.0 -> 9 us; 2^23 elements 5% to 20%); rows
// of 2048 and more are faster in launches of their own at every size.
GB_HD constexpr bool join_frame(int lr, int lc, int64_t elems) {
  return lr >= 4 && lr <= 11 && lc >= 4 && lc <= 10 && elems >= int64_t(3) << 22;
}
GB_HD constexpr int join_frame_tile_log(int lr) { return lr <= 8 ? 12 : 13; }

// ------------------------------------------------------------- the order --
// Tiles are handed out in one order to whichever block asks next (a counter),
// so a tile only ever waits for tiles handed out before it, which running
// blocks hold: no wait depends on blocks that have not started.
//
// A unit is a transform, a frame, or a tile's worth of smaller frames.  The
// second pass follows the first by `lag` tiles: a unit's, and as many more as
// keep every block busy on later units while the last tiles of its first pass
// finish.  So what the second pass reads was written a few tens of MB earlier
// and is still in L2.  The workspace of four-step transforms is a ring of
// `ring` units, large enough that a slot's second pass is over when its next
// first pass comes up: the intermediate is overwritten in L2 and need not reach
// HBM.  (Frames have their intermediate in the output; there the ring only
// numbers the counters.)
struct JoinOrder {
  int64_t nb;       // units
  int32_t tpt_log;  // log2 tiles per unit and pass
  int32_t ring;
  int64_t lag;      // tiles, at most nb << tpt_log
};
struct JoinTicket {
  int pass;     // 0 or 1
  int64_t b;    // unit
  int32_t tile;
};
GB_HD int64_t join_tickets(const JoinOrder& o) { return (2 * o.nb) << o.tpt_log; }
// lag tiles of the first pass, then second and first pass in turn, then the
// last lag tiles of the second.
GB_HD JoinTicket join_ticket(const JoinOrder& o, int64_t t) {
  JoinTicket k;
  const int64_t tiles = o.nb << o.tpt_log, both = t - o.lag;
  int64_t i = t;
  k.pass = 0;
  if (both >= 2 * (tiles - o.lag)) {
    k.pass = 1;
    i = t - tiles;
  } else if (both >= 0) {
    k.pass = both & 1 ? 0 : 1;
    i = (both >> 1) + (k.pass ? 0 : o.lag);
  }
  k.b = i >> o.tpt_log;
  k.tile = (int32_t)(i - (k.b << o.tpt_log));
  return k;
}
// The lag and the ring for `batch` units of 2^tpt_log tiles with `resident`
// blocks at work: a margin of 1.125 tiles per block (measured: 0.6 costs up to
// 20% in waits, 2.5 as much in L2 misses).
GB_HD void join_plan(int64_t batch, int tpt_log, int64_t resident, int64_t& lag, int64_t& ring) {
  const int64_t unit = int64_t(1) << tpt_log, margin = resident + resident / 8;
  lag = unit + margin;
  if (lag > batch * unit) lag = batch * unit;
  ring = 2 + (2 * margin + unit - 1) / unit;
  if (ring > batch) ring = batch;
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
