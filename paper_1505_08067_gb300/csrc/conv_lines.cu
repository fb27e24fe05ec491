// Fast convolution of contiguous lines and of the columns of frames (2^3 .. 2^11
// points): a tile of 4096 or 8192 elements per block, the stages of fft_join.h,
// the filter in registers, the stages in reverse order.
//
// These lengths ran the run-time-parameter kernel (address arithmetic, a radix-2
// to 16 switch per stage, two to three exchanges per round and one between the
// rounds unless the last radix is 16).  Here each round has one exchange up to
// 1024 points, and the reversed schedule makes a thread's last-stage outputs its
// next first-stage inputs at every length.  What bounds it now is the work of
// two transforms per line on 16 warps an SM; row and column passes are launches
// of their own: one kernel with a dispatching warp left 96 registers a thread,
// and the filter's loads spilled.
// Measured, 2^25 elements, one filter, before and now: lines of 16 226 -> 111 us,
// 64 202 -> 92, 256 176 -> 92, 512 264 -> 101, 1024 272 -> 107, 2048 281 -> 155;
// frames 128 x 128 410 -> 205, 512 x 512 543 -> 220, 1024 x 1024 595 -> 248,
// 2048 x 2048 617 -> 371; 2^17 elements: 6.3-14.5 -> 6.1-8.3 us, frames
// 20.7-39.2 -> 12.5-14.7.  Lines of 4096 and 8192 stay with the staged kernel
// (152 against 166 us, 162 against 197).
#include "joined.cuh"

namespace gbfft {

template <int TL, int LOGL>
__global__ void __launch_bounds__((1 << TL) / kJoinR, 1 << join_blocks_log(TL))
conv_lines(const cf* __restrict__ in, cf* out, const __grid_constant__ PassDesc d) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_ROWS, JoinMem>;
  using BR = JoinBody<typename JoinReverse<SH>::S, JOIN_ROWS, JoinMem>;
  extern __shared__ __align__(16) unsigned char smem_lines[];
  cf* sm = reinterpret_cast<cf*>(smem_lines);
  const int tid = threadIdx.x;
  const int64_t at = (int64_t)blockIdx.x << TL, line = (int64_t)blockIdx.x * B::G;
  grid_wait();
  cf v[kJoinR];
  B::template first_rows<false>(v, in + at, d.count_inner - line, tid);
  join_conv<SH, JOIN_ROWS>(v, sm, d.tw + d.tw_line, d.h, d.h_lines, d.h_first + line, d.h_scale, tid);
  BR::template store_rows<true>(v, out + at, d.count_inner - line, tid);
}

// Columns of 2^LOGL rows of d.in.e elements, in place or not.
template <int TL, int LOGL>
__global__ void __launch_bounds__((1 << TL) / kJoinR, 1 << join_blocks_log(TL))
conv_cols(const cf* in, cf* out, const __grid_constant__ PassDesc d) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_COLS, JoinMem>;
  using BR = JoinBody<typename JoinReverse<SH>::S, JOIN_COLS, JoinMem>;
  extern __shared__ __align__(16) unsigned char smem_lines[];
  cf* sm = reinterpret_cast<cf*>(smem_lines);
  const int tid = threadIdx.x, lc = 31 - __clz((int)d.in.e);
  const int64_t col0 = (int64_t)blockIdx.x * B::G, cols = d.tiles / d.tiles_inner * d.count_inner;
  grid_wait();
  cf v[kJoinR];
  B::first_frame(v, in, col0, cols, lc, tid);
  join_conv<SH, JOIN_COLS>(v, sm, d.tw + d.tw_line, d.h, d.h_lines, col0, d.h_scale, tid);
  BR::template store_frame<true>(v, out, col0, cols, lc, tid);
}

template <int TL, int LOGL>
static bool conv_lines_fn(PassLaunch* l) {
  l->fn = (const void*)conv_lines<TL, LOGL>;
  l->smem = join_conv_slots<typename JoinLen<TL, LOGL>::S, JOIN_ROWS>() * sizeof(cf);
  l->block = (1 << TL) / kJoinR;
  l->lines = TL;
  return true;
}

bool resolve_conv_lines(int logL, PassLaunch* l) {
  switch (logL) {
    case 3: return conv_lines_fn<12, 3>(l);
    case 4: return conv_lines_fn<12, 4>(l);
    case 5: return conv_lines_fn<12, 5>(l);
    case 6: return conv_lines_fn<12, 6>(l);
    case 7: return conv_lines_fn<12, 7>(l);
    case 8: return conv_lines_fn<12, 8>(l);
    case 9: return conv_lines_fn<12, 9>(l);
    case 10: return conv_lines_fn<12, 10>(l);
    case 11: return conv_lines_fn<12, 11>(l);
    default: return false;
  }
}

template <int TL, int LOGL>
static bool conv_cols_fn(PassLaunch* l) {
  l->fn = (const void*)conv_cols<TL, LOGL>;
  l->smem = join_conv_slots<typename JoinLen<TL, LOGL>::S, JOIN_COLS>() * sizeof(cf);
  l->block = (1 << TL) / kJoinR;
  l->lines = TL;
  return true;
}

bool resolve_conv_cols(int logL, PassLaunch* l) {
  switch (logL) {
    case 3: return conv_cols_fn<12, 3>(l);
    case 4: return conv_cols_fn<12, 4>(l);
    case 5: return conv_cols_fn<12, 5>(l);
    case 6: return conv_cols_fn<12, 6>(l);
    case 7: return conv_cols_fn<12, 7>(l);
    case 8: return conv_cols_fn<12, 8>(l);
    case 9: return conv_cols_fn<13, 9>(l);
    case 10: return conv_cols_fn<13, 10>(l);
    case 11: return conv_cols_fn<13, 11>(l);
    default: return false;
  }
}

}  // namespace gbfft
