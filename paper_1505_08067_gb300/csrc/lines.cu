// Batches of short contiguous transforms (2^3 .. 2^10 points): a tile of 4096
// elements per 128-thread block as a row pass of fft_join.h, 32 elements and one
// exchange per thread; and the column passes of frames of 2^3 .. 2^11 rows in the
// same way.  Server jobs run the same tiles alone (short_lines) or coalesced
// (grouped_lines), and the work queue's worker does (queue.cu).
//
// Lengths below 256 ran the run-time-parameter kernel, bound by its address
// arithmetic and, at 16 points (one transform per thread), by loads that touch
// a 128-byte line per lane.  Here a transform's first stage has at least four
// lanes, so every load fills whole 32-byte sectors, and memory is the bound.
// Four blocks per SM: five (96 registers) and six (80) measured 3% and 20%
// slower at 64 points and up, as for the joined kernels (L1).
// Measured, 2^26 elements, before and now: 8 points 297 -> 221 us, 16 516 -> 170,
// 32 333 -> 161, 64 213 -> 156, 128 201 -> 160 (2^26 elements of HBM: 160 us);
// 256 .. 1024 158 -> 158, 160 -> 160, 159 -> 160 there and one launch quantum
// less below 2^19 elements (6.2 -> 4.2 us), where 128-thread blocks of one
// exchange finish sooner.  Not 4 points (272 -> 283 us: two lanes per
// transform), nor 2048 and 4096 (166 -> 171, 164 -> 186: a third stage).
// Columns, both passes of frames, before (joined below 2^21 elements) and now:
// 2^20 elements of 512 x 2048 15.1 -> 8.7 us, of 256 x 256 11.5 -> 7.2; 2^25 of
// 64 x 64 242 -> 153.
#include "joined.cuh"

namespace gbfft {

template <int LOGL>
__global__ void __launch_bounds__(128, 4)
short_lines(const cf* __restrict__ in, cf* out, const __grid_constant__ PassDesc d) {
  extern __shared__ __align__(16) unsigned char smem_lines[];
  const int64_t tile = blockIdx.x, at = tile << 12;
  grid_wait();
  line_tile<LOGL>(in + at, out + at, d, d.count_inner - tile * (4096 >> LOGL),
                  reinterpret_cast<cf*>(smem_lines), threadIdx.x);
}

// The same for a coalesced launch (GroupTable): block t runs tile t of the jobs'
// tiles one after another, with the arithmetic of short_lines, so that a server
// job's bits do not depend on whether it was coalesced.
template <int LOGL>
__global__ void __launch_bounds__(128, 4)
grouped_lines(const __grid_constant__ PassDesc d, const __grid_constant__ GroupTable gt) {
  extern __shared__ __align__(16) unsigned char smem_lines[];
  int j = 0;
  while (j + 1 < gt.n && gt.e[j + 1].tile_begin <= blockIdx.x) ++j;
  const int64_t tile = blockIdx.x - gt.e[j].tile_begin, at = tile << 12;
  line_tile<LOGL>(gt.e[j].in + at, gt.e[j].out + at, d, gt.e[j].count - tile * (4096 >> LOGL),
                  reinterpret_cast<cf*>(smem_lines), threadIdx.x);
}

template <int LOGL>
static bool lines_fn(PassLaunch* l) {
  l->fn = (const void*)short_lines<LOGL>;
  l->smem = JoinBody<typename JoinLen<12, LOGL>::S, JOIN_ROWS, JoinMem>::kSlots * sizeof(cf);
  l->block = 128;
  l->lines = 12;
  return true;
}

// Columns of 2^LOGL rows of d.in.e elements, in place or not.
template <int TL, int LOGL>
__global__ void __launch_bounds__((1 << TL) / kJoinR, 1 << join_blocks_log(TL))
short_cols(const cf* in, cf* out, const __grid_constant__ PassDesc d) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_COLS, JoinMem>;
  extern __shared__ __align__(16) unsigned char smem_lines[];
  cf* sm = reinterpret_cast<cf*>(smem_lines);
  const int tid = threadIdx.x, lc = 31 - __clz((int)d.in.e);
  const int64_t col0 = (int64_t)blockIdx.x * B::G, cols = d.tiles / d.tiles_inner * d.count_inner;
  grid_wait();
  cf v[kJoinR];
  B::first_frame(v, in, col0, cols, lc, tid);
  join_stages<SH, JOIN_COLS, false>(v, sm, d.tw + d.tw_line, 0, 0, tid);
  if (d.conj_out) B::template store_frame<true>(v, out, col0, cols, lc, tid);
  else B::template store_frame<false>(v, out, col0, cols, lc, tid);
}

template <int TL, int LOGL>
static bool cols_fn(PassLaunch* l) {
  l->fn = (const void*)short_cols<TL, LOGL>;
  l->smem = JoinBody<typename JoinLen<TL, LOGL>::S, JOIN_COLS, JoinMem>::kSlots * sizeof(cf);
  l->block = (1 << TL) / kJoinR;
  l->lines = TL;
  return true;
}

bool resolve_cols(int logL, PassLaunch* l) {
  switch (logL) {
    case 3: return cols_fn<12, 3>(l);
    case 4: return cols_fn<12, 4>(l);
    case 5: return cols_fn<12, 5>(l);
    case 6: return cols_fn<12, 6>(l);
    case 7: return cols_fn<12, 7>(l);
    case 8: return cols_fn<12, 8>(l);
    case 9: return cols_fn<13, 9>(l);
    case 10: return cols_fn<13, 10>(l);
    case 11: return cols_fn<13, 11>(l);
    default: return false;
  }
}

bool resolve_lines(int logL, PassLaunch* l) {
  switch (logL) {
    case 3: return lines_fn<3>(l);
    case 4: return lines_fn<4>(l);
    case 5: return lines_fn<5>(l);
    case 6: return lines_fn<6>(l);
    case 7: return lines_fn<7>(l);
    case 8: return lines_fn<8>(l);
    case 9: return lines_fn<9>(l);
    case 10: return lines_fn<10>(l);
    default: return false;
  }
}

cudaError_t launch_grouped_lines(const PassLaunch& l, const GroupTable& gt, cudaStream_t st) {
  if (!l.lines || gt.n < 1 || gt.n > kMaxGroup) return cudaErrorInvalidValue;
  const int64_t tiles = gt.e[gt.n - 1].tile_begin + gt.e[gt.n - 1].tiles;
  if (tiles < 1 || tiles > 0x7fffffff) return cudaErrorInvalidValue;
  const void* f = nullptr;
  switch (l.d.logL) {
    case 3: f = (const void*)grouped_lines<3>; break;
    case 4: f = (const void*)grouped_lines<4>; break;
    case 5: f = (const void*)grouped_lines<5>; break;
    case 6: f = (const void*)grouped_lines<6>; break;
    case 7: f = (const void*)grouped_lines<7>; break;
    case 8: f = (const void*)grouped_lines<8>; break;
    case 9: f = (const void*)grouped_lines<9>; break;
    case 10: f = (const void*)grouped_lines<10>; break;
    default: return cudaErrorInvalidValue;
  }
  if (l.smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.smem);
    if (e != cudaSuccess) return e;
  }
  using GFn = void (*)(PassDesc, GroupTable);
  reinterpret_cast<GFn>(const_cast<void*>(f))<<<(int)tiles, l.block, l.smem, st>>>(l.d, gt);
  return cudaGetLastError();
}

}  // namespace gbfft
