// Two-pass kernels, joined and apart, of 2^18 .. 2^20 points (joined.cuh), and the
// launches.
#include <algorithm>

#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, bool apart, bool inv, JoinedLaunch& j);
void joined_frames_kernel(int tile_log, bool inv, JoinedLaunch& j);

static bool joined_kernel_b(int logn, bool apart, bool inv, JoinedLaunch& j) {
  switch (logn) {
    case 18: return apart ? apart_fn<18, join_tile_log(18, true)>(inv, j) : joined_fn<18, join_tile_log(18, false)>(inv, j);
    case 19: return apart ? apart_fn<19, join_tile_log(19, true)>(inv, j) : joined_fn<19, join_tile_log(19, false)>(inv, j);
    case 20: return apart ? apart_fn<20, join_tile_log(20, true)>(inv, j) : joined_fn<20, join_tile_log(20, false)>(inv, j);
    default: return false;
  }
}

static cudaError_t prepare(int sm_count, JoinedLaunch* j) {
  cudaError_t e =
      cudaFuncSetAttribute(j->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)j->smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, j->fn, j->block, j->smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  j->max_grid = per_sm * sm_count;
  return cudaSuccess;
}

cudaError_t prepare_joined(int logn, bool apart, bool inv, int sm_count, JoinedLaunch* j) {
  if (!joined_kernel_a(logn, apart, inv, *j) && !joined_kernel_b(logn, apart, inv, *j))
    return cudaErrorInvalidValue;
  j->tile_log = join_tile_log(logn, apart);
  if (!apart) return prepare(sm_count, j);
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(j->fn, attr, (int)j->smem);
  return e == cudaSuccess ? cudaFuncSetAttribute(j->second, attr, (int)j->second_smem) : e;
}

cudaError_t prepare_joined_frames(int lr, int lc, int tl, bool inv, int sm_count,
                                  JoinedLaunch* j) {
  if (!join_frame(lr, lc, int64_t(1) << 40) || tl != join_frame_tile_log(lr)) return cudaErrorInvalidValue;
  joined_frames_kernel(tl, inv, *j);
  j->frames = true;
  j->tile_log = tl;
  j->d.lr = lr;
  j->d.lc = lc;
  j->d.o.tpt_log = std::max(0, lr + lc - tl);
  return prepare(sm_count, j);
}

cudaError_t launch_joined(const JoinedLaunch& j, int64_t batch, const void* in, void* out,
                          void* work, cudaStream_t st) {
  if (!j.fn || batch < 1) return cudaErrorInvalidValue;
  JoinDesc d = j.d;
  d.o.nb = batch;
  if (j.second) {
    const int64_t tiles = batch << d.o.tpt_log;
    if (tiles > 0x7fffffff) return cudaErrorInvalidValue;
    const cudaError_t e = launch_early(j.fn, (int)tiles, j.block, j.smem, st,
                                       static_cast<const cf*>(in), static_cast<cf*>(work), d);
    if (e != cudaSuccess) return e;
    return launch_early(j.second, (int)tiles, j.block, j.second_smem, st,
                        static_cast<const cf*>(work), static_cast<cf*>(out), d);
  }
  if (j.frames) {
    d.total = batch << (d.lr + d.lc);
    const int unit = j.tile_log + d.o.tpt_log;
    d.o.nb = (d.total + (int64_t(1) << unit) - 1) >> unit;
    d.mapped = ((uintptr_t)in & 15) == 0;
  } else {
    d.mapped = encode_rows_map(in, j.n2, batch * j.n1, j.g1, j.box_rows, d.tmap_in);
  }
  d.o.lag = std::min<int64_t>(d.o.lag, d.o.nb << d.o.tpt_log);
  const int grid = (int)std::min<int64_t>(j.max_grid, join_tickets(d.o));
  const cf* ci = static_cast<const cf*>(in);
  cf* co = static_cast<cf*>(out);
  if (j.frames) return launch_early(j.fn, grid, j.block, j.smem, st, ci, co, d);
  return launch_early(j.fn, grid, j.block, j.smem, st, ci, co, static_cast<cf*>(work), d);
}

}  // namespace gbfft
