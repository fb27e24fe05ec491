// Joined two-pass kernels of 2^19 and 2^20 points (joined.cuh), and the launch.
#include <algorithm>

#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, bool inv, JoinedLaunch& j);
void joined_frames_kernel(int tile_log, bool inv, JoinedLaunch& j);

static bool joined_kernel_b(int logn, bool inv, JoinedLaunch& j) {
  switch (logn) {
    case 19: joined_fn<19>(inv, j); return true;
    case 20: joined_fn<20>(inv, j); return true;
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

cudaError_t prepare_joined(int logn, bool inv, int sm_count, JoinedLaunch* j) {
  if (!joined_kernel_a(logn, inv, *j) && !joined_kernel_b(logn, inv, *j))
    return cudaErrorInvalidValue;
  return prepare(sm_count, j);
}

cudaError_t prepare_joined_frames(int lr, int lc, bool inv, int sm_count, JoinedLaunch* j) {
  if (!join_frame(lr, lc)) return cudaErrorInvalidValue;
  const int tl = join_frame_tile_log(lr, lc);
  joined_frames_kernel(tl, inv, *j);
  j->frames = true;
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
  if (j.frames) {
    d.total = batch << (d.lr + d.lc);
    const int tl = join_frame_tile_log(d.lr, d.lc);
    d.o.nb = (d.total + (int64_t(1) << (tl + d.o.tpt_log)) - 1) >> (tl + d.o.tpt_log);
    d.mapped = ((uintptr_t)in & 15) == 0;
  } else {
    d.mapped = encode_rows_map(in, j.n2, batch * j.n1, j.g1, j.box_rows, d.tmap_in);
  }
  d.o.lag = std::min<int64_t>(d.o.lag, d.o.nb << d.o.tpt_log);
  const int grid = (int)std::min<int64_t>(j.max_grid, join_tickets(d.o));
  const cf* ci = static_cast<const cf*>(in);
  cf* co = static_cast<cf*>(out);
  if (j.frames) {
    using Fn = void (*)(const cf*, cf*, JoinDesc);
    reinterpret_cast<Fn>(const_cast<void*>(j.fn))<<<grid, j.block, j.smem, st>>>(ci, co, d);
  } else {
    using Fn = void (*)(const cf*, cf*, cf*, JoinDesc);
    reinterpret_cast<Fn>(const_cast<void*>(j.fn))<<<grid, j.block, j.smem, st>>>(
        ci, co, static_cast<cf*>(work), d);
  }
  return cudaGetLastError();
}

}  // namespace gbfft
