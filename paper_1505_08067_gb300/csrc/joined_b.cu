// Joined two-pass kernels of 2^19 and 2^20 points (joined.cuh), and the launch.
#include <algorithm>

#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, bool inv, JoinedLaunch& j);

static bool joined_kernel_b(int logn, bool inv, JoinedLaunch& j) {
  switch (logn) {
    case 19: joined_fn<19>(inv, j); return true;
    case 20: joined_fn<20>(inv, j); return true;
    default: return false;
  }
}

cudaError_t prepare_joined(int logn, bool inv, int sm_count, JoinedLaunch* j) {
  if (!joined_kernel_a(logn, inv, *j) && !joined_kernel_b(logn, inv, *j))
    return cudaErrorInvalidValue;
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

cudaError_t launch_joined(const JoinedLaunch& j, int64_t nb, const void* in, void* out, void* work,
                          cudaStream_t st) {
  using Fn = void (*)(const cf*, cf*, cf*, JoinDesc);
  if (!j.fn || nb < 1) return cudaErrorInvalidValue;
  JoinDesc d = j.d;
  d.o.nb = nb;
  d.o.lag = (int32_t)std::min<int64_t>(d.o.lag, nb);
  d.mapped = encode_rows_map(in, j.n2, nb * j.n1, j.g1, j.box_rows, d.tmap_in);
  const int grid = (int)std::min<int64_t>(j.max_grid, join_tickets(d.o));
  reinterpret_cast<Fn>(const_cast<void*>(j.fn))<<<grid, j.block, j.smem, st>>>(
      static_cast<const cf*>(in), static_cast<cf*>(out), static_cast<cf*>(work), d);
  return cudaGetLastError();
}

}  // namespace gbfft
