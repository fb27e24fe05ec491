// Joined kernels of transforms of 2^15 .. 2^17 points (joined.cuh).
#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, int tile_log, bool inv, JoinedLaunch& j) {
  switch (logn * 100 + tile_log) {
    case 1512: return joined_fn<15, 12>(inv, j);
    case 1612: return joined_fn<16, 12>(inv, j);
    case 1712: return joined_fn<17, 12>(inv, j);
    case 1713: return joined_fn<17, 13>(inv, j);
    default: return false;
  }
}

}  // namespace gbfft
