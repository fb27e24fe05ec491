// Two-pass kernels, joined and apart, of transforms of 2^15 .. 2^17 points (joined.cuh).
#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, bool apart, bool inv, JoinedLaunch& j) {
  switch (logn) {
    case 15: return apart ? apart_fn<15, join_tile_log(15, true)>(inv, j) : joined_fn<15, join_tile_log(15, false)>(inv, j);
    case 16: return apart ? apart_fn<16, join_tile_log(16, true)>(inv, j) : joined_fn<16, join_tile_log(16, false)>(inv, j);
    case 17: return apart ? apart_fn<17, join_tile_log(17, true)>(inv, j) : joined_fn<17, join_tile_log(17, false)>(inv, j);
    default: return false;
  }
}

}  // namespace gbfft
