// Joined two-pass kernels of 2^15 .. 2^18 points (joined.cuh).
#include "joined.cuh"

namespace gbfft {

bool joined_kernel_a(int logn, bool inv, JoinedLaunch& j) {
  switch (logn) {
    case 15: joined_fn<15>(inv, j); return true;
    case 16: joined_fn<16>(inv, j); return true;
    case 17: joined_fn<17>(inv, j); return true;
    case 18: joined_fn<18>(inv, j); return true;
    default: return false;
  }
}

}  // namespace gbfft
