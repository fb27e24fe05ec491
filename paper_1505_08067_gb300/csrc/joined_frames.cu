// Joined row and column passes of 2D frames (joined.cuh).
#include "joined.cuh"

namespace gbfft {

void joined_frames_kernel(int tile_log, bool inv, JoinedLaunch& j) {
  if (tile_log == 12) joined_frames_fn<12>(inv, j);
  else joined_frames_fn<13>(inv, j);
}

}  // namespace gbfft
