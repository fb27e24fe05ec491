// The joined two-pass kernel: both passes of a four-step transform of
// N = 2^15 .. 2^20 points in one persistent launch (bodies, tile order and
// workspace layout: fft_join.h).
//
// What bounds the two launches it replaces: not HBM but the SMs.  With every
// tile's input and output in L2 they took almost the time they take from HBM
// (2^18 x 256: 379 against 446 us, 2^20 x 64: 358 against 368 us): two
// shared-memory exchanges, in the longer passes in half-buffer rounds with
// eight barriers per tile.  Here a tile crosses shared memory once, and the
// order of the tiles keeps the intermediate in L2 (ncu, 2^18 x 64: 278 MB read and
// written in DRAM, input and output being 268 MB, where two launches move twice
// that).
//
// What bounds this kernel: the first pass (2^26 elements, 512 points: 161 us
// alone, the second 135), by latency -- issue 38% busy, FMA pipe 36%, DRAM 47%.
// More warps do not help: 3 blocks per SM of 80 registers measured 328 against
// 293 us (2^17), because a column load keeps a 128-byte line of L1 per row
// segment in flight and shared memory leaves little L1 (the same kernel with
// the smallest L1: 1.15-1.3 times the time).  Hence direct loads for the wide
// tiles (staging them by TMA into the exchange buffer measured 350 against
// 305 us at 2^18), 128-byte row segments where the tile allows (2^20: 16
// columns in one 512-thread block per SM, 336 us, against 8 columns in two
// blocks, 352 us) and smaller blocks where segments stay wide (2^15, 2^16:
// four 128-thread blocks, 242 / 245 us).
//
// Smaller batches run the same passes in a launch each (apart_first,
// apart_second; join_apart says where the line lies), and so do server jobs and
// fft_execute_noalloc at every size: that form needs no counters.
// Measured, 2^26 elements, before (two launches) and now: 2^15 349 -> 242 us,
// 2^16 363 -> 245, 2^17 396 -> 275, 2^18 446 -> 289, 2^19 421 -> 302,
// 2^20 368 -> 330.  2^21 and 2^22, whose 2048-point passes need three stages and
// 64-byte segments, measured slower joined (384 against 371 us, 592 against 387).
#pragma once
#include <cuda_runtime.h>

#include "fft_join.h"
#include "kernels_impl.cuh"

namespace gbfft {

struct JoinMem : DevMem {
  __device__ __forceinline__ static cf ldin(const cf* p, int off) {
    const float2 r = __ldcs(reinterpret_cast<const float2*>(p) + off);
    return mk(r.x, r.y);
  }
  // The workspace is written by other SMs during the kernel and its slots are
  // reused: L2 only, never a line of this SM's L1.
  __device__ __forceinline__ static cf ldw(const cf* p, int off) {
    const float2 r = __ldcg(reinterpret_cast<const float2*>(p) + off);
    return mk(r.x, r.y);
  }
  __device__ __forceinline__ static void stw(cf* p, int off, cf v) {
    __stcg(reinterpret_cast<float2*>(p) + off, make_float2(v.x, v.y));
  }
  __device__ __forceinline__ static void stout(cf* p, int off, cf v) {
    __stcs(reinterpret_cast<float2*>(p) + off, make_float2(v.x, v.y));
  }
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Finished-tile counters (JoinDesc::ctr): [0] tickets handed out, [1] blocks
// that have left, then per pass and ring slot the tiles finished.  All zero
// between launches: the last block to leave clears them.  A whole launch hands out
// one ticket per tile and one more per block, and as many blocks leave as it has.
// A block that gets a later ticket, or leaves after them, reports kStatusCounters:
// another execution of the plan drew on the counters meanwhile, which the plan's
// contract forbids and which would otherwise pass unseen, here and in the launches
// that find the counters it left.  (Comparing every counter before clearing it
// costs 1 to 4.7 us a launch; this costs nothing.)
__device__ __forceinline__ unsigned* join_done(const JoinDesc& d, int pass, int slot) {
  return d.ctr + 2 + pass * d.o.ring + slot;
}

// A barrier of the T computing threads only (the last warp does not take part).
template <int T>
__device__ __forceinline__ void join_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; "
      "selp.u32 %0, 1, 0, p; }"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done;
}

// The kernel's last warp hands out the tiles.  While the others work on one it
// raises the count of the tile before (the release waits for that tile's stores
// to reach L2; nobody else has to), takes the next ticket, waits for what that
// depends on and prepares it.  A wait may be for this block's own tile, so it
// raises that as soon as it is stored.  prefetch(k): one thread, as early as
// possible; prepare(k, set): the warp, for the tile after the one at work.
template <class Prefetch, class Prepare>
__device__ __forceinline__ void join_dispatch(const JoinDesc& d, uint64_t* stored,
                                              unsigned* s_ticket, int lane, Prefetch prefetch,
                                              Prepare prepare) {
  const unsigned total = (unsigned)join_tickets(d.o);
  unsigned* finished = nullptr;
  bool foreign = false;
  for (int n = 0;; ++n) {
    unsigned t = 0;
    if (lane == 0) {
      t = atomicAdd(d.ctr, 1u);
      foreign = t >= total && t - total >= gridDim.x;
      if (t < total) {
        const JoinTicket k = join_ticket(d.o, t);
        if (k.pass == 0) prefetch(k);
        const JoinDep dep = join_dep(d.o, k);
        const unsigned* c = join_done(d, dep.pass, dep.slot);
        bool ok = dep.count == 0;
        for (uint32_t it = 0; it < d.polls && !ok; ++it) {
          ok = ld_acquire_gpu(c) >= dep.count;
          if (!ok && finished && mbar_test(stored, (n - 1) & 1)) {
            red_release_gpu(finished);
            finished = nullptr;
          }
          if (!ok && it > 16) __nanosleep(64);
        }
        if (!ok) {
          atomicOr(d.status, kStatusGaveUp);
          t = total;
        }
      }
      s_ticket[n & 1] = t;
    }
    t = __shfl_sync(~0u, t, 0);
    const JoinTicket k = join_ticket(d.o, t < total ? t : 0);
    if (t < total) prepare(k, n & 1);
    __syncthreads();  // the tile before is stored, this one may start
    if (lane == 0 && finished) red_release_gpu(finished);
    if (t >= total) break;
    finished = join_done(d, k.pass, (int)(k.b % d.o.ring));
  }
  unsigned last = 0;
  if (lane == 0) {
    __threadfence();
    const unsigned left = atomicAdd(d.ctr + 1, 1u);
    last = left == gridDim.x - 1;
    if (foreign || left >= gridDim.x) atomicOr(d.status, kStatusCounters);
  }
  if (__shfl_sync(~0u, last, 0))
    for (int i = lane; i < 2 + 2 * d.o.ring; i += 32) d.ctr[i] = 0;
}

// The other warps: tile(k, set) for every ticket the last warp publishes.
template <class Tile>
__device__ __forceinline__ void join_work(const JoinDesc& d, uint64_t* stored,
                                          const unsigned* s_ticket, int tid, Tile tile) {
  const unsigned total = (unsigned)join_tickets(d.o);
  for (int n = 0;; ++n) {
    __syncthreads();  // every thread has read the last tile's shared memory
    const unsigned t = s_ticket[n & 1];
    if (t >= total) break;
    tile(join_ticket(d.o, t), n & 1);
    __syncwarp();
    if ((tid & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(stored)) : "memory");
  }
}

// The stages of a tile between its loads and its stores; TW4 as JoinBody::turn.
template <class SH, int KIND, bool TW4>
__device__ __forceinline__ void join_stages(cf (&v)[kJoinR], cf* sm, const cf* tw, int col0,
                                            int logN, int tid) {
  using B = JoinBody<SH, KIND, JoinMem>;
  B::dft0(v);
  B::template put<0>(v, sm, tid);
  join_sync<SH::kThreads>();
  if constexpr (SH::kNst == 3) {
    B::template get<1>(v, sm, tid);
    B::template turn<1, false>(v, tw, 0, 0, tid);
    join_sync<SH::kThreads>();
    B::template put<1>(v, sm, tid);
    join_sync<SH::kThreads>();
  }
  B::template get<SH::kLast>(v, sm, tid);
  B::template turn<SH::kLast, TW4>(v, tw, col0, logN, tid);
}

// A tile of 4096 elements of contiguous lines of 2^LOGL points, `valid` of them.
template <int LOGL>
__device__ __forceinline__ void line_tile(const cf* in, cf* out, const PassDesc& d, int64_t valid,
                                          cf* sm, int tid) {
  using SH = typename JoinLen<12, LOGL>::S;
  using B = JoinBody<SH, JOIN_ROWS, JoinMem>;
  cf v[kJoinR];
  if (d.conj_in) B::template first_rows<true>(v, in, valid, tid);
  else B::template first_rows<false>(v, in, valid, tid);
  join_stages<SH, JOIN_ROWS, false>(v, sm, d.tw + d.tw_line, 0, 0, tid);
  if (d.conj_out) B::template store_rows<true>(v, out, valid, tid);
  else B::template store_rows<false>(v, out, valid, tid);
}

// Both rounds of a fast convolution: forward stages, filter, the stages in
// reverse order on swapped data (the unnormalised inverse).
template <class SH, int KIND>
__device__ __forceinline__ void join_conv(cf (&v)[kJoinR], cf* sm, const cf* tw, const cf* h,
                                          int64_t lines, int64_t first, float scale, int tid) {
  join_stages<SH, KIND, false>(v, sm, tw, 0, 0, tid);
  JoinBody<SH, KIND, JoinMem>::filter(v, h, lines, first, scale, tid);
  join_sync<SH::kThreads>();  // every thread has read the last exchange
  join_stages<typename JoinReverse<SH>::S, KIND, false>(v, sm, tw, 0, 0, tid);
}
template <class SH, int KIND>
constexpr int join_conv_slots() {
  constexpr int a = JoinBody<SH, KIND, JoinMem>::kSlots;
  constexpr int b = JoinBody<typename JoinReverse<SH>::S, KIND, JoinMem>::kSlots;
  return a > b ? a : b;
}

// Four-step transforms of 2^LOGN points.
template <int LOGN, int TL, bool INV>
__global__ void __launch_bounds__((1 << TL) / kJoinR + 32, 1 << join_blocks_log(TL))
joined_pass(const cf* in, cf* out, cf* work, const __grid_constant__ JoinDesc d) {
  using PR = JoinPair<LOGN, TL>;
  using B1 = JoinBody<typename PR::P1, JOIN_FIRST, JoinMem>;
  using B2 = JoinBody<typename PR::P2, JOIN_COLS, JoinMem>;
  constexpr int T = PR::kThreads;
  constexpr int kSlots = B1::kSlots > B2::kSlots ? B1::kSlots : B2::kSlots;
  extern __shared__ __align__(16) unsigned char smem_join[];
  cf* sm = reinterpret_cast<cf*>(smem_join);
  cf* steps = sm + kSlots;     // two sets
  __shared__ uint64_t stored;  // completes a phase when a tile's stores are issued
  __shared__ unsigned s_ticket[2];
  const int tid = threadIdx.x;
  if (tid == 0) mbar_init(&stored, T / 32);
  __syncthreads();
  grid_wait();
  if (tid >= T) {
    join_dispatch(
        d, &stored, s_ticket, tid - T,
        [&](const JoinTicket& k) {  // the tile's columns, asynchronously into L2
          if (!d.mapped) return;
          constexpr int BR = PR::kN1 < 256 ? PR::kN1 : 256;
          const uint64_t map = reinterpret_cast<uint64_t>(&d.tmap_in[0]);
#pragma unroll 1
          for (int j = 0; j < PR::kN1 / BR; ++j)
            asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map),
                         "r"(k.tile * PR::kG1), "r"((int)(k.b * PR::kN1) + j * BR)
                         : "memory");
        },
        [&](const JoinTicket& k, int set) {
          if (k.pass == 0) B1::steps(steps + set * PR::kSteps, k.tile * PR::kG1, LOGN, tid - T);
        });
    return;
  }
  join_work(d, &stored, s_ticket, tid, [&](const JoinTicket& k, int set) {
    cf* w = work + (int64_t)(k.b % d.o.ring) * PR::kN;
    cf v[kJoinR];
    if (k.pass == 0) {
      const int col0 = k.tile * PR::kG1;
      B1::template first<INV, false>(v, in + k.b * PR::kN + col0, PR::kN2, tid);
      join_stages<typename PR::P1, JOIN_FIRST, true>(v, sm, d.tw1, col0, LOGN, tid);
      B1::template store_block<PR::kG2>(v, w + col0 * PR::kG2, steps + set * PR::kSteps, PR::kN2,
                                        tid);
    } else {
      B2::template first<false, true>(v, w + k.tile * PR::kTile, PR::kG2, tid);
      join_stages<typename PR::P2, JOIN_COLS, false>(v, sm, d.tw2, 0, 0, tid);
      B2::template store_cols<INV>(v, out + k.b * PR::kN + k.tile * PR::kG2, PR::kN1, tid);
    }
  });
}

// The same passes in a launch each, a tile per block: transform b's intermediate
// at work + b N.
template <int LOGN, int TL, bool INV>
__global__ void __launch_bounds__((1 << TL) / kJoinR, 1 << join_blocks_log(TL))
apart_first(const cf* in, cf* work, const __grid_constant__ JoinDesc d) {
  using PR = JoinPair<LOGN, TL>;
  using B = JoinBody<typename PR::P1, JOIN_FIRST, JoinMem>;
  extern __shared__ __align__(16) unsigned char smem_join[];
  cf* sm = reinterpret_cast<cf*>(smem_join);
  cf* steps = sm + B::kSlots;
  const int tid = threadIdx.x, col0 = (int)(blockIdx.x & (PR::kTiles - 1)) * PR::kG1;
  const int64_t at = (int64_t)(blockIdx.x / PR::kTiles) * PR::kN;
  B::steps(steps, col0, LOGN, tid, PR::kThreads);
  grid_wait();
  cf v[kJoinR];
  B::template first<INV, false>(v, in + at + col0, PR::kN2, tid);
  join_stages<typename PR::P1, JOIN_FIRST, true>(v, sm, d.tw1, col0, LOGN, tid);
  B::template store_block<PR::kG2>(v, work + at + col0 * PR::kG2, steps, PR::kN2, tid);
}
template <int LOGN, int TL, bool INV>
__global__ void __launch_bounds__((1 << TL) / kJoinR, 1 << join_blocks_log(TL))
apart_second(const cf* work, cf* out, const __grid_constant__ JoinDesc d) {
  using PR = JoinPair<LOGN, TL>;
  using B = JoinBody<typename PR::P2, JOIN_COLS, JoinMem>;
  extern __shared__ __align__(16) unsigned char smem_join[];
  cf* sm = reinterpret_cast<cf*>(smem_join);
  const int tid = threadIdx.x, tile = (int)(blockIdx.x & (PR::kTiles - 1));
  const int64_t at = (int64_t)(blockIdx.x / PR::kTiles) * PR::kN;
  grid_wait();
  cf v[kJoinR];
  B::template first<false, true>(v, work + at + tile * PR::kTile, PR::kG2, tid);
  join_stages<typename PR::P2, JOIN_COLS, false>(v, sm, d.tw2, 0, 0, tid);
  B::template store_cols<INV>(v, out + at + tile * PR::kG2, PR::kN1, tid);
}

// One tile of rows (from in to out) or of columns (in place) of frames.
template <int TL, int LOGL, bool INV>
__device__ __forceinline__ void join_rows(const cf* in, cf* out, const JoinDesc& d, int64_t tile,
                                          cf* sm, int tid) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_ROWS, JoinMem>;
  const int64_t valid = (d.total >> LOGL) - tile * B::G;
  cf v[kJoinR];
  B::template first_rows<INV>(v, in + (tile << TL), valid, tid);
  join_stages<SH, JOIN_ROWS, false>(v, sm, d.tw1, 0, 0, tid);
  B::store_rows(v, out + (tile << TL), valid, tid);
}
template <int TL, int LOGL, bool INV>
__device__ __forceinline__ void join_cols(cf* buf, const JoinDesc& d, int64_t tile, cf* sm,
                                          int tid) {
  using SH = typename JoinLen<TL, LOGL>::S;
  using B = JoinBody<SH, JOIN_COLS, JoinMem>;
  cf v[kJoinR];
  B::first_frame(v, buf, tile * B::G, d.total >> LOGL, d.lc, tid);
  join_stages<SH, JOIN_COLS, false>(v, sm, d.tw2, 0, 0, tid);
  B::template store_frame<INV>(v, buf, tile * B::G, d.total >> LOGL, d.lc, tid);
}

// 2D frames of 2^lr rows of 2^lc elements: row pass from in to out, column pass
// in out.  One kernel for all lengths (a block uses two of the bodies below):
// the column passes had compile-time shapes for 4096 rows only, and the
// run-time-parameter kernel is bound by its address arithmetic and its load
// queue.  Column passes read 64 bytes per row at 1024 rows and 32 at 2048;
// 4096 rows and more (16 bytes) keep the staged column kernel and its tensor-map
// loads.  Tiles of 4096 elements up to 256 rows (measured as for transforms
// above), else 8192.
// Measured, 2^25 elements, before (a launch per pass), now a launch per pass
// (lines.cu), and joined: 16 x 16 390, 158, 136 us, 64 x 64 242, 153, 120,
// 256 x 1024 201, 159, 143, 512 x 1024 245, 166, 149, 1024 x 1024 271, 182, 158,
// 2048 x 1024 272, 215, 206.
template <int TL, bool INV>
__global__ void __launch_bounds__((1 << TL) / kJoinR + 32, 1 << join_blocks_log(TL))
joined_frames(const cf* in, cf* out, const __grid_constant__ JoinDesc d) {
  constexpr int T = (1 << TL) / kJoinR;
  extern __shared__ __align__(16) unsigned char smem_join[];
  cf* sm = reinterpret_cast<cf*>(smem_join);
  __shared__ uint64_t stored;
  __shared__ unsigned s_ticket[2];
  const int tid = threadIdx.x;
  if (tid == 0) mbar_init(&stored, T / 32);
  __syncthreads();
  grid_wait();
  if (tid >= T) {
    join_dispatch(
        d, &stored, s_ticket, tid - T,
        [&](const JoinTicket& k) {
          if (!d.mapped) return;
          const int64_t at = (((k.b << d.o.tpt_log) + k.tile)) << TL;
          const int64_t n = d.total - at < (1 << TL) ? d.total - at : (1 << TL);
          if (n > 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(in + at),
                         "r"((unsigned)n * 8)
                         : "memory");
        },
        [](const JoinTicket&, int) {});
    return;
  }
  join_work(d, &stored, s_ticket, tid, [&](const JoinTicket& k, int) {
    const int64_t tile = (k.b << d.o.tpt_log) + k.tile;
    if (k.pass == 0) {
      switch (d.lc) {
        case 4: join_rows<TL, 4, INV>(in, out, d, tile, sm, tid); break;
        case 5: join_rows<TL, 5, INV>(in, out, d, tile, sm, tid); break;
        case 6: join_rows<TL, 6, INV>(in, out, d, tile, sm, tid); break;
        case 7: join_rows<TL, 7, INV>(in, out, d, tile, sm, tid); break;
        case 8: join_rows<TL, 8, INV>(in, out, d, tile, sm, tid); break;
        case 9: join_rows<TL, 9, INV>(in, out, d, tile, sm, tid); break;
        case 10: join_rows<TL, 10, INV>(in, out, d, tile, sm, tid); break;
        default: break;
      }
    } else {
      switch (d.lr) {
        case 4: join_cols<TL, 4, INV>(out, d, tile, sm, tid); break;
        case 5: join_cols<TL, 5, INV>(out, d, tile, sm, tid); break;
        case 6: join_cols<TL, 6, INV>(out, d, tile, sm, tid); break;
        case 7: join_cols<TL, 7, INV>(out, d, tile, sm, tid); break;
        case 8: join_cols<TL, 8, INV>(out, d, tile, sm, tid); break;
        default:
          if constexpr (TL >= 13) {
            if (d.lr == 9) join_cols<TL, 9, INV>(out, d, tile, sm, tid);
            else if (d.lr == 10) join_cols<TL, 10, INV>(out, d, tile, sm, tid);
            else join_cols<TL, 11, INV>(out, d, tile, sm, tid);
          }
          break;
      }
    }
  });
}

template <int LOGN, int TL>
inline bool joined_fn(bool inv, JoinedLaunch& j) {
  using PR = JoinPair<LOGN, TL>;
  constexpr int s1 = JoinBody<typename PR::P1, JOIN_FIRST, JoinMem>::kSlots;
  constexpr int s2 = JoinBody<typename PR::P2, JOIN_COLS, JoinMem>::kSlots;
  j.fn = inv ? (const void*)joined_pass<LOGN, TL, true> : (const void*)joined_pass<LOGN, TL, false>;
  j.smem = ((s1 > s2 ? s1 : s2) + 2 * PR::kSteps) * sizeof(cf);
  j.block = PR::kThreads + 32;
  j.d.o.tpt_log = LOGN - TL;
  j.n1 = PR::kN1;
  j.n2 = PR::kN2;
  j.g1 = PR::kG1;
  j.box_rows = PR::kN1 < 256 ? PR::kN1 : 256;
  return true;
}
template <int LOGN, int TL>
inline bool apart_fn(bool inv, JoinedLaunch& j) {
  using PR = JoinPair<LOGN, TL>;
  j.fn = inv ? (const void*)apart_first<LOGN, TL, true> : (const void*)apart_first<LOGN, TL, false>;
  j.second = inv ? (const void*)apart_second<LOGN, TL, true> : (const void*)apart_second<LOGN, TL, false>;
  j.smem = (JoinBody<typename PR::P1, JOIN_FIRST, JoinMem>::kSlots + PR::kSteps) * sizeof(cf);
  j.second_smem = JoinBody<typename PR::P2, JOIN_COLS, JoinMem>::kSlots * sizeof(cf);
  j.block = PR::kThreads;
  j.d.o.tpt_log = LOGN - TL;
  return true;
}

// Shared memory of the frame kernels: the largest tile of their bodies.
template <int TL, int LOGL, int TOP>
constexpr int join_frame_slots() {
  using SH = typename JoinLen<TL, LOGL>::S;
  constexpr int rows = JoinBody<SH, JOIN_ROWS, JoinMem>::kSlots;
  constexpr int cols = JoinBody<SH, JOIN_COLS, JoinMem>::kSlots;
  constexpr int here = rows > cols ? rows : cols;
  if constexpr (LOGL == TOP) return here;
  else return here > join_frame_slots<TL, LOGL + 1, TOP>() ? here : join_frame_slots<TL, LOGL + 1, TOP>();
}
template <int TL>
inline void joined_frames_fn(bool inv, JoinedLaunch& j) {
  j.fn = inv ? (const void*)joined_frames<TL, true> : (const void*)joined_frames<TL, false>;
  j.smem = join_frame_slots<TL, 4, 11>() * sizeof(cf);
  j.block = (1 << TL) / kJoinR + 32;
}

}  // namespace gbfft
