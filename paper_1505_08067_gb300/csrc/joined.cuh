// The joined two-pass kernel: both passes of a four-step transform of
// N = 2^15 .. 2^20 points in one persistent launch (bodies, tile order and
// workspace layout: fft_join.h).
//
// What bounds the two launches it replaces: not HBM but the SMs.  With every
// tile's input and output in L2 they took almost the time they take from HBM
// (2^18 x 256: 379 against 446 us, 2^20 x 64: 358 against 368 us): two
// shared-memory exchanges, in the longer passes in half-buffer rounds with
// eight barriers per tile.  Here a tile crosses shared memory once, and the
// order of the tiles keeps the intermediate in L2 (ncu, 2^18 x 64: DRAM reads
// equal to the input, DRAM writes 1.3 times the output, where two launches
// move twice both).
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
// Measured, 2^26 elements, before (two launches) and now: 2^15 349 -> 242 us,
// 2^16 363 -> 245, 2^17 396 -> 275, 2^18 446 -> 289, 2^19 421 -> 302,
// 2^20 368 -> 336; 2^21 elements 18.8-24.9 -> 18.7-22.3 us.  Below 2^21 elements
// the tiles no longer fill the GPU and two launches of smaller tiles are
// faster (2^20 elements: 14.3-18.3 against 16.6-20.7 us).  2^21 and 2^22, whose
// 2048-point passes need three stages and 64-byte segments, measured slower
// joined (384 against 371 us, 592 against 387 us).
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

constexpr uint32_t kJoinPolls = 1u << 21;  // about a second before a wait gives up

// Finished-tile counters (JoinDesc::ctr): [0] tickets handed out, [1] blocks
// that have left, then per pass and ring slot the tiles finished.  All zero
// between launches: the last block to leave clears them.
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

// Brings a first-pass tile's input into L2 (one thread; asynchronous).
template <class PR>
__device__ __forceinline__ void join_prefetch(const JoinDesc& d, const JoinTicket& k) {
  constexpr int BR = PR::kN1 < 256 ? PR::kN1 : 256;
  const uint64_t map = reinterpret_cast<uint64_t>(&d.tmap_in[0]);
#pragma unroll 1
  for (int j = 0; j < PR::kN1 / BR; ++j)
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(map),
                 "r"(k.tile * PR::kG1), "r"((int)(k.b * PR::kN1) + j * BR)
                 : "memory");
}

template <int LOGN, bool INV>
__global__ void __launch_bounds__(JoinPair<LOGN>::kThreads + 32, 1 << join_blocks_log(JoinPair<LOGN>::kTileLog))
joined_pass(const cf* in, cf* out, cf* work, const __grid_constant__ JoinDesc d) {
  using PR = JoinPair<LOGN>;
  using B1 = JoinBody<typename PR::P1, true, JoinMem>;
  using B2 = JoinBody<typename PR::P2, false, JoinMem>;
  constexpr int T = PR::kThreads;
  extern __shared__ __align__(16) unsigned char smem_join[];
  cf* sm = reinterpret_cast<cf*>(smem_join);
  cf* steps = sm + PR::kTileSlots;  // two sets
  __shared__ uint64_t stored;       // completes a phase when a tile's stores are issued
  __shared__ unsigned s_ticket[2];
  const int tid = threadIdx.x;
  const unsigned total = (unsigned)join_tickets(d.o);
  if (tid == 0) mbar_init(&stored, T / 32);
  __syncthreads();

  if (tid >= T) {
    // The last warp hands out the tiles.  While the others work on one it
    // raises the count of the tile before (the release waits for that tile's
    // stores to reach L2; nobody else has to), takes the next ticket, waits for
    // what that depends on and computes its steps.  A wait may be for this
    // block's own tile, so it raises that as soon as it is stored.
    const int lane = tid - T;
    unsigned* finished = nullptr;
    for (int n = 0;; ++n) {
      unsigned t = 0;
      if (lane == 0) {
        t = atomicAdd(d.ctr, 1u);
        if (t < total) {
          const JoinTicket k = join_ticket(d.o, t);
          if (k.pass == 0 && d.mapped) join_prefetch<PR>(d, k);
          const JoinDep dep = join_dep(d.o, k);
          const unsigned* c = join_done(d, dep.pass, dep.slot);
          bool ok = dep.count == 0;
          for (uint32_t it = 0; it < kJoinPolls && !ok; ++it) {
            ok = ld_acquire_gpu(c) >= dep.count;
            if (!ok && finished && mbar_test(&stored, (n - 1) & 1)) {
              red_release_gpu(finished);
              finished = nullptr;
            }
            if (!ok && it > 16) __nanosleep(64);
          }
          if (!ok) {
            atomicExch(d.status, 1);
            t = total;
          }
        }
        s_ticket[n & 1] = t;
      }
      t = __shfl_sync(~0u, t, 0);
      const JoinTicket k = join_ticket(d.o, t < total ? t : 0);
      if (t < total && k.pass == 0) B1::steps(steps + (n & 1) * PR::kSteps, k.tile * PR::kG1, LOGN, lane);
      __syncthreads();  // the tile before is stored, this one may start
      if (lane == 0 && finished) red_release_gpu(finished);
      if (t >= total) break;
      finished = join_done(d, k.pass, (int)(k.b % d.o.ring));
    }
    unsigned last = 0;
    if (lane == 0) {
      __threadfence();
      last = atomicAdd(d.ctr + 1, 1u) == gridDim.x - 1;
    }
    if (__shfl_sync(~0u, last, 0))
      for (int i = lane; i < 2 + 2 * d.o.ring; i += 32) d.ctr[i] = 0;
    return;
  }

  for (int n = 0;; ++n) {
    __syncthreads();  // every thread has read the last tile's shared memory
    const unsigned t = s_ticket[n & 1];
    if (t >= total) break;
    const JoinTicket k = join_ticket(d.o, t);
    cf* w = work + (int64_t)(k.b % d.o.ring) * PR::kN;
    const cf* st = steps + (n & 1) * PR::kSteps;
    cf v[kJoinR];
    if (k.pass == 0) {
      const int col0 = k.tile * PR::kG1;
      B1::template first<INV, false>(v, in + k.b * PR::kN + col0, PR::kN2, tid);
      B1::dft0(v);
      B1::template put<0>(v, sm, tid);
      join_sync<T>();
      if constexpr (PR::P1::kNst == 3) {
        B1::template get<1>(v, sm, tid);
        B1::template turn<1, false>(v, d.tw1, 0, 0, tid);
        join_sync<T>();
        B1::template put<1>(v, sm, tid);
        join_sync<T>();
      }
      B1::template get<PR::P1::kLast>(v, sm, tid);
      B1::template turn<PR::P1::kLast, true>(v, d.tw1, col0, LOGN, tid);
      B1::template store_block<PR::kG2>(v, w + col0 * PR::kG2, st, PR::kN2, tid);
    } else {
      B2::template first<false, true>(v, w + k.tile * PR::kTile, PR::kG2, tid);
      B2::dft0(v);
      B2::template put<0>(v, sm, tid);
      join_sync<T>();
      if constexpr (PR::P2::kNst == 3) {
        B2::template get<1>(v, sm, tid);
        B2::template turn<1, false>(v, d.tw2, 0, 0, tid);
        join_sync<T>();
        B2::template put<1>(v, sm, tid);
        join_sync<T>();
      }
      B2::template get<PR::P2::kLast>(v, sm, tid);
      B2::template turn<PR::P2::kLast, false>(v, d.tw2, 0, 0, tid);
      B2::template store_cols<INV>(v, out + k.b * PR::kN + k.tile * PR::kG2, PR::kN1, tid);
    }
    __syncwarp();
    if ((tid & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&stored)) : "memory");
  }
}

template <int LOGN>
inline void joined_fn(bool inv, JoinedLaunch& j) {
  using PR = JoinPair<LOGN>;
  j.fn = inv ? (const void*)joined_pass<LOGN, true> : (const void*)joined_pass<LOGN, false>;
  j.smem = (PR::kTileSlots + 2 * PR::kSteps) * sizeof(cf);
  j.block = PR::kThreads + 32;
  j.d.o.tpt_log = LOGN - PR::kTileLog;
  j.n1 = PR::kN1;
  j.n2 = PR::kN2;
  j.g1 = PR::kG1;
  j.box_rows = PR::kN1 < 256 ? PR::kN1 : 256;

}

}  // namespace gbfft
