// Grid-wide barrier and block-level helpers of the persistent kernels
// (triangulation maintenance, Verlet-list overlap correction).  The kernels
// are launched cooperatively (every block resident), and every wait of a grid
// is bounded: a barrier that waits longer than its limit (BD_BARRIER_TIMEOUT_NS,
// or the limit the host set in the control block) sets BD_ERR_DEVICE_TIMEOUT
// and every block leaves.  A small system's triangulation runs in one
// thread-block cluster and waits at the hardware's cluster barrier, which takes
// no limit: the blocks of a cluster are resident together and take every branch
// on the same words, so each of them arrives.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "bd_internal.h"

namespace bdgs {

#ifndef BD_BARRIER_TIMEOUT_NS
#define BD_BARRIER_TIMEOUT_NS 2000000000ull
#endif

struct Bar {
  unsigned gen;
  int ph;
};

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int ld_status(const int *p) {
  return *(volatile const int *)p;
}

// Words every thread needs after a barrier, read once per block by thread 0
// and handed to the block through shared memory (116k threads reading one
// global line would queue ~18k requests on one L2 slice per barrier).
enum { BC_CNT = 0, BC_CL = 8, BC_N = 11 };

// Bounded grid barrier; returns false if the grid must stop.  With bc (block
// shared, BC_N ints): bc[BC_CNT + k] = the counters of the phase that just
// ended, bc[BC_CL + l] = the lengths of the candidate lists.  HOLD: the barrier obeys the host's test hold
// (the kernels of a move do; the Verlet-list rebuild does not).
//
// A barrier is its chain of L2 round trips, kept to three: the arrival, the
// poll and the read of bc's words (one lane each).  Blocks arrive at and poll
// the same word: each adds 1, the first block what brings the sum of all to
// 2^31, so the last arrival flips the top bit and is itself the release; the
// word needs no reset between barriers (the launch's last block clears it).
// (The flipped bit is the scheme of cooperative groups' grid barrier, public in
// the CUDA toolkit's cooperative_groups/details/sync.h; the limit, the hold and
// the words read behind it are this kernel's.)
// Measured at 8 to 456 blocks: 1.5 us, against 2.5 with a separate word that the
// last block to arrive publishes and 3 with a count it also resets.
template <bool HOLD = true>
static __device__ bool grid_sync(BdCtl *ctl, Bar &b, int *bc = nullptr) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int ok = 1;
    if (lane == 0) {
      const unsigned hold = HOLD ? *(volatile const unsigned *)&ctl->bar_hold : 0u;
      unsigned add = 1u;
      if (blockIdx.x == 0) {
        add = 0x80000000u - (gridDim.x - 1u);
        if (hold != 0u && hold == b.gen + 1u) add -= 1u;   // held: one block more than the launch has, which never comes
      }
      __threadfence();
      const unsigned old = atomicAdd(&ctl->bar_count, add);
      // spin hot for a while (barriers are short), then back off; give up
      // after the time limit, or when another block has
      unsigned long long t0 = 0, limit = 0;
      for (unsigned it = 0; ((old ^ *(volatile const unsigned *)&ctl->bar_count) & 0x80000000u) == 0u; ++it) {
        if (it < 4096u) continue;
        if ((it & 63u) == 0) {
          if (t0 == 0) {
            t0 = gtimer();
            const unsigned long long lim_set = *(volatile const unsigned long long *)&ctl->bar_limit_ns;
            limit = lim_set ? lim_set : BD_BARRIER_TIMEOUT_NS;
          }
          if (gtimer() - t0 > limit || ld_status(&ctl->status) == BD_ERR_DEVICE_TIMEOUT) {
            atomicExch(&ctl->status, BD_ERR_DEVICE_TIMEOUT);
            ok = 0;
            break;
          }
        }
        __nanosleep(64);
      }
      __threadfence();
      s_ok = ok;
    }
    __syncwarp();
    if (bc && lane < BC_N)
      bc[lane] = lane < BC_CL ? ((const volatile int *)ctl->cnt[b.ph & 3])[lane]
                              : ((const volatile int *)ctl->cl_n)[lane - BC_CL];
  }
  __syncthreads();
  b.gen++;
  b.ph++;
  return s_ok != 0;
}

__device__ __forceinline__ int *cnt(BdCtl *ctl, int ph, int slot) { return &ctl->cnt[ph & 3][slot]; }


// every block calls this once on its way out; the last one resets the barrier
// words and phase counters so the next launch starts clean without a memset
static __device__ void block_exit(BdCtl *ctl) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    unsigned k = atomicAdd(&ctl->exit_count, 1u);
    if (k == gridDim.x - 1) {
      ctl->bar_count = 0;
      for (int l = 0; l < 3; ++l) ctl->cl_n[l] = 0;
      for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 8; ++b) ctl->cnt[a][b] = 0;
      __threadfence();
      ctl->exit_count = 0;
    }
  }
}

// ---- the same phases inside one thread-block cluster ----
// A small system's triangulation runs in one cluster: its barrier is the
// hardware's, and the phase counters and list lengths sit in the first block's
// shared memory (words: BW_N ints there, reached by every block of the
// cluster), so that a phase ends without a round trip through L2.
enum { BW_CNT = 0, BW_CL = 32, BW_N = 35 };

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// as grid_sync; hold: the host's test hold, read once at the launch's start.  A
// held barrier waits out the limit and gives up (every block of it), as the
// grid barrier does.
static __device__ bool cluster_sync(BdCtl *ctl, const int *words, unsigned hold, Bar &b, int *bc) {
  cluster_barrier();
  b.gen++;
  if (hold != 0u && hold == b.gen) {
    const unsigned long long lim_set = *(volatile const unsigned long long *)&ctl->bar_limit_ns;
    const unsigned long long limit = lim_set ? lim_set : BD_BARRIER_TIMEOUT_NS;
    const unsigned long long t0 = gtimer();
    while (gtimer() - t0 <= limit) __nanosleep(1000);
    if (threadIdx.x == 0) atomicExch(&ctl->status, BD_ERR_DEVICE_TIMEOUT);
    return false;
  }
  if (threadIdx.x < BC_N) {
    const int k = threadIdx.x;
    const int at = k < BC_CL ? BW_CNT + 8 * (b.ph & 3) + k : BW_CL + k - BC_CL;
    bc[k] = ((const volatile int *)words)[at];
  }
  __syncthreads();
  b.ph++;
  return true;
}

// reset the counters two phases ahead (see the rotation argument in BdCtl)
__device__ __forceinline__ void phase_begin(BdCtl *ctl, const Bar &b) {
  if (blockIdx.x == 0 && threadIdx.x < 8) ctl->cnt[(b.ph + 2) & 3][threadIdx.x] = 0;
}

// block-aggregated atomic adds of K counters at once
template <int K>
__device__ __forceinline__ void block_add(int *const (&dst)[K], const int (&v)[K]) {
  __shared__ int s_acc[K];
  if (threadIdx.x < K) s_acc[threadIdx.x] = 0;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int t = __reduce_add_sync(0xffffffffu, v[k]);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(&s_acc[k], t);
  }
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (s_acc[k]) atomicAdd(dst[k], s_acc[k]);
}
__device__ __forceinline__ void block_add(int *dst, int v) {
  int *const d[1] = {dst};
  const int w[1] = {v};
  block_add<1>(d, w);
}

}  // namespace bdgs
