// Grid-wide barrier and block-level helpers of the persistent kernels
// (triangulation maintenance, Verlet-list overlap correction).  The kernels
// are launched cooperatively (every block resident), and every wait is
// bounded: a barrier that waits longer than its limit (BD_BARRIER_TIMEOUT_NS,
// or the limit the host set in the control block) sets BD_ERR_DEVICE_TIMEOUT
// and every block leaves.
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

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

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
enum { BC_CNT = 0, BC_ACT = 8, BC_CL = 11, BC_N = 14 };

__device__ __forceinline__ void st_b128(void *p, unsigned x, unsigned y, unsigned z, unsigned w) {
  const unsigned long long lo = ((unsigned long long)y << 32) | x, hi = ((unsigned long long)w << 32) | z;
  asm volatile(
      "{ .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p), "l"(lo), "l"(hi)
      : "memory");
}
__device__ __forceinline__ uint4 ld_b128(const void *p) {
  unsigned long long lo, hi;
  asm volatile("{ .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t; }"
               : "=l"(lo), "=l"(hi)
               : "l"(p)
               : "memory");
  return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}

// Bounded grid barrier; returns false if the grid must stop.  With bc (block
// shared, BC_N ints): bc[BC_CNT + k] = the counters of the phase that just
// ended, bc[BC_ACT + l] = the lengths of the triangle lists, bc[BC_CL + l]
// those of the candidate lists.  HOLD: the barrier obeys the host's test hold
// (the kernels of a move do; the Verlet-list rebuild does not).
//
// A barrier costs its chain of L2 round trips, so the chain is kept short:
// arrivals are counted without a reset (the launch's last block resets the
// count), and the last block to arrive reads the words of bc once and publishes
// them with the generation, three to a 16-byte chunk that carries the
// generation as its tag; the other blocks poll the chunks themselves (one warp
// load of one line) and have everything when the tags match.
template <bool HOLD = true>
static __device__ bool grid_sync(BdCtl *ctl, Bar &b, int *bc = nullptr) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const unsigned target = b.gen + 1;
    constexpr int NC = (BC_N + 2) / 3;   // published chunks
    const int nc = bc ? NC : 1;
    int ok = 1, last = 0;
    if (lane == 0) {
      const unsigned hold = HOLD ? *(volatile const unsigned *)&ctl->bar_hold : 0u;
      __threadfence();
      const unsigned arrived = atomicAdd(&ctl->bar_count, 1u);
      // (held: one block more than the launch has, which never comes)
      last = arrived == target * gridDim.x - 1u && !(hold != 0u && hold == target);
      __threadfence();
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();
    if (last) {
      int w = 0;
      if (bc) {
        if (lane < 8) w = ((const volatile int *)ctl->cnt[b.ph & 3])[lane];
        else if (lane < BC_CL) w = ((const volatile int *)ctl->act_n)[lane - BC_ACT];
        else if (lane < BC_N) w = ((const volatile int *)ctl->cl_n)[lane - BC_CL];
        if (lane < BC_N) bc[lane] = w;
      }
      const int c = lane < NC ? 3 * lane : 0;
      const int w0 = __shfl_sync(0xffffffffu, w, c), w1 = __shfl_sync(0xffffffffu, w, c + 1),
                w2 = __shfl_sync(0xffffffffu, w, c + 2);
      if (lane < nc) st_b128(&ctl->bar_pub[lane], target, (unsigned)w0, (unsigned)w1, (unsigned)w2);
    } else {
      // spin hot for a while (barriers are short), then back off; give up
      // after the time limit, or when another block has
      unsigned long long t0 = 0, limit = 0;
      uint4 v = make_uint4(target, 0u, 0u, 0u);
      for (unsigned it = 0;; ++it) {
        if (lane < nc) v = ld_b128(&ctl->bar_pub[lane]);
        if (__all_sync(0xffffffffu, v.x == target)) break;
        if (it < 4096u) continue;
        if ((it & 63u) == 0) {
          if (lane == 0) {
            if (t0 == 0) {
              t0 = gtimer();
              const unsigned long long lim_set = *(volatile const unsigned long long *)&ctl->bar_limit_ns;
              limit = lim_set ? lim_set : BD_BARRIER_TIMEOUT_NS;
            }
            if (gtimer() - t0 > limit || ld_status(&ctl->status) == BD_ERR_DEVICE_TIMEOUT) {
              atomicExch(&ctl->status, BD_ERR_DEVICE_TIMEOUT);
              ok = 0;
            }
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
        }
        __nanosleep(64);
      }
      __threadfence();
      if (bc && lane < NC) {
        bc[3 * lane] = (int)v.y;
        if (3 * lane + 1 < BC_N) bc[3 * lane + 1] = (int)v.z;
        if (3 * lane + 2 < BC_N) bc[3 * lane + 2] = (int)v.w;
      }
    }
    if (lane == 0) s_ok = ok;
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
      for (int c = 0; c < 8; ++c) ctl->bar_pub[c] = make_uint4(0u, 0u, 0u, 0u);
      for (int l = 0; l < 3; ++l) ctl->act_n[l] = ctl->cl_n[l] = 0;
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
enum { BW_CNT = 0, BW_ACT = 32, BW_CL = 35, BW_N = 38 };

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
    const int at = k < BC_ACT ? BW_CNT + 8 * (b.ph & 3) + k : (k < BC_CL ? BW_ACT + k - BC_ACT : BW_CL + k - BC_CL);
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
