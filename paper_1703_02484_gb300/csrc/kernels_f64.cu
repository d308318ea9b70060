// FP64 all-pairs sweep (precision = 1): the long-range force of Sec. 2.2,
//   F_i = sum_{j != i} A[s_i][s_j] (r_i - r_j) / |r_i - r_j|^3,
// every unordered pair once, both disks updated, as the FP32 symmetric sweep
// does it.
//
// What bounds it is the FP64 pipe: two lanes per SM, so that one warp
// instruction occupies it for tens of cycles and integer and FP32 work beside
// it is nearly free.  The split follows from that:
//  - Per unordered pair 14 FP64 instructions: 2 subtractions, 2 for r^2, 6 for
//    |r|^-3 and 4 into the two force sums (about 18 per ordered pair in the
//    one-sided sweep with the library's reciprocal square root).
//  - |r|^-3 starts from the FP32 reciprocal square root of r^2's leading bits
//    (moved between the formats by integer operations, the exponent apart, so
//    the whole FP64 range is covered) and takes one third-order step of
//    (1 - e)^(-3/2), e = 1 - r^2 y^2: the series' next term is below 2^-63,
//    so what is left is the rounding of two products (measured against 64-bit
//    sums in the tests' bound of 1e-12 of the RMS force).
//  - A block is 128 disks i, one per thread; groups of 32 disks j go round each
//    warp's lanes by shuffles with their own sums, four steps unrolled so that
//    one warp per scheduler keeps the pipe busy.  The four warps' j sums are
//    added in shared memory in a fixed order, and the partial sums are reduced
//    by a second kernel in the order of the host's lists: deterministic.
// Measured on one GB300 at N = 1024 (one species, walls): the sweep took 36 us
// one-sided, and with the move's launch in blocks of one warp (32 us before) the
// whole step fell from 113 to 88 us.  With the move in the reduction and its
// draws in warps of their own the step fell from 67.5 to 61.9 us.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bd_internal.h"
#include "em.cuh"
#include "f32x2.cuh"

using namespace bdf;

template <bool PER>
__global__ void __launch_bounds__(BD_F64_SB) k_force_long_f64s(BdDev d, BdConst c) {
  if (ctl_failed(d.ctl)) return;
  constexpr int NW = BD_F64_SB / 32;
  __shared__ double2 shj[NW][BD_SG];
  const int4 item = d.sitems[blockIdx.x];
  const int P = item.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gsym = (P + 1) * (BD_F64_SB / BD_SG);   // first group met from both sides
  const int2 binfo = d.sblock[P / (BD_SB / BD_F64_SB)];
  const BdRep &R = d.rep[binfo.x];
  const int a = binfo.y;
  const double L = PER ? R.L : 0.0, hL = PER && R.periodic ? 0.5 * R.L : INFINITY;
  const int i = P * BD_F64_SB + tid;
  const double2 pi = d.pos[i];
  const bool live = d.ext_id[i] >= 0;
  double fx = 0.0, fy = 0.0;
  int njp = item.w;                                     // j-partial slot
  for (int g = item.y; g < item.z; ++g) {
    const int own = g - P * NW;                         // the warp whose disks i are this group's j
    const bool both = g >= gsym;
    const int j0 = g * BD_SG + lane;
    double2 pj = d.pos[j0];
    int jl = d.ext_id[j0] >= 0 ? 1 : 0;
    const int b = d.tile_species[g * BD_SG / BD_TJ];
    double ax = 0.0, ay = 0.0, hx = 0.0, hy = 0.0;
    const int src = (lane + 1) & 31;
    auto pair = [&](bool skip) {
      double rx = pj.x - pi.x, ry = pj.y - pi.y;
      if (PER) {
        // minimum image (Sec. 2.1)
        if (abs_above(rx, hL)) rx -= copysign(L, rx);
        if (abs_above(ry, hL)) ry -= copysign(L, ry);
      }
      const double r2 = __fma_rn(ry, ry, __dmul_rn(rx, rx));
      double cf = inv_r3(r2);
      if (!(live && jl) || skip) cf = 0.0;   // inert slots, the disk itself
      ax = __fma_rn(cf, rx, ax);
      ay = __fma_rn(cf, ry, ay);
      if (both) {
        hx = __fma_rn(cf, rx, hx);
        hy = __fma_rn(cf, ry, hy);
      }
      // on to the next lane
      pj.x = __shfl_sync(0xffffffffu, pj.x, src);
      pj.y = __shfl_sync(0xffffffffu, pj.y, src);
      jl = __shfl_sync(0xffffffffu, jl, src);
      if (both) {
        hx = __shfl_sync(0xffffffffu, hx, src);
        hy = __shfl_sync(0xffffffffu, hy, src);
      }
    };
    if (both) {
#pragma unroll 4
      for (int rot = 0; rot < 32; ++rot) pair(false);
    } else {
      // the block's own disks: the i side of every ordered pair
#pragma unroll 4
      for (int rot = 0; rot < 32; ++rot) pair(own == warp && rot == 0);
    }
    // i: F_i += A[s_i][s_j] sum_j (r_i - r_j) / r^3; j the other way round
    const double ali = -R.alpha_d[BD_MAX_SPECIES * a + b];
    fx = __fma_rn(ali, ax, fx);
    fy = __fma_rn(ali, ay, fy);
    if (both) {
      shj[warp][lane] = make_double2(hx, hy);
      __syncthreads();
      if (tid < BD_SG) {
        const double alj = R.alpha_d[BD_MAX_SPECIES * b + a];
        double sx = 0.0, sy = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          sx += shj[w][tid].x;
          sy += shj[w][tid].y;
        }
        d.jpart64[(size_t)njp * BD_SG + tid] = make_double2(alj * sx, alj * sy);
      }
      __syncthreads();
      ++njp;
    }
  }
  d.ipart64[(size_t)blockIdx.x * BD_F64_SB + tid] = make_double2(fx, fy);
}

// F_i = its block's i partials + its group's j partials, in the host's order,
// into partial-force slot 0.  One warp serves the 32 disks of a group in
// eight shares (every eighth partial), so that the loads of the few disks of a
// small system are spread over eight warps; the shares are added in order.
// MOVE: the disks' move (k_integrate's) in the same kernel.  A move is some 200
// dependent FP64 instructions of 71 cycles each; three warps of their own take
// the logarithm and circle functions of two normals, those of the third, and the
// direction's beside the shares that sum, so that the first share's warp has
// only the sums left to make.
template <bool MOVE>
__global__ void __launch_bounds__(MOVE ? 352 : 256) k_force_f64_reduce(BdDev d, BdConst c, long long step, int log_step,
                                                                      int node) {
  if (ctl_failed(d.ctl)) return;
  __shared__ double2 sh[8][32];
  __shared__ bdem::Draw<double> draws[MOVE ? 32 : 1];
  const int g = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = g * BD_SG + lane, P = i / BD_F64_SB;
  int e = -1;
  double2 p = make_double2(0.0, 0.0);
  float th = 0.f;
  if (MOVE && (w == 0 || w >= 8)) {
    e = d.ext_id[i];
    p = d.pos[i];
    th = d.theta[i];
    const long long step_dev = *(volatile const long long *)&d.ctl->step_dev;
    if (step < 0) step = step_dev;
  }
  if (MOVE && w >= 8) {
    if (e >= 0) {
      bdem::Draw<double> &o = draws[lane];
      if (w == 10) {
        sincos((double)th, &o.st, &o.ct);
      } else {
        const bdrng::U4 u = bdem::words_of(d.rep[d.rep_of[i]], (uint32_t)e, step, (uint32_t)node);
        const double2 z = w == 8 ? bdem::normal_pair(u.x, u.y) : bdem::normal_pair(u.z, u.w);
        if (w == 8) {
          o.z0 = z.x;
          o.z1 = z.y;
        } else {
          o.z2 = z.x;
        }
      }
    }
  }
  double fx = 0.0, fy = 0.0;
  if (w < 8) {
    for (int k = d.red_iptr[P] + w; k < d.red_iptr[P + 1]; k += 8) {
      const double2 v = d.ipart64[(size_t)d.red_iidx[k] * BD_F64_SB + (i - P * BD_F64_SB)];
      fx += v.x;
      fy += v.y;
    }
    for (int k = d.red_jptr[g] + w; k < d.red_jptr[g + 1]; k += 8) {
      const double2 v = d.jpart64[(size_t)d.red_jidx[k] * BD_SG + lane];
      fx += v.x;
      fy += v.y;
    }
    sh[w][lane] = make_double2(fx, fy);
  }
  __syncthreads();
  if (w) return;
  const int r = d.rep_of[i];
  if (MOVE && i == 0) d.ctl->in_move = 1;
  if (r < 0) return;
  const BdRep &R = d.rep[r];
  const bool law = R.law == BD_LAW_LONG;
  if (!MOVE && !law) return;
  fx = fy = 0.0;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    fx += sh[s][lane].x;
    fy += sh[s][lane].y;
  }
  if (law) d.fpart[i] = make_double2(fx, fy);
  else fx = fy = 0.0;
  if (MOVE) bdem::move_disk<double>(d, c, R, i, e, step, log_step, node, p, th, make_double2(fx, fy), &draws[lane]);
}

static void launch_sweep(const BdDev &d, const BdConst &c, cudaStream_t s) {
  if (c.any_periodic) k_force_long_f64s<true><<<c.n_sitems, BD_F64_SB, 0, s>>>(d, c);
  else k_force_long_f64s<false><<<c.n_sitems, BD_F64_SB, 0, s>>>(d, c);
}

cudaError_t bd_launch_force_f64s(const BdDev &d, const BdConst &c, cudaStream_t s) {
  if (c.n_sitems == 0) return cudaSuccess;
  launch_sweep(d, c, s);
  k_force_f64_reduce<false><<<c.np / BD_SG, 256, 0, s>>>(d, c, 0, 0, 0);
  return cudaGetLastError();
}

cudaError_t bd_launch_force_f64s_move(const BdDev &d, const BdConst &c, int64_t step, int log_step, cudaStream_t s,
                                      int node) {
  launch_sweep(d, c, s);
  k_force_f64_reduce<true><<<c.np / BD_SG, 352, 0, s>>>(d, c, (long long)step, log_step, node);
  return cudaGetLastError();
}
