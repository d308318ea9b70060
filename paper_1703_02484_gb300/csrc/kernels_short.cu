// Short-range force over Verlet lists (Sec. 2.1, Sec. 5).
//
// Pair law: a WCA core plus an attractive Yukawa tail, truncated (not
// shifted) at r_cut as in Eq. (displacement) / Fig. "cutoff":
//   U = 4 eps[(s/r)^12 - (s/r)^6] + eps   (r < 2^(1/6) s),  s = 2a
//     - eps (s/r) exp(-kappa (r - s)),
//   F_i = sum_j -U'(r_ij) (r_i - r_j)/r_ij   for r_ij < r_cut.
// The tail is evaluated in FP32; the WCA core, whose r^-13 force near contact
// turns FP32 rounding into errors above 1e-5 of the net force, in float-float
// FP32 arithmetic (FP64 issues at ~1/64 of the FP32 rate on this part).
//
// Lists: every disk keeps the disks within r_cut + skin of it, decided in
// FP64 as (x_i - x_j)^2 + (y_i - y_j)^2 < (r_cut + skin)^2 with two products
// and one sum, each rounded once (the same expression the oracle evaluates).
// Lists are rebuilt when some disk has moved more than skin/2 since the last
// build (then no pair can have come within r_cut unseen); the test and the
// whole rebuild run on the device behind a flag, so a step never waits for the
// host.  Rebuild: cell grid of side >= r_cut + skin (count, two-level scan,
// scatter), then one thread per disk scans its 3x3 cells, sorts its list by
// disk index and writes it column-major (entry k of disk i at k*np + i) so the
// force kernel's loads are coalesced.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bd_internal.h"
#include "em.cuh"
#include "gridsync.cuh"


#define BD_VF_THREADS 128   // threads per block of the force over the lists

namespace {

// float-float arithmetic (value = hi + lo, |lo| <= ulp(hi)/2), about 48
// significant bits from FP32 instructions only
struct ff {
  float hi, lo;
};
__device__ __forceinline__ ff ff_make(float a, float b) {  // exact a + b, |a| >= |b| not required
  float s = __fadd_rn(a, b);
  float bp = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
  return {s, e};
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  float s = __fadd_rn(p, e);
  return {s, __fsub_rn(e, __fsub_rn(s, p))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = ff_make(a.hi, b.hi);
  float lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  float h = __fadd_rn(s.hi, lo);
  return {h, __fsub_rn(lo, __fsub_rn(h, s.hi))};
}
__device__ __forceinline__ ff ff_scale(ff a, float b) { return ff_mul(a, {b, 0.f}); }
// a / b given rb, 1 / b.hi to within a few ulps (the fast FP32 reciprocal):
// the FP32 quotient a.hi rb (relative error ~2^-22) refined by one
// float-float residual step, which leaves ~2^-44 relative error
__device__ __forceinline__ ff ff_div_r(ff a, ff b, float rb) {
  float q1 = __fmul_rn(a.hi, rb);
  ff r = ff_add(a, ff_scale(b, -q1));
  float q2 = __fmul_rn(r.hi, rb);
  float s = __fadd_rn(q1, q2);
  return {s, __fsub_rn(q2, __fsub_rn(s, q1))};
}

__device__ __forceinline__ int failed(const BdCtl *ctl) { return *(volatile const int *)&ctl->status; }
__device__ __forceinline__ int need(const BdCtl *ctl) { return *(volatile const int *)&ctl->vl_need; }

__device__ __forceinline__ int cell_of(double2 p, const BdRep &R) {
  int cx = (int)(p.x / R.cell_size);
  int cy = (int)(p.y / R.cell_size);
  cx = cx < 0 ? 0 : (cx >= R.ncell ? R.ncell - 1 : cx);
  cy = cy < 0 ? 0 : (cy >= R.ncell ? R.ncell - 1 : cy);
  return R.cell_base + cy * R.ncell + cx;
}

// periodic box (Sec. 2.1): minimum image of an exact FP64 coordinate difference
__device__ __forceinline__ double dmin_image(double d, const BdRep &R) {
  if (!R.periodic) return d;
  if (d > 0.5 * R.L) return __dsub_rn(d, R.L);
  if (d < -0.5 * R.L) return __dadd_rn(d, R.L);
  return d;
}

// replica of slot i if it is a disk of a short-range replica, else null
__device__ __forceinline__ const BdRep *short_rep(const BdDev &d, int i) {
  const int r = d.rep_of[i];
  if (r < 0) return nullptr;
  const BdRep *R = &d.rep[r];
  return R->law == BD_LAW_SHORT ? R : nullptr;
}

}  // namespace

// Displacement trigger: some disk moved more than skin/2 since the build.
// Bound by memory (36 bytes a disk); every load of a thread is issued before
// the status is looked at.
__global__ void __launch_bounds__(BD_VL_THREADS) k_vl_check(BdDev d, BdConst c) {
  const int i = blockIdx.x * BD_VL_THREADS + threadIdx.x;
  const int bad = failed(d.ctl);
  bool hit = false;
  if (i < c.np) {
    const double2 p = d.pos[i], r = d.vl_ref[i];
    const BdRep *R = short_rep(d, i);
    if (R && !bad) {
      // displacement since the build in grid units (exact), screened in FP32
      // in steps of 2^vl_shift of them (2^-27 of skin/2 or finer); only a
      // displacement within 1e-5 of skin/2 is decided in FP64
      const bdpred::Grid g{c.q, c.inv_q, c.qshift};
      if (r.x > 1e29) {
        hit = true;   // never built (reference parked far away)
      } else {
        long long ex = bdpred::to_int(p.x, g) - bdpred::to_int(r.x, g);
        long long ey = bdpred::to_int(p.y, g) - bdpred::to_int(r.y, g);
        if (R->periodic) {
          // displacement across an edge: its minimum image
          const long long h = R->LQ / 2;
          ex = ex > h ? ex - R->LQ : (ex < -h ? ex + R->LQ : ex);
          ey = ey > h ? ey - R->LQ : (ey < -h ? ey + R->LQ : ey);
        }
        const long long sx = ex >> R->vl_shift, sy = ey >> R->vl_shift;
        const float fx = (float)(int)sx, fy = (float)(int)sy;
        const float d2 = __fadd_rn(__fmul_rn(fx, fx), __fmul_rn(fy, fy));
        const float thr = R->vl_thr;
        if (sx != (int)sx || sy != (int)sy || d2 > thr * 1.00001f) {
          hit = true;
        } else if (d2 >= thr * 0.99999f) {
          double dx = dmin_image(p.x - r.x, *R), dy = dmin_image(p.y - r.y, *R);
          hit = dx * dx + dy * dy > 0.25 * R->skin * R->skin;
        }
      }
    }
  }
  if (__any_sync(0xffffffffu, hit) && (threadIdx.x & 31) == 0) atomicExch(&d.ctl->vl_need, 1);
}

// neighbour list of disk i from the cell grid (sorted), and its reference position
__device__ __forceinline__ void vl_build_one(const BdDev &d, const BdConst &c, int i) {
  const BdRep *Rp = short_rep(d, i);
  if (!Rp || d.ext_id[i] < 0) {
    d.vl_cnt[i] = 0;
    return;
  }
  const BdRep &R = *Rp;
  const double2 p = d.pos[i];
  d.vl_ref[i] = p;
  const float4 wi = d.work[i];
  const float rl2f = (float)R.rl2;
  const int k = d.cell_of[i] - R.cell_base;
  const int cx = k % R.ncell, cy = k / R.ncell;
  int buf[BD_VL_MAX];
  int m = 0;
  bool over = false;
  for (int gy0 = cy - 1; gy0 <= cy + 1; ++gy0) {
    // periodic box: the cells wrap around (at least three per side)
    const int gy = R.periodic ? (gy0 + R.ncell) % R.ncell : gy0;
    if (gy < 0 || gy >= R.ncell) continue;
    for (int gx0 = cx - 1; gx0 <= cx + 1; ++gx0) {
      const int gx = R.periodic ? (gx0 + R.ncell) % R.ncell : gx0;
      if (gx < 0 || gx >= R.ncell) continue;
      const int cc = R.cell_base + gy * R.ncell + gx;
      const int b = d.cell_start[cc], e = b + d.cell_count[cc];
      for (int s = b; s < e; ++s) {
        const int j = d.cell_idx[s];
        if (j == i) continue;
        // FP32 screen from the (hi, lo) pairs: the hi difference is exact
        // (Sterbenz) or off by at most half an ulp of a coordinate below 12
        // (4.8e-7), so the computed r^2 is within 1e-6 of the exact one
        // relative to the reach; only pairs within 1e-5 of the reach (and
        // pairs across a periodic edge) take the FP64 decision
        const float4 wj = d.work[j];
        const float hx = __fsub_rn(wi.x, wj.x), hy = __fsub_rn(wi.y, wj.y);
        bool in;
        bool exact = R.periodic && (fabsf(hx) > R.hLf || fabsf(hy) > R.hLf);
        if (!exact) {
          const float fx = __fadd_rn(hx, __fsub_rn(wi.z, wj.z)), fy = __fadd_rn(hy, __fsub_rn(wi.w, wj.w));
          const float f2 = __fadd_rn(__fmul_rn(fx, fx), __fmul_rn(fy, fy));
          if (f2 < rl2f * 0.99999f) in = true;
          else if (f2 > rl2f * 1.00001f) in = false;
          else exact = true;
        }
        if (exact) {
          const double2 q = d.pos[j];
          const double dx = dmin_image(__dsub_rn(p.x, q.x), R), dy = dmin_image(__dsub_rn(p.y, q.y), R);
          in = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)) < R.rl2;
        }
        if (in) {
          if (m < BD_VL_MAX) {
            // insertion in sorted position
            int t = m++;
            while (t > 0 && buf[t - 1] > j) {
              buf[t] = buf[t - 1];
              --t;
            }
            buf[t] = j;
          } else {
            over = true;
          }
        }
      }
    }
  }
  for (int t = 0; t < m; ++t) d.vl_idx[(size_t)t * c.np + i] = buf[t];
  d.vl_cnt[i] = m;
  if (over) atomicCAS(&d.ctl->status, 0, BD_ERR_UNSUPPORTED);
}

// exclusive prefix sum over the block of one value per thread; *total = the sum
__device__ __forceinline__ int block_scan(int v, int *total) {
  __shared__ int ws[BD_VL_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int s = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += t;
  }
  if (lane == 31) ws[warp] = s;
  __syncthreads();
  int base = 0, all = 0;
#pragma unroll
  for (int w = 0; w < BD_VL_THREADS / 32; ++w) {
    if (w < warp) base += ws[w];
    all += ws[w];
  }
  __syncthreads();   // ws is reused by the next call
  *total = all;
  return base + s - v;
}

// Rebuild of the cell grid and the lists when the trigger fired, one
// cooperative launch (a step that needs none leaves at once).  As seven
// launches (clear, count, three of the scan, scatter, build) the seven of every
// step without a rebuild took about 20 us of the device's time under ncu; now a
// step at 2^20 disks takes 540 us instead of 549, at 20000 polydisperse disks 109
// instead of 113.  Phases, each ended by
// a bounded grid barrier: clear the cell counts; count; sum each block's share
// of the cells; scan it from the sums before it, setting the scatter cursors;
// scatter; build, which needs no barrier after it (its reads of the grid go
// through L1, which the barrier's acquire has emptied; past L1 ten steps at
// 2^20 disks with one rebuild took 6.06 instead of 5.40 ms).
__global__ void __launch_bounds__(BD_VL_THREADS, 4) k_vl_rebuild(BdDev d, BdConst c) {
  if (failed(d.ctl) || !need(d.ctl)) return;   // the same for every block: both words are set by earlier kernels
  bdgs::Bar b;
  b.gen = 0;
  b.ph = 0;
  const int tid = blockIdx.x * BD_VL_THREADS + threadIdx.x, nth = gridDim.x * BD_VL_THREADS;
  const int nc = c.ncell_total;
  for (int k = tid; k < nc; k += nth) d.cell_count[k] = 0;
  if (!bdgs::grid_sync<false>(d.ctl, b)) { bdgs::block_exit(d.ctl); return; }
  for (int i = tid; i < c.np; i += nth) {
    const BdRep *R = short_rep(d, i);
    if (!R || d.ext_id[i] < 0) {
      d.cell_of[i] = -1;
      continue;
    }
    const int k = cell_of(d.pos[i], *R);
    d.cell_of[i] = k;
    atomicAdd(&d.cell_count[k], 1);
  }
  if (!bdgs::grid_sync<false>(d.ctl, b)) { bdgs::block_exit(d.ctl); return; }
  const int per = (nc + (int)gridDim.x - 1) / (int)gridDim.x;
  const int k0 = min(nc, (int)blockIdx.x * per), k1 = min(nc, k0 + per);
  int total = 0;
  {
    int v = 0;
    for (int k = k0 + (int)threadIdx.x; k < k1; k += BD_VL_THREADS) v += d.cell_count[k];
    block_scan(v, &total);
    if (threadIdx.x == 0) d.scan_sums[blockIdx.x] = total;
  }
  if (!bdgs::grid_sync<false>(d.ctl, b)) { bdgs::block_exit(d.ctl); return; }
  {
    int v = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += BD_VL_THREADS) v += d.scan_sums[k];
    int base = 0;
    block_scan(v, &base);
    for (int kk = k0; kk < k1; kk += BD_VL_THREADS) {
      const int k = kk + (int)threadIdx.x;
      const int n = k < k1 ? d.cell_count[k] : 0;
      const int e = base + block_scan(n, &total);
      if (k < k1) {
        d.cell_start[k] = e;
        d.cell_cursor[k] = e;
      }
      base += total;
    }
  }
  if (!bdgs::grid_sync<false>(d.ctl, b)) { bdgs::block_exit(d.ctl); return; }
  for (int i = tid; i < c.np; i += nth) {
    const int k = d.cell_of[i];   // this thread's own store
    if (k >= 0) d.cell_idx[atomicAdd(&d.cell_cursor[k], 1)] = i;
  }
  if (!bdgs::grid_sync<false>(d.ctl, b)) { bdgs::block_exit(d.ctl); return; }
  for (int i = tid; i < c.np; i += nth) vl_build_one(d, c, i);
  bdgs::block_exit(d.ctl);
}

// r_i - r_j as FP32 (hi, lo) pairs: from the disks' own pairs, exact for near
// pairs; a pair across a periodic box edge is formed exactly in grid units from
// the FP64 masters instead (its hi parts differ by ~L)
__device__ __forceinline__ void pair_diff(const BdDev &d, const BdConst &c, const BdRep &R, int i, int j,
                                          const float4 &wi, const float4 &wj, float &hx, float &lx, float &hy,
                                          float &ly) {
  hx = __fsub_rn(wi.x, wj.x);
  hy = __fsub_rn(wi.y, wj.y);
  lx = __fsub_rn(wi.z, wj.z);
  ly = __fsub_rn(wi.w, wj.w);
  if (R.periodic && (fabsf(hx) > R.hLf || fabsf(hy) > R.hLf)) {
    const bdpred::Grid g{c.q, c.inv_q, c.qshift};
    const double2 pi = d.pos[i], pj = d.pos[j];
    long long X = bdpred::to_int(pi.x, g) - bdpred::to_int(pj.x, g);
    long long Y = bdpred::to_int(pi.y, g) - bdpred::to_int(pj.y, g);
    const long long h = R.LQ / 2;
    X = X > h ? X - R.LQ : (X < -h ? X + R.LQ : X);
    Y = Y > h ? Y - R.LQ : (Y < -h ? Y + R.LQ : Y);
    const float2 sx = bdem::grid_split(X, c.qshift), sy = bdem::grid_split(Y, c.qshift);
    hx = sx.x; lx = sx.y;
    hy = sy.x; ly = sy.y;
  }
}

// short-range force over the lists; clears the rebuild flag.
// Two passes over a disk's list.  The first adds the Yukawa tail of every entry
// within the cut-off and marks those inside the WCA core in a bit mask (a list
// holds at most 64); the second walks the mask and adds the float-float core,
// some 150 instructions for the two or three contacts of a disk.  In one pass a
// warp ran the core for nearly every list position, since at each one some lane
// of the 32 had a contact there.  The sums take the same terms in the same
// order.  32 warps per SM (64 registers, without spills now) in blocks of 128, whose
// last ones end sooner than those of 256; with that and a disk's own loads issued
// together (slot, replica, list length and the first four entries waited for one
// another) a step of 2^20 disks fell from 335.6 to 327 us, of 200003 from 112.1 to
// 111.0.  The gathers want the warps, and the polydisperse branch must not cost the
// equal-disk case its occupancy.  The law's constants come rounded from the
// host and the result is widened by its bits: formed here, their dozen FP64
// products and conversions a disk kept the FP64 pipe (two lanes per SM) busy for
// 59 % of the kernel's time.
__global__ void __launch_bounds__(BD_VF_THREADS, 1024 / BD_VF_THREADS) k_force_verlet(BdDev d, BdConst c) {
  const int i = blockIdx.x * BD_VF_THREADS + threadIdx.x;
  if (i >= c.np) return;
  // every load of a disk's own data is issued before any is looked at
  const bool bad = failed(d.ctl);
  const int e = d.ext_id[i], r = c.R == 1 ? 0 : d.rep_of[i], m = d.vl_cnt[i];
  const float4 wi = d.work[i];
  int jn[4];   // (the first rows of the lists, whatever their length)
#pragma unroll
  for (int u = 0; u < 4; ++u) jn[u] = d.vl_idx[(size_t)u * c.np + i];
  if (bad) return;
  if (i == 0) {
    if (need(d.ctl)) {
      d.ctl->vl_need = 0;
      d.ctl->st_verlet_rebuilds += 1;
    }
  }
  if (e < 0 || d.rep[r].law != BD_LAW_SHORT) return;
  const BdRep &R = d.rep[r];
  const float rc2 = R.rc2f;
  const float eps = R.epsf, kap = R.kapf;
  // the law's length scale s: 2a, or a_i + a_j for polydisperse disks (then
  // formed per pair from the radii's FP32 (hi, lo) pairs, exact to ~2^-48)
  const bool poly = d.radf != nullptr;
  const float2 ai = poly ? d.radf[i] : make_float2(0.f, 0.f);
  const float sg0 = c.sigf;
  const float rwca20 = c.rwca2f;   // (2^(1/6) s)^2
  float fx = 0.f, fy = 0.f;      // Yukawa tail, FP32
  unsigned long long core = 0ull;
  // four list entries at a time: their position gathers are issued before
  // any of them is used, and the next four indices are loaded while these
  // are evaluated
#pragma unroll
  for (int u = 0; u < 4; ++u) jn[u] = u < m ? jn[u] : i;
  for (int t0 = 0; t0 < m; t0 += 4) {
    int jj[4];
    float4 wv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) jj[u] = jn[u];
#pragma unroll
    for (int u = 0; u < 4; ++u) wv[u] = d.work[jj[u]];
#pragma unroll
    for (int u = 0; u < 4; ++u) jn[u] = t0 + 4 + u < m ? d.vl_idx[(size_t)(t0 + 4 + u) * c.np + i] : i;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (t0 + u >= m) break;
      const int j = jj[u];
      float hx, lx, hy, ly;
      pair_diff(d, c, R, i, j, wi, wv[u], hx, lx, hy, ly);
      const float dx = __fadd_rn(hx, lx);
      const float dy = __fadd_rn(hy, ly);
      const float r2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
      float sg = sg0, rwca2 = rwca20;
      if (poly) {
        const float2 aj = d.radf[j];
        const ff sp = ff_add(ff_make(ai.x, ai.y), ff_make(aj.x, aj.y));
        sg = sp.hi;
        rwca2 = 1.2599210498948732f * ff_mul(sp, sp).hi;
      }
      if (fabsf(r2 - rc2) < 1e-5f * rc2) {
        // at the cut-off the force jumps: decide as the FP64 reference does
        const double2 pi = d.pos[i], pj = d.pos[j];
        const double ex = dmin_image(__dsub_rn(pi.x, pj.x), R), ey = dmin_image(__dsub_rn(pi.y, pj.y), R);
        if (!(sqrt(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey))) < R.r_cut)) continue;
      } else if (r2 >= rc2) {
        continue;
      }
      // Yukawa tail: -U'(r) / r, smooth, in FP32 (approximate reciprocal
      // square root and exponential: relative error ~1e-7)
      const float ir = rsqrtf(r2);
      const float r = r2 * ir;
      const float my = -eps * sg * __expf(-kap * (r - sg)) * (ir * ir + kap * ir) * ir;
      fx = fmaf(my, dx, fx);
      fy = fmaf(my, dy, fy);
      if (r2 < rwca2) core |= 1ull << (t0 + u);
    }
  }
  // WCA core near contact: -U'(r) ~ r^-13 turns FP32 rounding into errors above
  // 1e-5 of the net force, so the core is evaluated in float-float arithmetic
  // (FP32 instructions, ~48-bit significands) from the exact coordinate differences
  ff gx = {0.f, 0.f}, gy = {0.f, 0.f};
  float s2h = c.s2h, s2l = c.s2l;   // s^2 as a float-float pair
  while (core) {
    const int t = __ffsll((long long)core) - 1;
    core &= core - 1ull;
    const int j = d.vl_idx[(size_t)t * c.np + i];
    float hx, lx, hy, ly;
    pair_diff(d, c, R, i, j, wi, d.work[j], hx, lx, hy, ly);
    if (poly) {
      const float2 aj = d.radf[j];
      const ff sp = ff_add(ff_make(ai.x, ai.y), ff_make(aj.x, aj.y));
      const ff sq = ff_mul(sp, sp);
      s2h = sq.hi;
      s2l = sq.lo;
    }
    ff ex = ff_make(hx, lx);
    ff ey = ff_make(hy, ly);
    ff q2 = ff_add(ff_mul(ex, ex), ff_mul(ey, ey));
    // 1 / r^2 once (one fast reciprocal, one residual step), then products
    const ff iq2 = ff_div_r({1.0f, 0.f}, q2, __fdividef(1.0f, q2.hi));
    ff s2 = ff_mul({s2h, s2l}, iq2);   // (s / r)^2 as a float-float pair
    ff s6 = ff_mul(ff_mul(s2, s2), s2);
    ff s12 = ff_mul(s6, s6);
    ff t2 = ff_add({2.0f * s12.hi, 2.0f * s12.lo}, {-s6.hi, -s6.lo});   // exact doubling
    ff cw = ff_mul(ff_scale(t2, 24.0f * eps), iq2);
    gx = ff_add(gx, ff_mul(cw, ex));
    gy = ff_add(gy, ff_mul(cw, ey));
  }
  // the float-float total, rounded once to FP32 (the move reads the force in
  // FP32), stored as a double without FP64 arithmetic
  const ff tx = ff_add(gx, {fx, 0.f}), ty = ff_add(gy, {fy, 0.f});
  d.fpart[i] = make_double2(bdem::f64_of(tx.hi), bdem::f64_of(ty.hi));
}

int bd_vl_grid_for(int np, int *grid) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_vl_rebuild, BD_VL_THREADS, 0) != cudaSuccess) return -1;
  if (per < 1) return -1;
  const int want = (np + BD_VL_THREADS - 1) / BD_VL_THREADS;   // at most one disk per thread
  int g = sms * per;
  if (g > BD_VL_MAXGRID) g = BD_VL_MAXGRID;
  *grid = want < 1 ? 1 : (want < g ? want : g);
  return 0;
}

cudaError_t bd_launch_force_short(const BdDev &d, const BdConst &c, cudaStream_t s) {
  if (!c.any_short) return cudaSuccess;
  const int gn = (c.np + BD_VL_THREADS - 1) / BD_VL_THREADS;
  k_vl_check<<<gn, BD_VL_THREADS, 0, s>>>(d, c);
  BdDev dd = d;
  BdConst cc = c;
  void *args[] = {&dd, &cc};
  cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_vl_rebuild, dim3(c.vl_grid), dim3(BD_VL_THREADS), args, 0, s);
  if (e != cudaSuccess) return e;
  k_force_verlet<<<(c.np + BD_VF_THREADS - 1) / BD_VF_THREADS, BD_VF_THREADS, 0, s>>>(d, c);
  return cudaGetLastError();
}

int bd_short_launches() { return 3; }
