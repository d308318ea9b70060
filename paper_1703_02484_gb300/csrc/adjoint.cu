// Adjoint of a rollout of the time step (reverse mode), for gradients of a
// loss of the final positions with respect to the pair-force table A (Sec.
// 2.2) and the self-propulsion speed v0 (Sec. 7).  No counterpart in the
// paper.
//
// The differentiated map is the step with its random and discrete choices
// frozen: the Philox noise, the wall reflections of every move, the
// overlapping pairs of every correction pass (Algorithm 2) and which disks
// had their displacement capped at sigma/4.  One step is
//   y   = R0( x + dt (F(x; A) + v0 e(theta)) + amp xi )          (Eq. (integration))
//   z_1 = y,   z_{j+1} = Rj( z_j + cap_j( d_j(z_j) ) )           (Algorithm 2 passes)
//   d_j(z)_u = -sum (sigma - r) r_hat,  d_j(z)_w = +sum (sigma - r) r_hat over the logged
//   pairs (u, w) of pass j, r_hat = (z_w - z_u)/r;  cap(d) = d or (sigma/4) d/|d|.
// Rounding to the position grid is taken as the identity.
//
// Backward through one pass: mu = R^T lambda (a reflected component changes
// sign); mu_d = cap'^T mu (for a capped disk (s/|d|)(I - d_hat d_hat^T) mu);
// lambda <- mu + sum over pairs G (mu_d_u - mu_d_w) at u and its negative at w,
// with G = d/dv [(sigma - |v|) v/|v|] = (sigma/r)(I - n n^T) - I.
// Backward through the move: mu = R0^T lambda; lambda <- mu + dt (dF/dx)^T mu,
//   ((dF/dx)^T mu)_i = sum_j M(r_ij) (A_ij mu_i - A_ji mu_j),  M(r) = I/r^3 - 3 r r^T/r^5,
// and the parameter gradients dL/dA_ab += dt sum_{i in a} mu_i . sum_{j in b} r_ij/r_ij^3,
// dL/dv0 += dt sum_i mu_i . e(theta_i).
// The force adjoint's pair terms are FP32, summed in FP32 over at most 128 disks
// j and in FP64 beyond; everything else is FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "bd_internal.h"
#include "em.cuh"
#include "f32x2.cuh"

using namespace bdf;

namespace {

__device__ __forceinline__ double atomic_add_d(double *p, double v) { return atomicAdd(p, v); }

}  // namespace

// ---------------------------------------------------------------- replay

// Euler-Maruyama move with the logged reflections (the forces are in fpart);
// sx, sth (or null) keep the positions and directions it starts from, z (or
// null) those it ends at
__global__ void k_rp_em(BdDev d, BdConst c, long long step, int k_local, double2 *sx, float *sth, double2 *z) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= c.np) return;
  const int e = d.ext_id[i];
  if (e < 0) return;
  const BdRep &R = d.rep[d.rep_of[i]];
  const double2 F = bdem::force_sum(d, c, R, i, d.fpart[i]);
  const double2 p = d.pos[i];
  const float th = d.theta[i];
  if (sx) {
    sx[i] = p;
    sth[i] = th;
  }
  float thn;
  const double2 y = bdem::em_move(c, R, (uint32_t)e, step, p, th, F, R.v0, &thn);
  const double2 pn = bdem::reflect_as(R, y, d.log_refl[(size_t)k_local * c.np + i]);
  d.pos[i] = pn;
  d.work[i] = bdem::split(pn);
  d.theta[i] = thn;
  if (z) z[i] = pn;
}

// Displacement of a logged pair (u, w) at positions pu, pw: w's; u's is its negative.
__device__ __forceinline__ double2 pair_disp(const BdConst &c, double2 pu, double2 pw) {
  const double dx = __dsub_rn(pw.x, pu.x), dy = __dsub_rn(pw.y, pu.y);
  const double r = sqrt(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
  const double del = c.sigma - r;
  return make_double2(del * (dx / r), del * (dy / r));
}

// position after a logged pass: dd capped where the log says so, moved, reflected as logged
__device__ __forceinline__ double2 pass_moved(const BdDev &d, const BdConst &c, int i, double2 p, double2 dd, int f) {
  const double cap = 0.25 * c.sigma;
  const double mag = sqrt(__dadd_rn(__dmul_rn(dd.x, dd.x), __dmul_rn(dd.y, dd.y)));
  const double sc = (f & 16) ? cap / mag : 1.0;
  const double2 y = make_double2(bdem::snapd(__dadd_rn(p.x, __dmul_rn(dd.x, sc)), c.q, c.inv_q),
                                 bdem::snapd(__dadd_rn(p.y, __dmul_rn(dd.y, sc)), c.q, c.inv_q));
  return bdem::reflect_as(d.rep[d.rep_of[i]], y, f & 15);
}

// A logged pass in one launch, for passes of few pairs.  What bounds these
// passes is launches: every block looks over all pairs of the pass and takes
// those with an end among its own BD_ADJ_OWN disks, so that their sums stay in
// shared memory and no second launch has to wait for them.  With k_vjp_pass
// forward and reverse step of a 4096-disk rollout fell from 171.6 to 159.3 us
// (three launches fewer per step with a pass).  z: the positions
// before the pass (all blocks read it), zn (or null): where those after it are
// kept for the next pass; zd: the displacement sums.
#define BD_ADJ_OWN 64
__global__ void __launch_bounds__(BD_ADJ_OWN) k_rp_pass(BdDev d, BdConst c, int pass, int pb, int pe, const double2 *z,
                                                        double2 *zd, double2 *zn) {
  __shared__ double2 acc[BD_ADJ_OWN];
  const int b0 = blockIdx.x * BD_ADJ_OWN, i = b0 + threadIdx.x;
  const int e = d.ext_id[i], f = d.log_pflags[(size_t)pass * c.np + i];
  const double2 p = z[i];
  acc[threadIdx.x] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int k = pb + threadIdx.x; k < pe; k += BD_ADJ_OWN) {
    const int2 pr = d.log_pairs[k];
    const int u = pr.x - b0, w = pr.y - b0;
    const bool ou = u >= 0 && u < BD_ADJ_OWN, ow = w >= 0 && w < BD_ADJ_OWN;
    if (!ou && !ow) continue;
    const double2 v = pair_disp(c, z[pr.x], z[pr.y]);
    if (ou) {
      atomic_add_d(&acc[u].x, -v.x);
      atomic_add_d(&acc[u].y, -v.y);
    }
    if (ow) {
      atomic_add_d(&acc[w].x, v.x);
      atomic_add_d(&acc[w].y, v.y);
    }
  }
  __syncthreads();
  if (e < 0) return;
  const double2 dd = acc[threadIdx.x];
  zd[i] = dd;
  double2 pn = p;
  if (dd.x != 0.0 || dd.y != 0.0 || f != 0) {
    pn = pass_moved(d, c, i, p, dd, f);
    d.pos[i] = pn;
    d.work[i] = bdem::split(pn);
  }
  if (zn) zn[i] = pn;
}

// displacements of a logged pass at the current positions (disp must be zero)
__global__ void k_rp_disp(BdDev d, BdConst c, int pair_begin, int pair_end) {
  const int k = pair_begin + blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= pair_end) return;
  const int2 pr = d.log_pairs[k];
  const double2 v = pair_disp(c, d.pos[pr.x], d.pos[pr.y]);
  atomic_add_d(&d.disp[pr.x].x, -v.x);
  atomic_add_d(&d.disp[pr.x].y, -v.y);
  atomic_add_d(&d.disp[pr.y].x, v.x);
  atomic_add_d(&d.disp[pr.y].y, v.y);
}

// apply a logged pass: cap where the log says so, move, reflect as logged; z, zd
// (or null) keep the positions before it and its displacement sums, zn (or null)
// the positions after it
__global__ void k_rp_apply(BdDev d, BdConst c, int pass, double2 *z, double2 *zd, double2 *zn) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= c.np || d.ext_id[i] < 0) return;
  const int f = d.log_pflags[(size_t)pass * c.np + i];
  const double2 dd = d.disp[i];
  if (z) {
    z[i] = d.pos[i];
    zd[i] = dd;
  }
  if (zn) zn[i] = d.pos[i];
  if (dd.x == 0.0 && dd.y == 0.0 && f == 0) return;
  const double2 pn = pass_moved(d, c, i, d.pos[i], dd, f);
  d.pos[i] = pn;
  d.work[i] = bdem::split(pn);
  if (zn) zn[i] = pn;
  d.disp[i] = make_double2(0.0, 0.0);
}

// ---------------------------------------------------------------- backward

// mu = R^T lambda
__device__ __forceinline__ double2 mirrored(double2 mu, int f) {
  if (((f & 1) != 0) != ((f & 2) != 0)) mu.x = -mu.x;   // an odd number of mirrors
  if (((f & 4) != 0) != ((f & 8) != 0)) mu.y = -mu.y;
  return mu;
}

// mu_d = cap'^T mu of disk i (zd holds d_j(z_j))
__device__ __forceinline__ double2 uncapped(const BdConst &c, double2 mu, int f, const double2 *zd, int i) {
  if (!(f & 16)) return mu;
  const double2 dd = zd[i];
  const double m = sqrt(dd.x * dd.x + dd.y * dd.y);
  const double ux = dd.x / m, uy = dd.y / m;
  const double s = 0.25 * c.sigma / m;
  const double dot = ux * mu.x + uy * mu.y;
  return make_double2(s * (mu.x - dot * ux), s * (mu.y - dot * uy));
}

// pair term G (mu_d_u - mu_d_w) of u at positions pu, pw; w's is its negative
__device__ __forceinline__ double2 pair_term(const BdConst &c, double2 pu, double2 pw, double2 mu, double2 mw) {
  const double vx = pw.x - pu.x, vy = pw.y - pu.y;
  const double r = sqrt(vx * vx + vy * vy);
  const double nx = vx / r, ny = vy / r;
  const double a = c.sigma / r;
  // G = a (I - n n^T) - I
  const double gxx = a * (1.0 - nx * nx) - 1.0, gyy = a * (1.0 - ny * ny) - 1.0, gxy = -a * nx * ny;
  const double wx = mu.x - mw.x, wy = mu.y - mw.y;
  return make_double2(gxx * wx + gxy * wy, gxy * wx + gyy * wy);
}

// pass, part 1: mu = R^T lambda; mu_d = cap'^T mu (zd holds d_j(z_j)); lambda = mu
__global__ void k_vjp_pass_mu(BdDev d, BdConst c, int pass, const double2 *zd, double2 *lam, double2 *mud) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= c.np || d.ext_id[i] < 0) return;
  const int f = d.log_pflags[(size_t)pass * c.np + i];
  const double2 mu = mirrored(lam[i], f);
  lam[i] = mu;
  mud[i] = uncapped(c, mu, f, zd, i);
}

// pass, part 2: pair terms lambda_u += G (mu_d_u - mu_d_w), lambda_w -= the same
__global__ void k_vjp_pass_pairs(BdDev d, BdConst c, const double2 *z, int pair_begin, int pair_end,
                                 double2 *lam, const double2 *mud) {
  const int k = pair_begin + blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= pair_end) return;
  const int2 pr = d.log_pairs[k];
  const double2 t = pair_term(c, z[pr.x], z[pr.y], mud[pr.x], mud[pr.y]);
  atomic_add_d(&lam[pr.x].x, t.x);
  atomic_add_d(&lam[pr.x].y, t.y);
  atomic_add_d(&lam[pr.y].x, -t.x);
  atomic_add_d(&lam[pr.y].y, -t.y);
}

// what k_vjp_em_refl does for one disk, from lambda after the step's passes
__device__ __forceinline__ double2 em_refl(const BdDev &d, const BdConst &c, int k_local, int i, bool live,
                                           const double2 *x, double2 lam, float4 *vx, float2 *vm) {
  if (!live) {
    vx[i] = make_float4(1.0e18f, 1.0e18f, 0.f, 0.f);
    vm[i] = make_float2(0.f, 0.f);
    return lam;
  }
  const double2 mu = mirrored(lam, d.log_refl[(size_t)k_local * c.np + i]);
  vx[i] = bdem::split(x[i]);
  vm[i] = make_float2((float)mu.x, (float)mu.y);
  return mu;
}

// Both parts of a pass in one launch, for passes of few pairs (see k_rp_pass):
// mu_d of a pair's ends is formed where the pair is taken, lambda goes from lin
// to lout.  x not null: the pass is the step's first, and the mirrors of its
// move and the force adjoint's FP32 copies are done with it.
__global__ void __launch_bounds__(BD_ADJ_OWN) k_vjp_pass(BdDev d, BdConst c, int pass, int pb, int pe, const double2 *z,
                                                         const double2 *zd, const double2 *lin, double2 *lout,
                                                         int k_local, const double2 *x, float4 *vx, float2 *vm) {
  __shared__ double2 acc[BD_ADJ_OWN];
  const unsigned char *const flags = d.log_pflags + (size_t)pass * c.np;
  const int b0 = blockIdx.x * BD_ADJ_OWN, i = b0 + threadIdx.x;
  const bool live = d.ext_id[i] >= 0;
  const double2 lam = lin[i];
  const int f = flags[i];
  acc[threadIdx.x] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int k = pb + threadIdx.x; k < pe; k += BD_ADJ_OWN) {
    const int2 pr = d.log_pairs[k];
    const int u = pr.x - b0, w = pr.y - b0;
    const bool ou = u >= 0 && u < BD_ADJ_OWN, ow = w >= 0 && w < BD_ADJ_OWN;
    if (!ou && !ow) continue;
    const int fu = flags[pr.x], fw = flags[pr.y];
    const double2 mu = uncapped(c, mirrored(lin[pr.x], fu), fu, zd, pr.x);
    const double2 mw = uncapped(c, mirrored(lin[pr.y], fw), fw, zd, pr.y);
    const double2 t = pair_term(c, z[pr.x], z[pr.y], mu, mw);
    if (ou) {
      atomic_add_d(&acc[u].x, t.x);
      atomic_add_d(&acc[u].y, t.y);
    }
    if (ow) {
      atomic_add_d(&acc[w].x, -t.x);
      atomic_add_d(&acc[w].y, -t.y);
    }
  }
  __syncthreads();
  double2 out = lam;
  if (live) {
    const double2 mu = mirrored(lam, f), a = acc[threadIdx.x];
    out = make_double2(mu.x + a.x, mu.y + a.y);
  }
  if (x) out = em_refl(d, c, k_local, i, live, x, out, vx, vm);
  lout[i] = out;
}

// move, part 1: mu = R0^T lambda (in place), and the FP32 copies the force
// adjoint reads: the positions' (hi, lo) pairs (inert slots far away) and mu
__global__ void k_vjp_em_refl(BdDev d, BdConst c, int k_local, const double2 *x, double2 *lam, float4 *vx,
                              float2 *vm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= c.np) return;
  const bool live = d.ext_id[i] >= 0;
  const double2 mu = em_refl(d, c, k_local, i, live, x, lam[i], vx, vm);
  if (live) lam[i] = mu;
}

__device__ __forceinline__ double adj_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// move, part 2: all-pairs force adjoint over one chunk of j (blockIdx.y).
// vx, vm: positions at the step start and mu = R0^T lambda, FP32 (k_vjp_em_refl).
// jpart[chunk][i] = sum over the chunk's j of M(r_ij)(A_ij mu_i - A_ji mu_j);
// gpart[block][0..3] = sum over the block's i of mu_i . S_{i,b} sorted by
// (s_i, b), gpart[block][4] = sum mu_i . e(theta_i) (chunk 0 only).  Partial
// sums are reduced in a fixed order by k_vjp_force_sum.
// A single-system handle only: every slot is one system's disk.
//
// Bound by the FP32 pipe: 22 lane operations per ordered pair, in packed f32x2
// instructions for two disks i per thread.  Blocks and tiles of j hold one
// species each (slots are species-major in whole 512-disk blocks), so both table
// entries are constants of the tile.  In a tile of the block's own species
// A_ij = A_ji is taken out of the sum, w = mu_i - mu_j, and the pair j = i needs
// no test: w and r are exactly 0 there.  Between two species A_ji mu_j is formed
// once per j.  A tile's sums are FP32, sums beyond a tile FP64 (sixteen FP64
// instructions a thread and tile, a sixth of the time its FP32 work takes).
// Chunks go down to one tile of 128 j so that small systems still have about
// eight blocks per SM.  One scalar pair at a time in 256 blocks, with FP64
// staging and shared FP64 atomics, it took 62 us at 4096 disks; a 40-step
// rollout with its reverse pass went from 10.8 to 8.0 ms.
__global__ void __launch_bounds__(BD_ADJ_T, 6) k_vjp_force(BdDev d, BdConst c, const float4 *vx, const float2 *vm,
                                                           const float *th, const double2 *mu, int jchunk,
                                                           double2 *jpart, double *gpart) {
  __shared__ ulonglong2 sh[BD_ADJ_T], sl[BD_ADJ_T], sm[BD_ADJ_T];   // ((v, v), (w, w)) of the hi, lo parts, -A_ji mu_j
  __shared__ double sg[BD_ADJ_T / 32][3];
  const int tid = threadIdx.x;
  const int ib = blockIdx.x * 2 * BD_ADJ_T;
  const BdRep &R = d.rep[0];
  const int si = d.tile_species[ib / BD_TJ];
  const int i0 = ib + tid, i1 = i0 + BD_ADJ_T;
  const float4 p0 = vx[i0], p1 = vx[i1];
  const float2 m0 = vm[i0], m1 = vm[i1];
  const u64 xh = pk2(p0.x, p1.x), yh = pk2(p0.y, p1.y), xl = pk2(p0.z, p1.z), yl = pk2(p0.w, p1.w);
  const u64 mx = pk2(m0.x, m1.x), my = pk2(m0.y, m1.y);
  double js[2][2] = {{0.0, 0.0}, {0.0, 0.0}};   // [i0, i1][x, y]
  double gs[2][2][2] = {};                      // [species of j][i0, i1][x, y]
  const u64 eps2 = pk2(1e-20f, 1e-20f), m3 = pk2(-3.f, -3.f);
  const int jb = blockIdx.y * jchunk, je = min(c.np, jb + jchunk);
  for (int j0 = jb; j0 < je; j0 += BD_ADJ_T) {
    const int sj = d.tile_species[j0 / BD_TJ];
    const bool same = sj == si;
    const float aij = R.alpha[BD_MAX_SPECIES * si + sj], aji = R.alpha[BD_MAX_SPECIES * sj + si];
    {
      const float4 q = vx[j0 + tid];
      const float2 m = vm[j0 + tid];
      const float nx = same ? -m.x : -__fmul_rn(aji, m.x), ny = same ? -m.y : -__fmul_rn(aji, m.y);
      sh[tid] = make_ulonglong2(pk2(q.x, q.x), pk2(q.y, q.y));
      sl[tid] = make_ulonglong2(pk2(q.z, q.z), pk2(q.w, q.w));
      sm[tid] = make_ulonglong2(pk2(nx, nx), pk2(ny, ny));
    }
    __syncthreads();
    const float ai = same ? 1.f : aij;
    const double sc = same ? (double)aij : 1.0;
    const u64 ai2 = pk2(ai, ai);
    u64 ax = 0ull, ay = 0ull, tx = 0ull, ty = 0ull;
#pragma unroll 4
    for (int k = 0; k < BD_ADJ_T; ++k) {
      const ulonglong2 qh = sh[k], ql = sl[k], qm = sm[k];
      const u64 rx = add2(sub2(xh, qh.x), sub2(xl, ql.x));
      const u64 ry = add2(sub2(yh, qh.y), sub2(yl, ql.y));
      const u64 r2 = fma2(rx, rx, fma2(ry, ry, eps2));
      float ra, rb;
      up2(r2, ra, rb);
      const u64 ir = pk2(rsqrt_apx(ra), rsqrt_apx(rb));
      const u64 ir2 = mul2(ir, ir);
      const u64 q3 = mul2(ir2, ir);
      const u64 wx = fma2(ai2, mx, qm.x), wy = fma2(ai2, my, qm.y);   // A_ij mu_i - A_ji mu_j, less the factor sc
      const u64 u = mul2(mul2(fma2(rx, wx, mul2(ry, wy)), ir2), m3);
      ax = fma2(fma2(rx, u, wx), q3, ax);   // (w - 3 r (r . w) / r^2) / r^3
      ay = fma2(fma2(ry, u, wy), q3, ay);
      tx = fma2(rx, q3, tx);   // r_ij / r^3
      ty = fma2(ry, q3, ty);
    }
    float a[2], b[2];
    up2(ax, a[0], a[1]);
    up2(ay, b[0], b[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      js[h][0] = __fma_rn(sc, (double)a[h], js[h][0]);
      js[h][1] = __fma_rn(sc, (double)b[h], js[h][1]);
    }
    up2(tx, a[0], a[1]);
    up2(ty, b[0], b[1]);
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if ((sj ? 1 : 0) == s)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          gs[s][h][0] += (double)a[h];
          gs[s][h][1] += (double)b[h];
        }
    __syncthreads();
  }
  double g[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = h ? i1 : i0;
    jpart[(size_t)blockIdx.y * c.np + i] = make_double2(js[h][0], js[h][1]);
    if (d.ext_id[i] < 0) continue;
    const double2 m = mu[i];
#pragma unroll
    for (int s = 0; s < 2; ++s) g[s] += m.x * gs[s][h][0] + m.y * gs[s][h][1];
    if (blockIdx.y == 0) {
      float st, ct;
      sincosf(th[i], &st, &ct);
      g[2] += m.x * (double)ct + m.y * (double)st;
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double v = adj_warp_sum(g[k]);
    if ((tid & 31) == 0) sg[tid >> 5][k] = v;
  }
  __syncthreads();
  if (tid < 5) {
    // slots 2 s_i + (species of j), and the v0 term
    const int k = tid == 4 ? 2 : tid - 2 * (si ? 1 : 0);
    double v = 0.0;
    if (k >= 0 && k < 2 || tid == 4)
      for (int w = 0; w < BD_ADJ_T / 32; ++w) v += sg[w][k];
    gpart[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 5 + tid] = v;
  }
}

// lambda_i = mu_i + dt sum over chunks of jpart; the last block instead adds
// dt times the sums over the nblocks of gpart to the gradient, in a fixed order
__global__ void __launch_bounds__(64) k_vjp_force_sum(BdDev d, BdConst c, int nchunk, const double2 *jpart, double2 *lam,
                                                      int nblocks, const double *gpart, double *grad) {
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double s[5][64];
    for (int k = 0; k < 5; ++k) {
      double v = 0.0;
      for (int b = threadIdx.x; b < nblocks; b += 64) v += gpart[(size_t)b * 5 + k];
      s[k][threadIdx.x] = v;
    }
    for (int w = 32; w > 0; w >>= 1) {
      __syncthreads();
      if ((int)threadIdx.x < w)
        for (int k = 0; k < 5; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + w];
    }
    if (threadIdx.x == 0)
      for (int k = 0; k < 5; ++k) grad[k] += d.rep[0].dt * s[k][0];
    return;
  }
  const int i = blockIdx.x * 64 + threadIdx.x;
  if (i >= c.np || d.ext_id[i] < 0) return;
  double jx = 0.0, jy = 0.0;
#pragma unroll 8
  for (int k = 0; k < nchunk; ++k) {
    const double2 v = jpart[(size_t)k * c.np + i];
    jx += v.x;
    jy += v.y;
  }
  const double dt = d.rep[0].dt;
  const double2 m = lam[i];
  lam[i] = make_double2(m.x + dt * jx, m.y + dt * jy);
}

// ---------------------------------------------------------------- loss

// per-species sums of |x_T - x_0|^2 and counts (acc[0..1] sums, acc[2..3] counts)
// per-species sums of |x_T - x_0|^2 and counts, in a fixed order (one block:
// thread t takes disks t, t + 1024, ...; then a fixed tree), so that the loss
// is the same number on every run
__global__ void __launch_bounds__(1024) k_msd_sums(BdDev d, BdConst c, const double2 *x0, double *acc) {
  __shared__ double sh[4][1024];
  const int t = threadIdx.x;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = t; i < c.np; i += 1024) {
    if (d.ext_id[i] < 0) continue;
    const double2 p = d.pos[i], q = x0[i];
    const double dx = p.x - q.x, dy = p.y - q.y;
    const int s = d.species[i] ? 1 : 0;
    v[s] += dx * dx + dy * dy;
    v[2 + s] += 1.0;
  }
  for (int k = 0; k < 4; ++k) sh[k][t] = v[k];
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (t < w)
      for (int k = 0; k < 4; ++k) sh[k][t] += sh[k][t + w];
    __syncthreads();
  }
  if (t < 4) acc[t] = sh[t][0];
}

// loss = sum_s (MSD_s - target)^2 and its gradient lambda_i = dscale dL/dx_i
__global__ void k_msd_loss_grad(BdDev d, BdConst c, const double2 *x0, const double *acc,
                                double target, double dscale, double2 *lam, double *loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double msd[2], cnt[2];
  for (int s = 0; s < 2; ++s) {
    cnt[s] = acc[2 + s];
    msd[s] = cnt[s] > 0 ? acc[s] / cnt[s] : 0.0;
  }
  if (i == 0 && loss) {
    double L = 0.0;
    for (int s = 0; s < 2; ++s)
      if (cnt[s] > 0) L += (msd[s] - target) * (msd[s] - target);
    *loss = L;
  }
  if (!lam || i >= c.np) return;
  if (d.ext_id[i] < 0) {
    lam[i] = make_double2(0.0, 0.0);
    return;
  }
  const int s = d.species[i] ? 1 : 0;
  const double2 p = d.pos[i], q = x0[i];
  const double f = dscale * 2.0 * (msd[s] - target) * 2.0 / cnt[s];
  lam[i] = make_double2(f * (p.x - q.x), f * (p.y - q.y));
}

// ---------------------------------------------------------------- pair-distance histogram loss
// h_b(x) = (1/n) sum over pairs i < j of K(r_ij - c_b), K(u) = exp(-u^2 / (2 s^2)),
// c_b = 2a + (b + 1/2) a/4 (b = 0..31), s = a/4; L = sum_b (h_b(x_T) - h_b(x_0))^2.
// Pairs farther than 12.5a are skipped: their kernel weight at the last
// centre (9.875a) is exp(-55) ~ 1e-24.  One warp per disk i; its lanes take
// the disks j in a fixed stride, and the warp's sums are combined by a
// shuffle tree, so every sum is in a fixed order (deterministic).

#define BD_HIST_BINS 32

__device__ __forceinline__ double hist_centre(double a, int b) {
  return __dadd_rn(__dmul_rn(2.0, a), __dmul_rn((double)b + 0.5, __dmul_rn(0.25, a)));
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// per-disk partial histograms: hpart[i][b] = sum over j > i of K(r_ij - c_b)
__global__ void k_hist_pairs(BdDev d, BdConst c, const double2 *x, double *hpart) {
  const int i = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= c.np) return;
  double acc[BD_HIST_BINS];
#pragma unroll
  for (int b = 0; b < BD_HIST_BINS; ++b) acc[b] = 0.0;
  if (d.ext_id[i] >= 0) {
    const double a = c.a, s = 0.25 * a, inv2s2 = 1.0 / (2.0 * s * s), rc = 12.5 * a;
    const double2 p = x[i];
    for (int j = i + 1 + lane; j < c.np; j += 32) {
      if (d.ext_id[j] < 0) continue;
      const double2 q = x[j];
      const double dx = __dsub_rn(q.x, p.x), dy = __dsub_rn(q.y, p.y);
      const double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
      if (r2 > rc * rc) continue;
      const double r = sqrt(r2);
#pragma unroll
      for (int b = 0; b < BD_HIST_BINS; ++b) {
        const double u = __dsub_rn(r, hist_centre(a, b));
        acc[b] += exp(-__dmul_rn(__dmul_rn(u, u), inv2s2));
      }
    }
  }
  double mine = 0.0;
#pragma unroll
  for (int b = 0; b < BD_HIST_BINS; ++b) {
    const double t = warp_sum_d(acc[b]);
    if (lane == b) mine = t;
  }
  hpart[(size_t)i * BD_HIST_BINS + lane] = mine;
}

// h = sum over disks of hpart / n in a fixed order (8 row groups per bin,
// combined in order); with h0: w_b = 2 (h_b - h0_b) / n and the loss
__global__ void __launch_bounds__(256) k_hist_reduce(BdConst c, const double *hpart, double inv_n,
                                                     const double *h0, double *h, double *w, double *loss) {
  __shared__ double part[8][BD_HIST_BINS];
  __shared__ double sq[BD_HIST_BINS];
  const int b = threadIdx.x & 31, g = threadIdx.x >> 5;
  double t = 0.0;
  for (int i = g; i < c.np; i += 8) t += hpart[(size_t)i * BD_HIST_BINS + b];
  part[g][b] = t;
  __syncthreads();
  if (g != 0) return;
  double hb = 0.0;
  for (int k = 0; k < 8; ++k) hb += part[k][b];
  hb *= inv_n;
  h[b] = hb;
  if (!h0) return;
  const double df = hb - h0[b];
  w[b] = 2.0 * df * inv_n;
  sq[b] = df * df;
  __syncwarp();
  if (b == 0 && loss) {
    double L = 0.0;
    for (int k = 0; k < BD_HIST_BINS; ++k) L += sq[k];
    *loss = L;
  }
}

// lam_i = dscale dL/dx_i = dscale sum_{j != i} g(r_ij) (x_i - x_j) / r_ij,
// g(r) = sum_b w_b dK/du(r - c_b), dK/du = -(u / s^2) K(u)
__global__ void k_hist_grad(BdDev d, BdConst c, const double2 *x, const double *w, double dscale,
                            double2 *lam) {
  const int i = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= c.np) return;
  double gx = 0.0, gy = 0.0;
  if (d.ext_id[i] >= 0) {
    const double a = c.a, s = 0.25 * a, inv_s2 = 1.0 / (s * s), inv2s2 = 0.5 * inv_s2, rc = 12.5 * a;
    double wb[BD_HIST_BINS];
#pragma unroll
    for (int b = 0; b < BD_HIST_BINS; ++b) wb[b] = w[b];
    const double2 p = x[i];
    for (int j = lane; j < c.np; j += 32) {
      if (j == i || d.ext_id[j] < 0) continue;
      const double2 q = x[j];
      const double dx = __dsub_rn(p.x, q.x), dy = __dsub_rn(p.y, q.y);
      const double r2 = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
      if (r2 > rc * rc) continue;
      const double r = sqrt(r2);
      double g = 0.0;
#pragma unroll
      for (int b = 0; b < BD_HIST_BINS; ++b) {
        const double u = __dsub_rn(r, hist_centre(a, b));
        g += wb[b] * (-u * inv_s2) * exp(-__dmul_rn(__dmul_rn(u, u), inv2s2));
      }
      gx += g / r * dx;
      gy += g / r * dy;
    }
  }
  gx = warp_sum_d(gx);
  gy = warp_sum_d(gy);
  if (lane == 0) lam[i] = make_double2(dscale * gx, dscale * gy);
}

// ---------------------------------------------------------------- launchers

cudaError_t bd_adj_hist(const BdDev &d, const BdConst &c, int n, const double2 *x, double *hpart, double *h,
                        const double *h0, double *w, double *loss, double2 *lam, double dscale, cudaStream_t s) {
  if (n <= 0) return cudaErrorInvalidValue;
  const int blocks = (int)(((size_t)c.np * 32 + 255) / 256);
  k_hist_pairs<<<blocks, 256, 0, s>>>(d, c, x, hpart);
  k_hist_reduce<<<1, 256, 0, s>>>(c, hpart, 1.0 / (double)n, h0, h, w, loss);
  if (h0 && lam) k_hist_grad<<<blocks, 256, 0, s>>>(d, c, x, w, dscale, lam);
  return cudaGetLastError();
}

cudaError_t bd_adj_rp_em(const BdDev &d, const BdConst &c, long long step, int k_local, double2 *sx, float *sth,
                         double2 *z, cudaStream_t s) {
  const int b = c.precision == 1 ? 32 : 256;   // as bd_launch_integrate
  k_rp_em<<<(c.np + b - 1) / b, b, 0, s>>>(d, c, step, k_local, sx, sth, z);
  return cudaGetLastError();
}

cudaError_t bd_adj_rp_pass(const BdDev &d, const BdConst &c, int pass, int pb, int pe, double2 *z, double2 *zd,
                           double2 *zn, cudaStream_t s) {
  if (z && pe - pb <= c.adj_pairs) {   // (np is a multiple of the blocks' 64 disks)
    k_rp_pass<<<c.np / BD_ADJ_OWN, BD_ADJ_OWN, 0, s>>>(d, c, pass, pb, pe, z, zd, zn);
    return cudaGetLastError();
  }
  if (pe > pb) k_rp_disp<<<(pe - pb + 255) / 256, 256, 0, s>>>(d, c, pb, pe);
  k_rp_apply<<<(c.np + 255) / 256, 256, 0, s>>>(d, c, pass, z, zd, zn);
  return cudaGetLastError();
}

cudaError_t bd_adj_vjp_pass(const BdDev &d, const BdConst &c, int pass, int pb, int pe, const double2 *z,
                            const double2 *zd, double2 *lam, double2 *mud, cudaStream_t s) {
  k_vjp_pass_mu<<<(c.np + 255) / 256, 256, 0, s>>>(d, c, pass, zd, lam, mud);
  if (pe > pb) k_vjp_pass_pairs<<<(pe - pb + 255) / 256, 256, 0, s>>>(d, c, z, pb, pe, lam, mud);
  return cudaGetLastError();
}

cudaError_t bd_adj_vjp_pass1(const BdDev &d, const BdConst &c, int pass, int pb, int pe, const double2 *z,
                             const double2 *zd, const double2 *lin, double2 *lout, int k_local, const double2 *x,
                             float4 *vx, float2 *vm, cudaStream_t s) {
  k_vjp_pass<<<c.np / BD_ADJ_OWN, BD_ADJ_OWN, 0, s>>>(d, c, pass, pb, pe, z, zd, lin, lout, k_local, x, vx, vm);
  return cudaGetLastError();
}

// chunks of j of the force adjoint: about eight blocks for each SM, of whole tiles
int bd_adj_force_chunks(const BdConst &c, int *jchunk) {
  const int nbi = c.np / (2 * BD_ADJ_T), ntile = c.np / BD_ADJ_T;   // np is a multiple of 512
  int nch = (8 * 152 + nbi - 1) / nbi;
  nch = nch < 1 ? 1 : (nch > ntile ? ntile : nch);
  const int tiles_per = (ntile + nch - 1) / nch;
  *jchunk = tiles_per * BD_ADJ_T;
  return (c.np + *jchunk - 1) / *jchunk;
}

// vx, vm: np FP32 positions and multipliers of scratch; ready: a pass has set them
cudaError_t bd_adj_vjp_em(const BdDev &d, const BdConst &c, int k_local, const double2 *x, const float *th,
                          double2 *lam, float4 *vx, float2 *vm, double2 *jpart, double *gpart, double *grad,
                          bool ready, cudaStream_t s) {
  if (!ready) k_vjp_em_refl<<<(c.np + 255) / 256, 256, 0, s>>>(d, c, k_local, x, lam, vx, vm);
  int jchunk = 0;
  const int nch = bd_adj_force_chunks(c, &jchunk);
  const int nbi = c.np / (2 * BD_ADJ_T);
  k_vjp_force<<<dim3(nbi, nch), BD_ADJ_T, 0, s>>>(d, c, vx, vm, th, lam, jchunk, jpart, gpart);
  k_vjp_force_sum<<<(c.np + 63) / 64 + 1, 64, 0, s>>>(d, c, nch, jpart, lam, nbi * nch, gpart, grad);
  return cudaGetLastError();
}

cudaError_t bd_adj_msd(const BdDev &d, const BdConst &c, const double2 *x0, double *acc, double target,
                       double dscale, double2 *lam, double *loss, cudaStream_t s) {
  k_msd_sums<<<1, 1024, 0, s>>>(d, c, x0, acc);
  k_msd_loss_grad<<<(c.np + 255) / 256, 256, 0, s>>>(d, c, x0, acc, target, dscale, lam, loss);
  return cudaGetLastError();
}
