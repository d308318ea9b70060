// Triangulation stages of one time step, as one persistent cooperative
// kernel (Algorithm 1 lines 5-7, Sec. 4.3-4.4):
//
//   P  validity (Sec. 4.3): r0_ij . r1_ij < 0 on any triangulation edge with a
//      moved end point rejects the step; every triangle with a moved corner is
//      re-oriented and flagged "inverted" when not strictly counter-clockwise;
//      in the same pass the Lawson marks (L) and the overlap scan (O) below.
//   R  inversion repair: an edge between an inverted triangle and its
//      neighbour is flipped when both triangles of the other diagonal come out
//      counter-clockwise -- the orientation form of Eq. (predicate) (the
//      moved vertex lies inside the neighbour's triangle, Fig. 4).  Rounds
//      repeat until no triangle is inverted; no candidate left => reject.
//   F  Lawson flips (Sec. 4.1, Navarro et al.): an edge whose opposite vertex
//      lies strictly inside the circumcircle of the other triangle is flipped;
//      rounds repeat until none is left.  Only edges touching a triangle that
//      moved or flipped are re-tested: by the flip itself, which tests the
//      four outer edges of its quadrilateral and registers the illegal ones
//      for the next round (fused rounds), or by a check pass after the round.
//   A  overlap correction (Algorithm 2): every real edge with r < sigma adds
//      -+ (sigma - r) r_hat to its end points' displacement (fixed-point
//      integer atomics: the sums do not depend on the order); each
//      disk then moves by its sum capped at sigma/4 (Sec. 4.4) and reflects at
//      the walls.  The sums are those of the scan of P, kept through fused
//      Lawson rounds (a flip withdraws the contribution of the diagonal it
//      removes and adds that of the one it draws).  Then P-R-F run again on
//      the moved disks, and the loop ends
//      when a pass over the Delaunay edges of the current positions finds no
//      overlap (the closest pair of a point set is a Delaunay edge, so no pair
//      anywhere is closer than sigma).
//
// Parallel flips: a candidate edge claims the six triangles its flip touches
// (the pair and the four across its outer edges) with a 64-bit atomicMax of
// (round, corner id); an edge that holds all six claims flips in place (the
// two triangle slots are reused) and rewrites its neighbours' back-pointers in
// the same round, since no other flip of the round touches them.
//
// Predicates: orientation and incircle are exact (integer arithmetic on the
// position grid, predicates.cuh), behind an FP32 filter that decides the clear
// cases from the disks' FP32 (hi, lo) position pairs.
//
// Grid-wide barriers spin with a time limit: a barrier that waits longer
// than BD_BARRIER_TIMEOUT_NS sets BD_ERR_DEVICE_TIMEOUT and every block leaves.
// On any failure the step is undone from the launch's undo journal: the first
// change a launch makes to a triangle (a flip, its back-pointers, a periodic
// shift) records the triangle's corners and neighbours as they were.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include "bd_internal.h"
#include "em.cuh"
#include "gridsync.cuh"
#include "predicates.cuh"

#define BD_DT_THREADS 256
#define BD_DT_LIST 2048       // triangles a block looks over at a time for the dirty ones
#define BD_DTC_THREADS 512   // threads per block of the cluster form

using namespace bdgs;

namespace {

enum { STAGE_P = 0, STAGE_R = 1, STAGE_F = 2, STAGE_A = 3, STAGE_PL = 4 };

// lead thread only: charge the time since the last mark to a stage
__device__ __forceinline__ void stage_tick(BdCtl *ctl, int stage, unsigned long long &mark) {
  const unsigned long long now = gtimer();
  ctl->st_stage_ns[stage] += now - mark;
  ctl->st_stage_cnt[stage] += 1;
  mark = now;
}

__device__ __forceinline__ int vk(const int4 &v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }
__device__ __forceinline__ void set_vk(int4 &v, int k, int val) {
  if (k == 0) v.x = val; else if (k == 1) v.y = val; else v.z = val;
}

struct Ctx {
  const BdDev &d;     // the kernel's parameters, where they lie
  const BdConst &c;
  bdpred::Grid g;
  int T;
  int np;
  float sig2f;   // sigma^2 (1 + 1e-5): FP32 screen of the overlap scan
  unsigned jstamp;   // this launch's undo-journal mark (odd)
  int *cl_n;         // lengths of the candidate lists
};

// FP32 filters in front of the exact integer predicates.  Every disk's
// position is also held as an FP32 pair (x_hi, x_lo) with x_hi + x_lo equal to
// the FP64 position to ~1e-11 a (the sweeps' copy), so a coordinate
// difference (b_hi - a_hi) + (b_lo - a_lo) carries one FP32 rounding of
// itself (relative 2^-24).  The determinant is then evaluated in FP32 with
// explicit rounding and compared with a bound on its error relative to the
// permanent (the same expression with absolute values): Shewchuk's bounds for
// exact inputs (3e-16 / 1.1e-15 relative in FP64, i.e. about 4 and 11 units
// of the working precision) plus one unit per input factor, times a safety
// factor of about four.  Outside the bound the FP32 sign is the exact sign;
// inside it the integer path decides.  Ghost points hold the same pairs (rows
// beside the walls: a test with one used to take the integer path, and the
// threads that did set the length of the whole pass), and a corner with an
// image shift takes its differences from the integer grid instead, one
// rounding each.
__device__ __forceinline__ float fdiff(float bh, float bl, float ah, float al) {
  return __fadd_rn(__fsub_rn(bh, ah), __fsub_rn(bl, al));
}

// The exact integer paths are rare (the filters decide almost every case) and
// long; they are kept out of line, one copy each, so that a thread that needs
// one fetches a single shared instruction stream rather than a cold inlined
// copy at every call site (a miss in the instruction cache costs about an L2
// round trip per line, and the slowest thread of a pass sets its length).  For
// the same reason the overlap of a pair and the registration of a candidate are
// out of line, and the loops over a triangle's edges and a flip's outer edges
// are not unrolled: in a small system a launch runs each phase's code once or
// twice, and waiting for instructions was the largest stall after the barriers.
__device__ __noinline__ int orient_exact(const double2 *__restrict__ pos, bdpred::Grid g, int a, int b, int c) {
  const double2 pa = pos[a], pb = pos[b], pc = pos[c];
  return bdpred::orient(pa.x, pa.y, pb.x, pb.y, pc.x, pc.y, g);
}

__device__ __noinline__ int incircle_exact(const double2 *__restrict__ pos, bdpred::Grid g, int a, int b, int c,
                                           int p) {
  const double2 pa = pos[a], pb = pos[b], pc = pos[c], pp = pos[p];
  return bdpred::incircle(pa.x, pa.y, pb.x, pb.y, pc.x, pc.y, pp.x, pp.y, g);
}

__device__ __noinline__ int orient_lifted(long long ax, long long ay, long long bx, long long by, long long cx,
                                          long long cy) {
  return bdpred::orient_int(ax, ay, bx, by, cx, cy);
}

__device__ __noinline__ int incircle_lifted(long long ax, long long ay, long long bx, long long by, long long cx,
                                            long long cy, long long px, long long py) {
  return bdpred::incircle_int(ax, ay, bx, by, cx, cy, px, py);
}

// Algorithm 2's per-disk displacement sums as fixed-point integers in the
// disp words: integer adds are associative, so the sum (and every position
// after the pass) does not depend on the order the edges arrive in.  A
// contribution is rounded to disp_unscale (a small fraction of the position
// grid) once; zero is the same bit pattern in both readings of the words.
// (A pass applies the sums of the disks marked in hit; a disk whose contributions
// were withdrawn again keeps its mark and a sum of 0.)
__device__ __forceinline__ void disp_add(const BdDev &d, const BdConst &c, int i, double vx, double vy) {
  long long *w = (long long *)&d.disp[i];
  atomicAdd((unsigned long long *)&w[0], (unsigned long long)__double2ll_rn(__dmul_rn(vx, c.disp_scale)));
  atomicAdd((unsigned long long *)&w[1], (unsigned long long)__double2ll_rn(__dmul_rn(vy, c.disp_scale)));
}
__device__ __forceinline__ double2 disp_get(const Ctx &x, int i) {
  const longlong2 w = *(const longlong2 *)&x.d.disp[i];
  return make_double2(__dmul_rn((double)w.x, x.c.disp_unscale), __dmul_rn((double)w.y, x.c.disp_unscale));
}

// Algorithm 2's overlap test of the disk pair (u, w), w's image shifted by
// (rsx, rsy) L: an exact pre-test in grid units, |r_w - r_u|^2 <= (sigma/q)^2
// (1 + 1e-9), then the decision r < a_u + a_w in FP64 as the reference makes
// it (the difference of two grid values is exact in FP64).  On overlap the push
// of w, (a_u + a_w - r) (r_w - r_u) / r, and u's, the negative, are added to the
// sums (sgn = -1: withdrawn), the disks are marked, and the depth
// a_u + a_w - r is returned (0: no overlap).
__device__ __noinline__ double overlap_push(const BdDev &d, const BdConst &c, int u, int w, int rsx, int rsy,
                                            long long LQ, int sgn) {
  const bdpred::Grid g{c.q, c.inv_q, c.qshift};
  const double2 pu = d.pos[u], pw = d.pos[w];
  const int64_t ix = bdpred::to_int(pw.x, g) - bdpred::to_int(pu.x, g) + rsx * LQ;
  const int64_t iy = bdpred::to_int(pw.y, g) - bdpred::to_int(pu.y, g) + rsy * LQ;
  const bdpred::i128 ir2 = bdpred::add128(bdpred::smul64(ix, ix), bdpred::smul64(iy, iy));
  const bool near = ir2.hi < c.sig2q_hi || (ir2.hi == c.sig2q_hi && ir2.lo <= c.sig2q_lo);
  if (!near) return 0.0;
  const double dx = bdem::grid_to_double(ix, g.s), dy = bdem::grid_to_double(iy, g.s);
  const double r = sqrt(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
  const double sg = d.rad ? d.rad[u] + d.rad[w] : c.sigma;   // polydisperse: a_u + a_w
  if (!(r < sg)) return 0.0;
  const double del = sg - r;
  const double vx = sgn * (del * (dx / r)), vy = sgn * (del * (dy / r));
  disp_add(d, c, u, -vx, -vy);
  disp_add(d, c, w, vx, vy);
  d.hit[u] = 1;
  d.hit[w] = 1;
  return del;
}

// a test the FP32 filter could not decide (rare: near-degenerate inputs)
__device__ __forceinline__ void count_exact(const Ctx &x) {
  atomicAdd((unsigned long long *)&x.d.ctl->st_exact, 1ull);
}

// the filters themselves, on coordinate differences that each carry about one
// FP32 rounding of themselves: the sign, or 0 when the bound does not decide
__device__ __forceinline__ int orient_f(float bax, float bay, float cax, float cay) {
  const float l = __fmul_rn(bax, cay), r = __fmul_rn(bay, cax);
  const float det = __fsub_rn(l, r);
  const float bound = 1.5e-6f * __fadd_rn(fabsf(l), fabsf(r));
  return det > bound ? 1 : (-det > bound ? -1 : 0);
}

__device__ __forceinline__ int incircle_f(float adx, float ady, float bdx, float bdy, float cdx, float cdy) {
  const float bcl = __fmul_rn(bdx, cdy), bcr = __fmul_rn(bdy, cdx);
  const float cal = __fmul_rn(cdx, ady), car = __fmul_rn(cdy, adx);
  const float abl = __fmul_rn(adx, bdy), abr = __fmul_rn(ady, bdx);
  const float al = __fadd_rn(__fmul_rn(adx, adx), __fmul_rn(ady, ady));
  const float bl = __fadd_rn(__fmul_rn(bdx, bdx), __fmul_rn(bdy, bdy));
  const float cl = __fadd_rn(__fmul_rn(cdx, cdx), __fmul_rn(cdy, cdy));
  const float det = __fadd_rn(__fadd_rn(__fmul_rn(al, __fsub_rn(bcl, bcr)), __fmul_rn(bl, __fsub_rn(cal, car))),
                              __fmul_rn(cl, __fsub_rn(abl, abr)));
  const float perm =
      __fadd_rn(__fadd_rn(__fmul_rn(al, __fadd_rn(fabsf(bcl), fabsf(bcr))), __fmul_rn(bl, __fadd_rn(fabsf(cal), fabsf(car)))),
                __fmul_rn(cl, __fadd_rn(fabsf(abl), fabsf(abr))));
  const float bound = 4e-6f * perm;
  return det > bound ? 1 : (-det > bound ? -1 : 0);
}

// the filters on preloaded FP32 pairs (disks: all corners are disks, whose
// undecided tests are counted; ghost points hold the same FP32 pairs)
__device__ __forceinline__ int orient_pre(const Ctx &x, bool disks, const float4 &wa, const float4 &wb,
                                          const float4 &wc, int a, int b, int c) {
  const int o = orient_f(fdiff(wb.x, wb.z, wa.x, wa.z), fdiff(wb.y, wb.w, wa.y, wa.w),
                         fdiff(wc.x, wc.z, wa.x, wa.z), fdiff(wc.y, wc.w, wa.y, wa.w));
  if (o) return o;
  if (disks) count_exact(x);
  return orient_exact(x.d.pos, x.g, a, b, c);
}

__device__ __forceinline__ int incircle_pre(const Ctx &x, bool disks, const float4 &wa, const float4 &wb,
                                            const float4 &wc, const float4 &wp, int a, int b, int c, int p) {
  const int o = incircle_f(fdiff(wa.x, wa.z, wp.x, wp.z), fdiff(wa.y, wa.w, wp.y, wp.w),
                           fdiff(wb.x, wb.z, wp.x, wp.z), fdiff(wb.y, wb.w, wp.y, wp.w),
                           fdiff(wc.x, wc.z, wp.x, wp.z), fdiff(wc.y, wc.w, wp.y, wp.w));
  if (o) return o;
  if (disks) count_exact(x);
  return incircle_exact(x.d.pos, x.g, a, b, c, p);
}

// FP32 (hi, lo) pair of a disk or ghost point
__device__ __forceinline__ float4 work_of(const Ctx &x, int v) { return x.d.work[v]; }

__device__ __forceinline__ int orient_v(const Ctx &x, int a, int b, int c) {
  const bool disks = a < x.np && b < x.np && c < x.np;
  return orient_pre(x, disks, work_of(x, a), work_of(x, b), work_of(x, c), a, b, c);
}

__device__ __forceinline__ int incircle_v(const Ctx &x, int a, int b, int c, int p) {
  const bool disks = a < x.np && b < x.np && c < x.np && p < x.np;
  return incircle_pre(x, disks, work_of(x, a), work_of(x, b), work_of(x, c), work_of(x, p), a, b, c, p);
}

// Sec. 4.3 reversal test r0 . r1 < 0 of the edge u -> w, exact on the grid:
// r1 from the present positions, r0 from those before the move (ox, oy: the
// edge's image shift before the move, in units of LQ); only a disk that moved
// (mu, mw) has its position before the move in prev (for the launch's first
// pass, pos0)
__device__ __noinline__ bool reversed_grid(const double2 *__restrict__ prev, const double2 *__restrict__ pos,
                                           bdpred::Grid g, int u, int w, bool mu, bool mw, int ox, int oy, int rsx,
                                           int rsy, long long LQ) {
  const double2 a1 = pos[u], b1 = pos[w];
  const double2 a0 = mu ? prev[u] : a1, b0 = mw ? prev[w] : b1;
  const int64_t ux = bdpred::to_int(b0.x, g) - bdpred::to_int(a0.x, g) + ox * LQ;
  const int64_t uy = bdpred::to_int(b0.y, g) - bdpred::to_int(a0.y, g) + oy * LQ;
  const int64_t vx = bdpred::to_int(b1.x, g) - bdpred::to_int(a1.x, g) + rsx * LQ;
  const int64_t vy = bdpred::to_int(b1.y, g) - bdpred::to_int(a1.y, g) + rsy * LQ;
  return bdpred::sign128(bdpred::add128(bdpred::smul64(ux, vx), bdpred::smul64(uy, vy))) < 0;
}

// ---- periodic box: image shifts of triangle corners (Sec. 2.1, 4.1) ----
// Corner k of a triangle lies at pos[v_k] + L (sx_k, sy_k); the shifts are
// 2-bit two's-complement fields of tv.w (BD_TRI_SHIFT_BITS), all zero with
// walls, and corner 0 is kept at shift 0.  Straddling triangles are decided
// by the exact integer predicates on lifted grid coordinates.
__device__ __forceinline__ int sh2(int w, int bit) { return (((w >> bit) & 3) ^ 2) - 2; }
__device__ __forceinline__ int shx(int w, int k) { return sh2(w, 8 + 4 * k); }
__device__ __forceinline__ int shy(int w, int k) { return sh2(w, 10 + 4 * k); }
// the kernel is compiled twice: with walls (PER = false) every shift is the
// constant 0 and the shift arithmetic disappears
template <bool PER>
__device__ __forceinline__ int tshx(int w, int k) { return PER ? shx(w, k) : 0; }
template <bool PER>
__device__ __forceinline__ int tshy(int w, int k) { return PER ? shy(w, k) : 0; }
// the check-pass stamp of a triangle (bits 24-31 of tv.w)
__device__ __forceinline__ uint8_t tstamp(int w) { return (uint8_t)((unsigned)w >> BD_TRI_STAMP_SHIFT); }
__device__ __forceinline__ int with_stamp(int w, uint8_t s) {
  return (int)(((unsigned)w & ((1u << BD_TRI_STAMP_SHIFT) - 1u)) | ((unsigned)s << BD_TRI_STAMP_SHIFT));
}
__device__ __forceinline__ int put_shift(int k, int sx, int sy) {
  return ((sx & 3) << (8 + 4 * k)) | ((sy & 3) << (10 + 4 * k));
}
// the wrap of the last move of disk v: stored = geometric - L k
__device__ __forceinline__ int wrapx(uint8_t w) { return ((w & 3) ^ 2) - 2; }
__device__ __forceinline__ int wrapy(uint8_t w) { return (((w >> 2) & 3) ^ 2) - 2; }

struct Lift {
  long long x, y;
};

__device__ __forceinline__ Lift lift(const Ctx &x, int v, int sx, int sy, long long LQ) {
  const double2 p = x.d.pos[v];
  return {bdpred::to_int(p.x, x.g) + sx * LQ, bdpred::to_int(p.y, x.g) + sy * LQ};
}

// difference of two lifted coordinates, exact in grid units, rounded once to FP32
__device__ __forceinline__ float lift_diff(const Ctx &x, long long b, long long a) {
  return bdem::grid_to_float(b - a, x.g.s);
}

__device__ __forceinline__ long long rep_LQ(const Ctx &x, int v) { return x.d.rep[x.d.rep_of[v]].LQ; }

// orientation of corners (a, b, c) with shifts (sa, sb, sc)
__device__ __forceinline__ int orient_s(const Ctx &x, int a, int sax, int say, int b, int sbx, int sby, int c,
                                        int scx, int scy) {
  if ((sax | say | sbx | sby | scx | scy) == 0) return orient_v(x, a, b, c);
  const long long LQ = rep_LQ(x, a);
  const Lift A = lift(x, a, sax, say, LQ), B = lift(x, b, sbx, sby, LQ), C = lift(x, c, scx, scy, LQ);
  const int o = orient_f(lift_diff(x, B.x, A.x), lift_diff(x, B.y, A.y), lift_diff(x, C.x, A.x),
                         lift_diff(x, C.y, A.y));
  if (o) return o;
  return orient_lifted(A.x, A.y, B.x, B.y, C.x, C.y);
}

// in-circle test of p (shift sp) against triangle t's corners (shifts in w)
template <bool PER>
__device__ __forceinline__ int incircle_s(const Ctx &x, const int4 &v, int p, int spx, int spy) {
  const int w = v.w;
  if (!PER || ((w & BD_TRI_SHIFT_BITS) | spx | spy) == 0) return incircle_v(x, v.x, v.y, v.z, p);
  const long long LQ = rep_LQ(x, v.x);
  const Lift A = lift(x, v.x, shx(w, 0), shy(w, 0), LQ), B = lift(x, v.y, shx(w, 1), shy(w, 1), LQ);
  const Lift C = lift(x, v.z, shx(w, 2), shy(w, 2), LQ), P = lift(x, p, spx, spy, LQ);
  const int o = incircle_f(lift_diff(x, A.x, P.x), lift_diff(x, A.y, P.y), lift_diff(x, B.x, P.x),
                           lift_diff(x, B.y, P.y), lift_diff(x, C.x, P.x), lift_diff(x, C.y, P.y));
  if (o) return o;
  return incircle_lifted(A.x, A.y, B.x, B.y, C.x, C.y, P.x, P.y);
}

// shift, in the frame of triangle t (corner tab w), of the vertex opposite
// the edge facing corner k, read from the neighbour (tab w1, corner k1):
// t's corner k+1 is the neighbour's corner k1+2
template <bool PER>
__device__ __forceinline__ void opp_shift(int w, int k, int w1, int k1, int &sx, int &sy) {
  if (!PER) {
    sx = sy = 0;
    return;
  }
  const int ku = (k + 1) % 3, ku1 = (k1 + 2) % 3;
  sx = shx(w1, k1) + shx(w, ku) - shx(w1, ku1);
  sy = shy(w1, k1) + shy(w, ku) - shy(w1, ku1);
}

__device__ __forceinline__ double snap(double v, const bdpred::Grid &g) {
  return __dmul_rn(rint(__dmul_rn(v, g.inv_q)), g.q);
}

__device__ __forceinline__ float4 split_pos(double2 p) {
  float xh = __double2float_rn(p.x), yh = __double2float_rn(p.y);
  return make_float4(xh, yh, __double2float_rn(p.x - (double)xh), __double2float_rn(p.y - (double)yh));
}

// Claim the six triangles that flipping the edge facing corner cc touches:
// the pair and the four triangles across its outer edges.  An edge that
// holds all six claims owns them for the round, so its flip can rewrite the
// neighbours' back-pointers directly.
// the claims of the round of epoch e
__device__ __forceinline__ unsigned long long *claims(const Ctx &x, unsigned long long e) {
  return x.d.claim + (size_t)(e & 1ull) * x.T;
}

__device__ __forceinline__ void claim6(const int4 *tn, unsigned long long *cb, int t, int k, const int4 &nn, int o,
                                       unsigned long long key) {
  const int t1 = o / 3, k1 = o % 3;
  const int4 nn1 = tn[t1];
  atomicMax(&cb[t], key);
  atomicMax(&cb[t1], key);
  int e[4] = {vk(nn, (k + 1) % 3), vk(nn, (k + 2) % 3), vk(nn1, (k1 + 1) % 3), vk(nn1, (k1 + 2) % 3)};
  for (int m = 0; m < 4; ++m)
    if (e[m] >= 0) atomicMax(&cb[e[m] / 3], key);
}

__device__ __forceinline__ bool owns6(const Ctx &x, const unsigned long long *cb, int t0, int k0, const int4 &N0,
                                      int o0, unsigned long long key) {
  const int t1 = o0 / 3, k1 = o0 % 3;
  if (cb[t1] != key) return false;
  const int4 N1 = x.d.tn[t1];
  int e[4] = {vk(N0, (k0 + 1) % 3), vk(N0, (k0 + 2) % 3), vk(N1, (k1 + 1) % 3), vk(N1, (k1 + 2) % 3)};
  for (int m = 0; m < 4; ++m)
    if (e[m] >= 0 && cb[e[m] / 3] != key) return false;
  return true;
}

// Record triangle t, whose corners and neighbours are (V, N), in the undo
// journal before the launch first changes it (in its own slot: no list and no
// shared counter; an undo scans the marks).  A triangle is changed by one
// thread per phase (flips own the triangles they touch; the shift pass visits
// each triangle once), so the test of the mark needs no atomic.  A flip's
// outer neighbours are not journaled: their one change, the back-pointer, is
// rebuilt by the undo from the restored pair (they were adjacent before).
__device__ __forceinline__ void journal(const Ctx &x, int t, const int4 &V, const int4 &N, unsigned mark) {
  if (mark == x.jstamp) return;
  x.d.jmark[t] = x.jstamp;
  x.d.jtv[t] = V;
  x.d.jtn[t] = N;
}
// undo of a journaled triangle t: its corners and neighbours as they were, and
// its neighbours' back-pointers
__device__ __forceinline__ void unjournal(const BdDev &d, int t) {
  const int4 vs = d.jtv[t], ns = d.jtn[t];
  d.tv[t] = vs;
  d.tn[t] = ns;
  const int nk[3] = {ns.x, ns.y, ns.z};
  for (int k = 0; k < 3; ++k)
    if (nk[k] >= 0) ((int *)&d.tn[nk[k] / 3])[nk[k] % 3] = 3 * t + k;
}

// Flip the edge facing corner c0 in place (the two triangle slots are reused)
// and point the four outer neighbours, owned by this flip, at the new corners.
// Quad a-b-d-c with t0 = (a, b, c), t1 = (d, c, b) becomes t0 = (b, d, a),
// t1 = (c, a, d): the edge bc is replaced by ad.
template <bool PER>
__device__ void flip_owned(const Ctx &x, int c0, int o0, uint8_t stamp) {
  const int t0 = c0 / 3, k0 = c0 % 3, t1 = o0 / 3, k1 = o0 % 3;
  // the journal marks are loaded with the pair, and the pair's old values
  // journaled after the flip's own stores (they are held in registers)
  const unsigned m0 = x.d.jmark[t0], m1 = x.d.jmark[t1];
  int4 V0 = x.d.tv[t0], V1 = x.d.tv[t1], N0 = x.d.tn[t0], N1 = x.d.tn[t1];
  const int4 oV0 = V0, oV1 = V1, oN0 = N0, oN1 = N1;
  const int a = vk(V0, k0), b = vk(V0, (k0 + 1) % 3), c = vk(V0, (k0 + 2) % 3), dd = vk(V1, k1);
  const int n_ca = vk(N0, (k0 + 1) % 3), n_ab = vk(N0, (k0 + 2) % 3);
  const int n_bd = vk(N1, (k1 + 1) % 3), n_dc = vk(N1, (k1 + 2) % 3);
  set_vk(V0, k0, b);
  set_vk(V0, (k0 + 1) % 3, dd);
  set_vk(V0, (k0 + 2) % 3, a);
  set_vk(V1, k1, c);
  set_vk(V1, (k1 + 1) % 3, a);
  set_vk(V1, (k1 + 2) % 3, dd);
  set_vk(N0, k0, 3 * t1 + k1);
  set_vk(N0, (k0 + 1) % 3, n_ab);
  set_vk(N0, (k0 + 2) % 3, n_bd);
  set_vk(N1, k1, 3 * t0 + k0);
  set_vk(N1, (k1 + 1) % 3, n_dc);
  set_vk(N1, (k1 + 2) % 3, n_ca);
  // image shifts (periodic box): the new corners in t0's frame; d comes from
  // t1's frame, offset by b's shift difference between the two frames
  const int w0 = V0.w, w1 = V1.w;
  int nw0 = 0, nw1 = 0;
  if (PER && ((w0 | w1) & BD_TRI_SHIFT_BITS)) {
    const int Ax = shx(w0, k0), Ay = shy(w0, k0);
    const int Bx = shx(w0, (k0 + 1) % 3), By = shy(w0, (k0 + 1) % 3);
    const int Cx = shx(w0, (k0 + 2) % 3), Cy = shy(w0, (k0 + 2) % 3);
    const int Dx = shx(w1, k1) + Bx - shx(w1, (k1 + 2) % 3), Dy = shy(w1, k1) + By - shy(w1, (k1 + 2) % 3);
    // t0 = (b, d, a) at (k0, k0+1, k0+2); t1 = (c, a, d) at (k1, k1+1, k1+2)
    int sx0[3], sy0[3], sx1[3], sy1[3];
    sx0[k0] = Bx; sy0[k0] = By;
    sx0[(k0 + 1) % 3] = Dx; sy0[(k0 + 1) % 3] = Dy;
    sx0[(k0 + 2) % 3] = Ax; sy0[(k0 + 2) % 3] = Ay;
    sx1[k1] = Cx; sy1[k1] = Cy;
    sx1[(k1 + 1) % 3] = Ax; sy1[(k1 + 1) % 3] = Ay;
    sx1[(k1 + 2) % 3] = Dx; sy1[(k1 + 2) % 3] = Dy;
    for (int k = 0; k < 3; ++k) {
      nw0 |= put_shift(k, sx0[k] - sx0[0], sy0[k] - sy0[0]);
      nw1 |= put_shift(k, sx1[k] - sx1[0], sy1[k] - sy1[0]);
    }
  }
  // both new triangles: their edges are tested by the next check pass
  V0.w = with_stamp(nw0, stamp);
  V1.w = with_stamp(nw1, stamp);
  x.d.tv[t0] = V0;
  x.d.tv[t1] = V1;
  x.d.tn[t0] = N0;
  x.d.tn[t1] = N1;
  x.d.tinv[t0] = 0;
  x.d.tinv[t1] = 0;
  // t0 = (b, d, a), t1 = (c, a, d)
  if (n_ab >= 0) ((int *)&x.d.tn[n_ab / 3])[n_ab % 3] = 3 * t0 + (k0 + 1) % 3;
  if (n_bd >= 0) ((int *)&x.d.tn[n_bd / 3])[n_bd % 3] = 3 * t0 + (k0 + 2) % 3;
  if (n_dc >= 0) ((int *)&x.d.tn[n_dc / 3])[n_dc % 3] = 3 * t1 + (k1 + 1) % 3;
  if (n_ca >= 0) ((int *)&x.d.tn[n_ca / 3])[n_ca % 3] = 3 * t1 + (k1 + 2) % 3;
  journal(x, t0, oV0, oN0, m0);
  journal(x, t1, oV1, oN1, m1);
}

__device__ __forceinline__ unsigned long long claim_key(unsigned long long epoch, int corner) {
  return (epoch << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)corner);
}
__device__ __forceinline__ int key_corner(unsigned long long key) {
  return (int)(0xFFFFFFFFu - (unsigned)(key & 0xFFFFFFFFull));
}

// Register the edge facing corner cc (o: the corner across it) as a flip
// candidate of the round of epoch e: its six claims (cb), and its triangle in
// the round's list of owners -- once: the marking pass and the previous fused
// round both register owners for a round, and an owner listed twice would be
// flipped by two threads at once.
__device__ __noinline__ void register_edge(const int4 *tn, unsigned long long *cb, unsigned *clmark, int *list, int *n,
                                           unsigned long long e, int cc, int o) {
  const int t = cc / 3;
  claim6(tn, cb, t, cc % 3, tn[t], o, claim_key(e, cc));
  if (atomicExch(&clmark[t], (unsigned)e) == (unsigned)e) return;
  list[atomicAdd(n, 1)] = t;
}
__device__ __forceinline__ void register_edge(const Ctx &x, unsigned long long *cb, unsigned long long e, int cc, int o) {
  const int l = (int)(e % 3);
  register_edge(x.d.tn, cb, x.d.clmark, x.d.clist + (size_t)l * x.T, &x.cl_n[l], e, cc, o);
}

// Stamp triangle t for the check pass of generation byte s.  The word is
// shared with the corners' image shifts, which a flip of t by another thread
// may rewrite meanwhile: compare-and-swap keeps whichever shifts are current.
__device__ __forceinline__ void stamp_tri(const Ctx &x, int t, uint8_t s) {
  int *w = &x.d.tv[t].w;
  int old = *(volatile int *)w, seen;
  do {
    seen = old;
    old = atomicCAS(w, seen, with_stamp(seen, s));
  } while (old != seen);
}

// A fused Lawson round's flip of the candidate that triangle t0 registered for
// the round of epoch ce, if it holds its six claims (cb).  Its loads are issued
// by level, before any store and before the claims have decided -- t0's claim,
// tables and journal mark; the other triangle's, with t0's corners' FP32 pairs;
// the four outer neighbours' claims and corner tables; the opposite vertices'
// FP32 pairs -- since a round is as long as this chain (what a candidate that
// lost has read of triangles others are flipping is dropped).  It withdraws the
// overlap of diagonal bc, adds that of ad, flips, and tests the four outer
// edges, registering the illegal ones (claims in nb, keys of epoch ce + 1, owners
// listed once).  Returns the other triangle (-1: claims lost), the change in
// overlapping edges and the depth of an added overlap (0 if none).
struct FusedOut {
  int t1;
  int adj;
  double mx;
};
template <bool PER>
__device__ __forceinline__ FusedOut fused_flip(const Ctx &x, int t0, unsigned long long ce, const unsigned long long *cb,
                                               unsigned long long *nb) {
  const BdDev &d = x.d;
  FusedOut r = {-1, 0, 0.0};
  const unsigned long long ne = ce + 1;
  const unsigned long long key = cb[t0];
  const unsigned m0 = d.jmark[t0];
  const int4 oV0 = d.tv[t0], oN0 = d.tn[t0];
  const int c0 = key_corner(key);
  if ((key >> 32) != ce || c0 / 3 != t0) return r;
  const int k0 = c0 % 3, o0 = vk(oN0, k0), t1 = o0 / 3, k1 = o0 % 3;
  const int a = vk(oV0, k0), b = vk(oV0, (k0 + 1) % 3), c = vk(oV0, (k0 + 2) % 3);
  bool own = cb[t1] == key;
  const unsigned m1 = d.jmark[t1];
  const int4 oV1 = d.tv[t1], oN1 = d.tn[t1];
  const float4 Pa = work_of(x, a), Pb = work_of(x, b), Pc = work_of(x, c);
  const int dd = vk(oV1, k1);
  const int n_ca = vk(oN0, (k0 + 1) % 3), n_ab = vk(oN0, (k0 + 2) % 3);
  const int n_bd = vk(oN1, (k1 + 1) % 3), n_dc = vk(oN1, (k1 + 2) % 3);
  // outer edges in the order (t0, facing k0+1), (t0, k0+2), (t1, k1+1), (t1, k1+2)
  const int nbr[4] = {n_ab, n_bd, n_dc, n_ca};
  int4 Wn[4];
  unsigned long long cn[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    cn[m] = nbr[m] >= 0 ? cb[nbr[m] / 3] : key;
    Wn[m] = nbr[m] >= 0 ? d.tv[nbr[m] / 3] : make_int4(0, 0, 0, 0);
  }
  const float4 Pd = work_of(x, dd);
#pragma unroll
  for (int m = 0; m < 4; ++m) own = own && cn[m] == key;
  if (!own) return r;
  r.t1 = t1;
  int q[4];
  float4 Pq[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    q[m] = nbr[m] >= 0 ? vk(Wn[m], nbr[m] % 3) : 0;
    Pq[m] = nbr[m] >= 0 ? work_of(x, q[m]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // the new pair: t0 = (b, d, a) at (k0, k0+1, k0+2), t1 = (c, a, d) at (k1, k1+1, k1+2)
  int4 V0 = oV0, V1 = oV1, N0 = oN0, N1 = oN1;
  set_vk(V0, k0, b);
  set_vk(V0, (k0 + 1) % 3, dd);
  set_vk(V0, (k0 + 2) % 3, a);
  set_vk(V1, k1, c);
  set_vk(V1, (k1 + 1) % 3, a);
  set_vk(V1, (k1 + 2) % 3, dd);
  set_vk(N0, k0, 3 * t1 + k1);
  set_vk(N0, (k0 + 1) % 3, n_ab);
  set_vk(N0, (k0 + 2) % 3, n_bd);
  set_vk(N1, k1, 3 * t0 + k0);
  set_vk(N1, (k1 + 1) % 3, n_dc);
  set_vk(N1, (k1 + 2) % 3, n_ca);
  const int w0 = oV0.w, w1 = oV1.w;
  int nw0 = 0, nw1 = 0;
  int Ax = 0, Ay = 0, Bx = 0, By = 0, Cx = 0, Cy = 0, Dx = 0, Dy = 0;
  if (PER && ((w0 | w1) & BD_TRI_SHIFT_BITS)) {
    Ax = shx(w0, k0); Ay = shy(w0, k0);
    Bx = shx(w0, (k0 + 1) % 3); By = shy(w0, (k0 + 1) % 3);
    Cx = shx(w0, (k0 + 2) % 3); Cy = shy(w0, (k0 + 2) % 3);
    Dx = shx(w1, k1) + Bx - shx(w1, (k1 + 2) % 3); Dy = shy(w1, k1) + By - shy(w1, (k1 + 2) % 3);
    int sx0[3], sy0[3], sx1[3], sy1[3];
    sx0[k0] = Bx; sy0[k0] = By;
    sx0[(k0 + 1) % 3] = Dx; sy0[(k0 + 1) % 3] = Dy;
    sx0[(k0 + 2) % 3] = Ax; sy0[(k0 + 2) % 3] = Ay;
    sx1[k1] = Cx; sy1[k1] = Cy;
    sx1[(k1 + 1) % 3] = Ax; sy1[(k1 + 1) % 3] = Ay;
    sx1[(k1 + 2) % 3] = Dx; sy1[(k1 + 2) % 3] = Dy;
    for (int k = 0; k < 3; ++k) {
      nw0 |= put_shift(k, sx0[k] - sx0[0], sy0[k] - sy0[0]);
      nw1 |= put_shift(k, sx1[k] - sx1[0], sy1[k] - sy1[0]);
    }
  }
  V0.w = with_stamp(nw0, tstamp(w0));
  V1.w = with_stamp(nw1, tstamp(w1));
  // overlaps of the old and the new diagonal (a shifted edge takes the exact
  // test directly; a plain one is screened in FP32 first, as in a check pass)
  auto diag = [&](int u, int w, const float4 &Pu, const float4 &Pw, int sx, int sy, int sgn) {
    if (u >= x.np || w >= x.np) return;
    if ((sx | sy) == 0) {
      const float fx = fdiff(Pw.x, Pw.z, Pu.x, Pu.z), fy = fdiff(Pw.y, Pw.w, Pu.y, Pu.w);
      if (__fadd_rn(__fmul_rn(fx, fx), __fmul_rn(fy, fy)) > x.sig2f) return;
    }
    const long long LQ = (sx | sy) ? rep_LQ(x, u) : 0;
    const double del = overlap_push(d, x.c, u, w, sx, sy, LQ, sgn);
    if (del == 0.0) return;
    r.adj += sgn;
    if (sgn > 0) r.mx = fmax(r.mx, del);
  };
  diag(b, c, Pb, Pc, Cx - Bx, Cy - By, -1);
  diag(a, dd, Pa, Pd, Dx - Ax, Dy - Ay, 1);
  // the flip
  d.tv[t0] = V0;
  d.tv[t1] = V1;
  d.tn[t0] = N0;
  d.tn[t1] = N1;
  d.tinv[t0] = 0;
  d.tinv[t1] = 0;
  if (n_ab >= 0) ((int *)&d.tn[n_ab / 3])[n_ab % 3] = 3 * t0 + (k0 + 1) % 3;
  if (n_bd >= 0) ((int *)&d.tn[n_bd / 3])[n_bd % 3] = 3 * t0 + (k0 + 2) % 3;
  if (n_dc >= 0) ((int *)&d.tn[n_dc / 3])[n_dc % 3] = 3 * t1 + (k1 + 1) % 3;
  if (n_ca >= 0) ((int *)&d.tn[n_ca / 3])[n_ca % 3] = 3 * t1 + (k1 + 2) % 3;
  journal(x, t0, oV0, oN0, m0);
  journal(x, t1, oV1, oN1, m1);
  // the four outer edges: the opposite vertex inside the new triangle's
  // circumcircle makes the edge illegal (a candidate of the next round)
#pragma unroll 1
  for (int m = 0; m < 4; ++m) {
    if (nbr[m] < 0) continue;
    // t0 = (b, d, a), t1 = (c, a, d)
    const bool first = m < 2;
    const int tt = first ? t0 : t1, k = ((first ? k0 : k1) + 1 + (m & 1)) % 3;
    const int i0 = first ? b : c, i1 = first ? dd : a, i2 = first ? a : dd;
    const float4 P0 = first ? Pb : Pc, P1 = first ? Pd : Pa, P2 = first ? Pa : Pd;
    const int w = first ? V0.w : V1.w;
    int sqx, sqy;
    opp_shift<PER>(w, k, Wn[m].w, nbr[m] % 3, sqx, sqy);
    const bool flat = (w & BD_TRI_SHIFT_BITS) == 0 && (sqx | sqy) == 0;
    const int ic = flat ? incircle_pre(x, i0 < x.np && i1 < x.np && i2 < x.np && q[m] < x.np, P0, P1, P2, Pq[m], i0, i1,
                                       i2, q[m])
                        : incircle_s<PER>(x, first ? V0 : V1, q[m], sqx, sqy);
    if (ic > 0) register_edge(x, nb, ne, 3 * tt + k, nbr[m]);
  }
  return r;
}

// the replica of a triangle (its first disk corner; -1 if it has none)
__device__ __forceinline__ int tri_rep(const BdDev &d, int np, const int4 &v) {
  const int c = v.x < np ? v.x : (v.y < np ? v.y : (v.z < np ? v.z : -1));
  return c < 0 ? -1 : d.rep_of[c];
}

}  // namespace

// One time step's triangulation work (mode 0), the repair of the
// triangulation after new positions are set (mode 1: no overlap correction; an
// overlapping pair rejects the positions with BD_ERR_INIT_OVERLAP),
// or one piece of a halved step (mode 2: as mode 0, but the step counter does
// not advance).
//
// Phases, each ended by a grid barrier:
//   P  one pass over the triangles: orientation of triangles with a moved
//      corner (inverted => flag), the reversal test on edges with a moved end,
//      Lawson marks on edges touching a dirty triangle, and the overlap scan
//      of every disk-disk edge.  The scan is used only when the pass found no
//      inverted triangle and no illegal edge, i.e. when the triangulation it
//      scanned is the Delaunay triangulation of the current positions.
//   R  inversion repair rounds (candidate marks, owned flips) when P found an
//      inverted triangle; then P again.
//   F  owned Lawson flips of the marked edges; fused: the next round at once
//      with the candidates its flips registered, or, if a candidate lost a
//      claim, P marking without a scan; unfused: P again.
//   A  apply the capped displacements (Algorithm 2) and reflect; then P again.
// Three resident blocks per SM (at most 80 registers): the passes are
// latency-bound chains of dependent loads, and the spills this costs sit in
// the exact-predicate fallbacks (measured: 3 blocks 20 % faster than 2 on
// 2^20 disks; 4 blocks (64 registers) the same there, 337 us per step, and 1 to
// 3 % of a step slower at 16384 to 350000 disks).
//
// CL: the launch is one thread-block cluster (a small system): hardware
// barriers, the phase words in the first block's shared memory, 128 registers.
// QUEUE: the check pass of a triangulation of many triangles per thread.
template <bool PER, bool CL, bool QUEUE>
__device__ __forceinline__ void triangulation_body(const BdDev &d, const BdConst &c, int mode, int log_step) {
  Ctx x = {d, c, {c.q, c.inv_q, c.qshift}, c.nt, c.np, c.sig2f, 0u, d.ctl->cl_n};
  BdCtl *ctl = d.ctl;
  if (ld_status(&ctl->status) != 0 || (mode == 1 && *(volatile const int *)&ctl->n_set_moved == 0)) {
    // (bd_set_state that moved no disk: the triangulation stands as it was)
    if (blockIdx.x == 0 && threadIdx.x == 0 && ld_status(&ctl->status) == 0) ctl->in_move = 0;
    if (!CL) block_exit(ctl);
    return;
  }
  Bar b;
  b.gen = 0;
  b.ph = 0;
  __shared__ int bc[BC_N];                // phase counters and list lengths, per barrier
  // the phase words: in the control block, or in the cluster's first block
  __shared__ int s_words[CL ? BW_N : 1];
  int *words = nullptr, *wcnt = &ctl->cnt[0][0];
  unsigned hold = 0;
  if (CL) {
    hold = *(volatile const unsigned *)&ctl->bar_hold;
    if (threadIdx.x < BW_N) s_words[threadIdx.x] = 0;
    words = cooperative_groups::this_cluster().map_shared_rank(s_words, 0);
    wcnt = words + BW_CNT;
    x.cl_n = words + BW_CL;
    cluster_barrier();
  }
  auto sync = [&]() -> bool { return CL ? cluster_sync(ctl, words, hold, b, bc) : grid_sync(ctl, b, bc); };
  auto leave = [&]() {
    if (CL) cluster_barrier();   // the first block's words are read until the last one is here
    else block_exit(ctl);
  };
  auto pcnt = [&](int slot) -> int * { return wcnt + 8 * (b.ph & 3) + slot; };
  auto phase_start = [&]() {   // clear the counters two phases ahead
    if (blockIdx.x == 0 && threadIdx.x < 8) wcnt[8 * ((b.ph + 2) & 3) + threadIdx.x] = 0;
  };
  unsigned long long t_mark = gtimer();   // stage timing (lead thread)
  // CL: a few thousand items are spread over the blocks warp by warp, so that
  // every scheduler of the cluster's SMs has its share of them
  const int tid = CL ? (int)(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31))
                     : (int)(blockIdx.x * blockDim.x + threadIdx.x);
  const int nth = gridDim.x * blockDim.x;
  const bool lead = (blockIdx.x == 0 && threadIdx.x == 0);
  unsigned long long epoch = ctl->epoch;   // written only at kernel end by the lead thread
  x.jstamp = ((unsigned)epoch << 1) | 1u;   // distinct per launch: the epoch grows across launches
  const double sigma = c.sigma;
  int status = 0;
  int corr_iter = 0;
  long long st_overlap = 0, st_flips = 0, st_rflips = 0, st_inv = 0, st_rounds = 0;
  bool fresh = true;       // the moved flags describe the latest move
  int lawson_rounds = 0;
  // rollout log (adjoint): committed passes and their overlapping pairs
  const bool logging = log_step >= 0 && d.log_pairs != nullptr;
  int log_head = logging ? ctl->log_npairs : 0;
  int log_npass = logging ? ctl->log_npass : 0;
  int log_pidx = -1;
  // Check passes.  The first pass of a move (and the pass after an inversion
  // repair) tests every triangle; a later pass only the dirty ones: those with a
  // corner that the last correction pushed, and those stamped with the pass's
  // generation byte (flips, flip candidates left unresolved).  Every other edge
  // kept its end points and its place in the triangulation since it was last
  // checked and was not overlapping then (both ends of an overlapping edge
  // count as pushed, even when their pushes cancel and they stay), so its
  // earlier verdicts (legal, not overlapping) stand.  A clean
  // triangle costs its corner table and three flags.  (Lists of the triangles
  // to visit, kept by the flips and by walks round the moved disks, measured
  // slower at every size: 513 against 492 us per step in a batch of 350000 disks,
  // 378 against 373 at 2^20.)
  const unsigned g0 = *(volatile unsigned *)&ctl->act_gen;
  int kp = 0;
  long long tri_visits = 0;
  // the next iteration opens with a check pass (need_p) that scans the
  // overlaps (scan); the overlapping edges of the current triangulation
  // (ov_now); Lawson rounds fused with their re-tests (not while a rollout
  // logs its pairs, which wants every pair of a pass from one scan)
  bool need_p = true, scan = true;
  // the next pass tests every edge: the first pass of a launch, and a pass whose
  // overlap sums start from nothing
  bool sweep_all = true;
  int ov_now = 0;
  const bool fuse = c.tri_fuse && !logging;

  for (;;) {
    ++epoch;
    if (lead) {
      x.cl_n[(epoch + 2) % 3] = 0;   // the candidate list two rounds ahead
    }
    const unsigned gen = g0 + (unsigned)kp, ngen = gen + 1u;
    const uint8_t gen8 = (uint8_t)gen, ngen8 = (uint8_t)ngen;   // check-pass stamps of this pass and the next
    // ---------------- W: shifts of triangles whose corners re-entered (periodic box) ----------------
    if (PER && fresh && *(volatile int *)&ctl->n_wrapped != 0) {
      phase_start();
      for (int t = tid; t < x.T; t += nth) {
        const int4 v = d.tv[t];
        const uint8_t w0 = d.wrap[v.x], w1 = d.wrap[v.y], w2 = d.wrap[v.z];
        if ((w0 | w1 | w2) == 0) continue;
        journal(x, t, v, d.tn[t], d.jmark[t]);
        // a corner stored L k lower than where it geometrically is: shift += k
        const int kx[3] = {wrapx(w0), wrapx(w1), wrapx(w2)}, ky[3] = {wrapy(w0), wrapy(w1), wrapy(w2)};
        int sx[3], sy[3];
        for (int k = 0; k < 3; ++k) {
          sx[k] = tshx<PER>(v.w, k) + kx[k];
          sy[k] = tshy<PER>(v.w, k) + ky[k];
        }
        int nw = with_stamp(0, tstamp(v.w));
        for (int k = 0; k < 3; ++k) nw |= put_shift(k, sx[k] - sx[0], sy[k] - sy[0]);
        d.tv[t].w = nw;
      }
      if (!sync()) { leave(); return; }
      if (lead) ctl->n_wrapped = 0;
    }
    // ---------------- P: check, mark, scan ----------------
    // (skipped between fused Lawson rounds: their flips test the edges they
    // change; a pass that follows such rounds only marks, scan = false, since
    // the rounds keep the overlap sums of the triangulation they leave)
    int n_ov = 0;
    if (need_p) {
      phase_start();
      {
        int inv = 0, rej = 0, cand = 0, vis = 0;
        double mx = 0.0;
        const bool skip = !sweep_all && !c.tri_all;
        __shared__ int s_list[BD_DT_LIST], s_nd, s_queue[QUEUE ? BD_DT_THREADS / 32 : 1][QUEUE ? 128 : 1];
        auto clean = [&](const int4 &v) -> bool {
          if (tstamp(v.w) == gen8) return false;
          return !(fresh && (d.moved[v.x] | d.moved[v.y] | d.moved[v.z]));
        };
        // orientation of triangle t after a move of one of its corners
        auto turned = [&](int t, const int4 &v, const float4 &Wa, const float4 &Wb, const float4 &Wc) {
          const int in = !PER || (v.w & BD_TRI_SHIFT_BITS) == 0
                             ? orient_pre(x, v.x < x.np && v.y < x.np && v.z < x.np, Wa, Wb, Wc, v.x, v.y, v.z)
                             : orient_s(x, v.x, tshx<PER>(v.w, 0), tshy<PER>(v.w, 0), v.y, tshx<PER>(v.w, 1),
                                        tshy<PER>(v.w, 1), v.z, tshx<PER>(v.w, 2), tshy<PER>(v.w, 2));
          if (in <= 0) {
            // (the marks and the scan of a pass that finds one are void)
            d.tinv[t] = 1;
            ++inv;
            if (d.rep_stats) {
              const int rr = tri_rep(d, x.np, v);
              if (rr >= 0) atomicAdd((unsigned long long *)&d.rep_stats[3 * rr + 2], 1ull);
            }
          }
        };
        // One corner of a triangle per item, testing the edge that faces it (and
        // for the first corner the triangle's orientation): the chain of loads and
        // tests behind an item, which sets the length of a pass in all but the
        // largest systems, is a third of a whole triangle's.
        // The first pass takes the corners of all triangles in turn; a later pass
        // those of the block's dirty triangles, put in a list first.
        // QUEUE, for triangulations of many triangles per thread, whose passes are
        // bound by instructions, spends no lanes on the half of the corners whose
        // edge is the other side's to test: a lane takes a triangle, tests its
        // orientation and puts the corners it has to test into its warp's queue,
        // and the warp takes corners from there 32 at a time.
        const int lane = threadIdx.x & 31;
        int *const queue = s_queue[QUEUE ? threadIdx.x >> 5 : 0];
        const int share = skip ? (x.T + (int)gridDim.x - 1) / (int)gridDim.x : 0;
        const int s0 = min(x.T, (int)blockIdx.x * share), s1 = min(x.T, s0 + share);
        int base = s0;
        do {
          int items = x.T, it = tid, stride = nth;   // triangles, this thread's first item, the step to its next
          if (skip) {
            __syncthreads();   // (the list of the chunk before has been worked off)
            if (threadIdx.x == 0) s_nd = 0;
            __syncthreads();
            const int e1 = min(s1, base + BD_DT_LIST);
            for (int t = base + (int)threadIdx.x; t < e1; t += blockDim.x)
              if (!clean(d.tv[t])) s_list[atomicAdd(&s_nd, 1)] = t;
            __syncthreads();
            items = s_nd;
            it = threadIdx.x;
            stride = blockDim.x;
            base += BD_DT_LIST;
          }
          // triangles a warp puts into its queue at a time: fewer than 32 if that keeps all warps busy
          const int cw = min(32, (items + (stride >> 5) - 1) / (stride >> 5));
          int w0 = (it >> 5) * cw, queued = 0;
          for (;;) {
            int cc;
            if (!QUEUE) {
              if (it >= 3 * items) break;
              cc = skip ? 3 * s_list[it / 3] + it % 3 : it;
              it += stride;
            } else {
              while (queued < 32 && w0 < items) {
                unsigned own3 = 0u;
                int t = w0 + lane;
                if (lane < cw && t < items) {
                  if (skip) t = s_list[t];
                  const int4 v = d.tv[t], nn = d.tn[t];
                  const int on[3] = {nn.x, nn.y, nn.z};
#pragma unroll
                  for (int k = 0; k < 3; ++k)
                    if (on[k] >= 0 && (on[k] > 3 * t + k || (skip && clean(d.tv[on[k] / 3])))) own3 |= 1u << k;
                  ++vis;
                  if (fresh && ((d.moved[v.x] | d.moved[v.y] | d.moved[v.z]) & 1))
                    turned(t, v, work_of(x, v.x), work_of(x, v.y), work_of(x, v.z));
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                  const unsigned m = __ballot_sync(0xffffffffu, own3 >> k & 1u);
                  if (own3 >> k & 1u) queue[queued + __popc(m & ((1u << lane) - 1u))] = 3 * t + k;
                  queued += __popc(m);
                }
                w0 += (stride >> 5) * cw;
                __syncwarp();
              }
              if (queued == 0) break;
              const int take = min(32, queued);
              queued -= take;
              cc = lane < take ? queue[queued + lane] : -1;
              __syncwarp();   // (read before the next corners are put in)
              if (cc < 0) break;   // (the last of this warp's corners: fewer than 32, none left to fetch)
            }
            const int t = cc / 3, k = cc % 3;
            const int4 v = d.tv[t];
            const int o = ((const int *)&d.tn[t])[k];
            // corners in order: the edge faces ia and runs from ib to ic
            const int ia = vk(v, k), ib = vk(v, (k + 1) % 3), ic = vk(v, (k + 2) % 3);
            const bool own = QUEUE || (o >= 0 && (o > cc || (skip && clean(d.tv[o / 3]))));
            if (k && !own) continue;
            const float4 Wa = work_of(x, ia), Wb = work_of(x, ib), Wc = work_of(x, ic);
            uint8_t ma = 0, mb = 0, mc = 0;   // moved; periodic box: bits 1-4 its re-entry
            if (fresh) {
              ma = d.moved[ia];
              mb = d.moved[ib];
              mc = d.moved[ic];
              if (PER) {
                if (ib < x.np) mb |= (uint8_t)(d.wrap[ib] << 1);
                if (ic < x.np) mc |= (uint8_t)(d.wrap[ic] << 1);
              }
            }
            int4 v1 = make_int4(0, 0, 0, 0);
            if (own) v1 = d.tv[o / 3];
            const int q = own ? vk(v1, o % 3) : 0;
            const bool flat = !PER || (v.w & BD_TRI_SHIFT_BITS) == 0;
            const bool all_disks = ia < x.np && ib < x.np && ic < x.np;
            const bool mvd = ((ma | mb | mc) & 1) != 0;
            const bool due = own && (mvd || tstamp(v.w) == gen8 || tstamp(v1.w) == gen8 || (fresh && d.moved[q]));
            float4 Wq = make_float4(0.f, 0.f, 0.f, 0.f);
            if (due) Wq = work_of(x, q);
            if (!QUEUE && k == 0) {
              ++vis;
              if (mvd) turned(t, v, Wa, Wb, Wc);
              if (!own) continue;
            }
            const int u = ib, w = ic;
            const bool disks = u < x.np && w < x.np;
            // image shift of w relative to u in this triangle (periodic box; 0 with walls)
            const int ku = (k + 1) % 3, kw = (k + 2) % 3;
            const int rsx = tshx<PER>(v.w, kw) - tshx<PER>(v.w, ku);
            const int rsy = tshy<PER>(v.w, kw) - tshy<PER>(v.w, ku);
            const bool plain = (rsx | rsy) == 0;   // the edge carries no image shift
            long long LQ = plain ? 0 : rep_LQ(x, u);
            // r1 = r_w - r_u from the FP32 pairs, or for a shifted edge from the grid (one rounding)
            float r1x, r1y;
            if (plain) {
              r1x = fdiff(Wc.x, Wc.z, Wb.x, Wb.z);
              r1y = fdiff(Wc.y, Wc.w, Wb.y, Wb.w);
            } else {
              const Lift U = lift(x, u, 0, 0, LQ), V = lift(x, w, rsx, rsy, LQ);
              r1x = lift_diff(x, V.x, U.x);
              r1y = lift_diff(x, V.y, U.y);
            }
            if (disks && ((mb | mc) & 1)) {
              // Sec. 4.3 first criterion r0 . r1 < 0; r0 = r1 - (move of w - move
              // of u), screened in FP32 unless an end re-entered, exact on the
              // grid there and near zero (the edge's shift before the move is
              // the present one less the re-entries of its end points)
              int dec = 0;   // 1 reversed, -1 not, 0 undecided
              if (!PER || ((mb | mc) >> 1) == 0) {
                const float2 mu = (mb & 1) ? d.dmove[u] : make_float2(0.f, 0.f);
                const float2 mw = (mc & 1) ? d.dmove[w] : make_float2(0.f, 0.f);
                const float r0x = __fsub_rn(r1x, __fsub_rn(mw.x, mu.x)), r0y = __fsub_rn(r1y, __fsub_rn(mw.y, mu.y));
                // every rounding above is relative (one FP32 rounding of a grid
                // value or of a sum): the computed dot is within ~8 2^-24 S of
                // the exact one, S = |r0|^2 + |r1|^2 + |m_u|^2 + |m_w|^2
                const float dot = __fadd_rn(__fmul_rn(r0x, r1x), __fmul_rn(r0y, r1y));
                const float S = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(r0x, r0x), __fmul_rn(r0y, r0y)),
                                                    __fadd_rn(__fmul_rn(r1x, r1x), __fmul_rn(r1y, r1y))),
                                          __fadd_rn(__fadd_rn(__fmul_rn(mu.x, mu.x), __fmul_rn(mu.y, mu.y)),
                                                    __fadd_rn(__fmul_rn(mw.x, mw.x), __fmul_rn(mw.y, mw.y))));
                const float bound = 4e-6f * S;
                dec = dot > bound ? -1 : (-dot > bound ? 1 : 0);
                if (dec == 0 && plain) count_exact(x);
              }
              if (dec == 0) {
                int ox = rsx, oy = rsy;
                if (PER) {
                  ox -= wrapx((uint8_t)(mc >> 1)) - wrapx((uint8_t)(mb >> 1));
                  oy -= wrapy((uint8_t)(mc >> 1)) - wrapy((uint8_t)(mb >> 1));
                  if ((ox | oy) && LQ == 0) LQ = rep_LQ(x, u);
                }
                dec = reversed_grid(kp == 0 ? d.pos0 : d.prev, d.pos, x.g, u, w, mb & 1, mc & 1, ox, oy, rsx, rsy, LQ) ? 1 : -1;
              }
              if (dec == 1) {
                ++rej;
                atomicExch(&ctl->st_fail_item, cc);
              }
            }
            // the edge's in-circle test is due when a triangle on either side is
            // dirty or one of its four points moved
            if (due) {
              int sqx, sqy;
              opp_shift<PER>(v.w, k, v1.w, o % 3, sqx, sqy);
              const int in = (flat && (sqx | sqy) == 0)
                                 ? incircle_pre(x, all_disks && q < x.np, Wa, Wb, Wc, Wq, ia, ib, ic, q)
                                 : incircle_s<PER>(x, v, q, sqx, sqy);
              if (in > 0) {
                ++cand;
                register_edge(x, claims(x, epoch), epoch, min(cc, o), max(cc, o));   // by its smaller corner
              }
            }
            // FP32 screen: a pair whose FP32 squared distance exceeds
            // sigma^2 (1 + 1e-5) is farther than sigma (FP32 error ~3e-7)
            if (disks && scan && !(__fadd_rn(__fmul_rn(r1x, r1x), __fmul_rn(r1y, r1y)) > x.sig2f)) {
              const double del = overlap_push(d, c, u, w, rsx, rsy, LQ, 1);
              if (del > 0.0) {
                const int k_ov = atomicAdd(pcnt(C_OVERLAP), 1);
                if (logging) {
                  if (log_head + k_ov < c.log_pairs_cap) d.log_pairs[log_head + k_ov] = make_int2(u, w);
                  else atomicExch(&ctl->log_overflow, 1);
                }
                mx = fmax(mx, del);
              }
            }
          }
        } while (skip && base < s1);
        {
          int *const to[4] = {pcnt(C_INV), pcnt(C_REJECT), pcnt(C_CAND), pcnt(C_VISIT)};
          const int n[4] = {inv, rej, cand, vis};
          block_add(to, n);
        }
        if (mx > 0.0) atomicMax(&ctl->st_max_overlap_bits, (unsigned long long)__double_as_longlong(mx));
      }
      if (!sync()) { leave(); return; }
      if (lead) {
        stage_tick(ctl, sweep_all || c.tri_all ? STAGE_P : STAGE_PL, t_mark);
        tri_visits += bc[BC_CNT + C_VISIT];
      }
      const int n_inv = bc[BC_CNT + C_INV];
      const int n_rej = bc[BC_CNT + C_REJECT];
      n_ov = bc[BC_CNT + C_OVERLAP];
      if (n_rej) {
        status = BD_ERR_STEP_REJECTED;
        if (lead) { ctl->st_fail_phase = 1; ctl->st_fail_count = n_rej; }
        break;
      }

      if (n_inv > 0) {
        // ---------------- R: inversion repair (this pass's marks and scan are void) ----------------
        st_inv += n_inv;
        int rounds = 0;
        bool first_round = true;
        for (;;) {
          ++epoch;
          if (lead) x.cl_n[(epoch + 2) % 3] = 0;   // the candidate list two rounds ahead
          phase_start();
          {
            if (first_round) {
              for (int i = tid; i < x.np; i += nth) d.disp[i] = make_double2(0.0, 0.0);
              // the check pass skipped the marks (and the pass after the repair
              // is not fresh): a triangle with a moved corner stays dirty for it
              for (int t = tid; t < x.T; t += nth) {
                const int4 v = d.tv[t];
                if (d.moved[v.x] | d.moved[v.y] | d.moved[v.z]) d.tv[t].w = with_stamp(v.w, ngen8);
              }
            }
            int inv = 0, ncand = 0;
            for (int t = tid; t < x.T; t += nth) {
              if (!d.tinv[t]) continue;
              const int4 v = d.tv[t];
              ++inv;
              atomicExch(&ctl->st_fail_item, t);
              const int4 nn = d.tn[t];
              for (int k = 0; k < 3; ++k) {
                const int o = vk(nn, k);
                if (o < 0) continue;
                const int p = vk(v, k), u = vk(v, (k + 1) % 3), w = vk(v, (k + 2) % 3);
                const int4 v1 = d.tv[o / 3];
                const int q = vk(v1, o % 3);
                int sqx, sqy;
                opp_shift<PER>(v.w, k, v1.w, o % 3, sqx, sqy);
                const int spx = tshx<PER>(v.w, k), spy = tshy<PER>(v.w, k);
                const int sux = tshx<PER>(v.w, (k + 1) % 3), suy = tshy<PER>(v.w, (k + 1) % 3);
                const int swx = tshx<PER>(v.w, (k + 2) % 3), swy = tshy<PER>(v.w, (k + 2) % 3);
                // orientation form of Eq. (predicate): both triangles of the
                // other diagonal strictly counter-clockwise
                if (orient_s(x, u, sux, suy, q, sqx, sqy, p, spx, spy) > 0 &&
                    orient_s(x, w, swx, swy, p, spx, spy, q, sqx, sqy) > 0) {
                  const int cm = min(3 * t + k, o);
                  const int tt = cm / 3, kk = cm % 3;
                  const int4 ncm = d.tn[tt];
                  claim6(d.tn, claims(x, epoch), tt, kk, ncm, vk(ncm, kk), claim_key(epoch, cm));
                  ++ncand;
                }
              }
            }
            block_add(pcnt(C_INV), inv);
            block_add(pcnt(C_CAND), ncand);
          }
          if (!sync()) { leave(); return; }
          if (lead) stage_tick(ctl, STAGE_R, t_mark);
          first_round = false;
          const int ni = bc[BC_CNT + C_INV];
          const int nc = bc[BC_CNT + C_CAND];
          if (ni == 0) break;
          if (nc == 0 || rounds++ >= c.max_flip_rounds) {
            status = BD_ERR_STEP_REJECTED;
            if (lead) { ctl->st_fail_phase = nc == 0 ? 2 : 3; ctl->st_fail_count = ni; }
            break;
          }
          phase_start();
          {
            int nf = 0;
            for (int t = tid; t < x.T; t += nth) {
              const unsigned long long key = claims(x, epoch)[t];
              if ((key >> 32) != epoch) continue;
              const int cm = key_corner(key);
              if (cm / 3 != t) continue;
              const int4 N0 = d.tn[t];
              const int o = vk(N0, cm % 3);
              if (!owns6(x, claims(x, epoch), t, cm % 3, N0, o, key)) continue;
              flip_owned<PER>(x, cm, o, ngen8);   // both new triangles are counter-clockwise by the rule
              ++nf;
            }
            block_add(pcnt(C_FLIPS), nf);
          }
          if (!sync()) { leave(); return; }
          if (lead) stage_tick(ctl, STAGE_R, t_mark);
          st_rflips += bc[BC_CNT + C_FLIPS];
        }
        if (status) break;
        fresh = false;
        sweep_all = true;   // the repaired region's marks and scan were skipped: check everything
        need_p = scan = true;
        ++kp;
        continue;
      }
      if (scan) ov_now = n_ov;
    }

    // candidates for this round: the marking pass's and those the previous
    // fused round registered
    if (bc[BC_CL + (int)(epoch % 3)] > 0) {
      // ---------------- F: owned Lawson flips ----------------
      if (lawson_rounds++ >= c.max_flip_rounds) {
        status = BD_ERR_FLIP_NOT_CONVERGED;
        if (lead) ctl->st_fail_phase = 4;
        break;
      }
      phase_start();
      {
        const bool voided = !fuse && n_ov;   // unfused: the marking pass's scan is void
        if (voided)
          for (int i = tid; i < x.np; i += nth) d.disp[i] = make_double2(0.0, 0.0);
        if (fresh)
          for (int i = tid; i < x.np / 4; i += nth) ((unsigned *)d.moved)[i] = 0u;   // np is a multiple of 512
        int nf = 0, nlose = 0, adj = 0;
        double fmx = 0.0;
        // the triangles that registered a candidate for this round (in the
        // marking pass, or in the previous fused round): each candidate is
        // owned by the triangle that tested it.  An owner whose flip lost a
        // claim is stamped, so its edges are tested again by a check pass.
        // Unfused, a flip stamps its two triangles for the next pass, and
        // every other edge the marking pass tested keeps its verdict unless a
        // flip changes it.  Fused, a flip tests the four outer edges of its
        // quadrilateral itself -- the six triangles it owns do not change
        // during the round -- and registers the illegal ones for the next
        // round (claims of the other parity, the next candidate list); it
        // also withdraws the overlap of the diagonal it removes and adds that
        // of the one it draws (exact fixed-point sums), so the sums stay those
        // of the current triangulation.
        const int cs = (int)(epoch % 3);
        const int ncl = bc[BC_CL + cs];
        const int *cl = d.clist + (size_t)cs * x.T;
        unsigned long long *cb = claims(x, epoch), *nb = claims(x, epoch + 1);
        // consecutive entries go to different blocks (a few hundred flips on
        // one SM would queue on its load/store unit)
        for (int it = blockIdx.x + threadIdx.x * gridDim.x; it < ncl; it += nth) {
          const int t = cl[it];
          int t1 = -1;   // the triangle t was flipped with
          if (fuse) {
            const FusedOut fo = fused_flip<PER>(x, t, epoch, cb, nb);
            t1 = fo.t1;
            adj += fo.adj;
            fmx = fmax(fmx, fo.mx);
          } else {
            const unsigned long long key = cb[t];
            const int cm = key_corner(key);
            if ((key >> 32) == epoch && cm / 3 == t) {
              const int4 N0 = d.tn[t];
              const int o = vk(N0, cm % 3);
              if (owns6(x, cb, t, cm % 3, N0, o, key)) {
                t1 = o / 3;
                flip_owned<PER>(x, cm, o, ngen8);
              }
            }
          }
          if (t1 >= 0) {
            ++nf;
            if (d.rep_stats) {
              // the four points of a flipped edge include a disk (ghost
              // points never move, so an edge among them stays legal); one
              // of the two new triangles may hold only ghost points
              int rr = tri_rep(d, x.np, d.tv[t]);
              if (rr < 0) rr = tri_rep(d, x.np, d.tv[t1]);
              if (rr >= 0) atomicAdd((unsigned long long *)&d.rep_stats[3 * rr + 1], 1ull);
            }
          } else {
            ++nlose;
            stamp_tri(x, t, ngen8);
          }
        }
        {
          int *const to[3] = {pcnt(C_FLIPS), pcnt(C_LOSE), pcnt(C_OVADJ)};
          const int v[3] = {nf, fuse ? nlose : 0, adj};
          block_add(to, v);
        }
        if (fuse) {
          if (fmx > 0.0) atomicMax(&ctl->st_max_overlap_bits, (unsigned long long)__double_as_longlong(fmx));
        }
      }
      if (!sync()) { leave(); return; }
      if (lead) stage_tick(ctl, STAGE_F, t_mark);
      st_flips += bc[BC_CNT + C_FLIPS];
      st_rounds += 1;
      fresh = false;
      if (!fuse) {
        need_p = scan = sweep_all = true;   // the next pass marks and scans afresh
        ++kp;
        continue;
      }
      ov_now += bc[BC_CNT + C_OVADJ];
      if (bc[BC_CNT + C_LOSE] > 0) {
        need_p = true;          // a pass marks the losers' edges again
        scan = sweep_all = false;
        ++kp;
        continue;
      }
      if (bc[BC_CL + (int)((epoch + 1) % 3)] > 0) {
        need_p = false;         // the next round flips what this one registered
        ++kp;
        continue;
      }
      // no candidate left: the triangulation is Delaunay
    }

    // Delaunay triangulation of the current positions: the overlap sums (the
    // last scan's, kept by the fused rounds) are Algorithm 2's
    if (mode == 1) {
      // new positions set from outside: they must not overlap (the scan of
      // this Delaunay triangulation finds the closest pair)
      if (ov_now) {
        status = BD_ERR_INIT_OVERLAP;
        if (lead) { ctl->st_fail_phase = 7; ctl->st_fail_count = ov_now; }
      }
      break;
    }
    if (ov_now == 0) break;
    if (corr_iter >= c.max_corr_iters) {
      status = BD_ERR_OVERLAP_NOT_CONVERGED;
      if (lead) ctl->st_fail_phase = 5;
      break;
    }
    ++corr_iter;
    st_overlap += ov_now;
    lawson_rounds = 0;
    if (logging) {
      // commit this pass to the rollout log
      log_pidx = log_npass < c.log_pass_cap ? log_npass : -1;
      if (lead) {
        if (log_pidx >= 0) {
          d.log_pass_begin[log_pidx] = log_head;
          d.log_pass_begin[log_pidx + 1] = log_head + n_ov;
        } else {
          atomicExch(&ctl->log_overflow, 1);
        }
      }
      log_head += n_ov;
      ++log_npass;
    }
    // ---------------- A: apply (capped at sigma/4) ----------------
    phase_start();
    {
      // Only the marked disks have a sum: the others cost their mark and their
      // cleared flag, 2 bytes a disk (with every disk's position, sum and
      // previous position, some 50 bytes, the pass took 59 us at 2^20 disks for a
      // few thousand that move).  Four marks are loaded ahead of their use; a
      // marked disk has a thread to itself, since its chain of loads sets the
      // length of the pass (four neighbouring disks per thread doubled it).
      int nwrap = 0;
      for (int i0 = tid; i0 < x.np; i0 += 4 * nth) {
        unsigned marks = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + u * nth < x.np && d.hit[i0 + u * nth]) marks |= 1u << u;
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * nth;
          if (i >= x.np) break;
          if (!(marks >> u & 1u)) {
            d.moved[i] = 0;
            if (PER) d.wrap[i] = 0;
            if (log_pidx >= 0) d.log_pflags[(size_t)log_pidx * x.np + i] = 0;
            continue;
          }
          d.hit[i] = 0;
          if (PER) d.wrap[i] = 0;
          const double2 p = d.pos[i];
          const double2 dd = disp_get(x, i);
          d.prev[i] = p;
          if (dd.x == 0.0 && dd.y == 0.0) {
            // Its pushes cancel: it stays where it is, overlapping.  Flagged as
            // moved, its edges are looked at again by the next pass, which
            // would otherwise pass over an edge both of whose ends stay.
            d.dmove[i] = make_float2(0.f, 0.f);
            d.moved[i] = 1;
            if (log_pidx >= 0) d.log_pflags[(size_t)log_pidx * x.np + i] = 0;
            continue;
          }
          if (d.rep_stats) {
            // the first disk of a replica moved by this pass counts the pass
            const int rr = d.rep_of[i];
            const unsigned long long stamp = epoch;   // distinct per pass (grows across launches), never 0
            if (atomicExch(&d.rep_mark[rr], stamp) != stamp)
              atomicAdd((unsigned long long *)&d.rep_stats[3 * rr], 1ull);
          }
          const double mag = sqrt(__dadd_rn(__dmul_rn(dd.x, dd.x), __dmul_rn(dd.y, dd.y)));
          // Sec. 4.4: sigma/4, half the disk's radius (its own for polydisperse disks)
          const double cap = d.rad ? 0.5 * d.rad[i] : 0.25 * sigma;
          const bool capped = mag > cap;
          const double sc = capped ? cap / mag : 1.0;
          const double2 y = make_double2(snap(__dadd_rn(p.x, __dmul_rn(dd.x, sc)), x.g),
                                         snap(__dadd_rn(p.y, __dmul_rn(dd.y, sc)), x.g));
          int rfl = 0;
          const BdRep &R = d.rep[d.rep_of[i]];
          double2 np2;
          if (PER && R.periodic) {
            // Algorithm 2 "applying the periodic boundary conditions": re-entry
            long long X = bdpred::to_int(y.x, x.g), Y = bdpred::to_int(y.y, x.g);
            d.dmove[i] = make_float2(bdem::grid_to_float(X - bdpred::to_int(p.x, x.g), x.g.s),
                                     bdem::grid_to_float(Y - bdpred::to_int(p.y, x.g), x.g.s));
            const int wr = bdem::wrap_grid(R.LQ, X, Y);
            d.wrap[i] = (uint8_t)wr;
            if (wr) ++nwrap;
            np2 = make_double2(bdem::grid_to_double(X, x.g.s), bdem::grid_to_double(Y, x.g.s));
          } else {
            np2 = bdem::reflect_w(bdem::walls_of(d, R, i), y, &rfl);
          }
          if (log_pidx >= 0) d.log_pflags[(size_t)log_pidx * x.np + i] = (uint8_t)(rfl | (capped ? 16 : 0));
          d.pos[i] = np2;
          d.work[i] = split_pos(np2);
          if (!(PER && R.periodic)) {
            d.dmove[i] = make_float2(bdem::grid_to_float(bdpred::to_int(np2.x, x.g) - bdpred::to_int(p.x, x.g), x.g.s),
                                     bdem::grid_to_float(bdpred::to_int(np2.y, x.g) - bdpred::to_int(p.y, x.g), x.g.s));
          }
          d.disp[i] = make_double2(0.0, 0.0);
          d.moved[i] = 1;
        }
      }
      if (PER) block_add(&ctl->n_wrapped, nwrap);
    }
    if (!sync()) { leave(); return; }
    if (lead) stage_tick(ctl, STAGE_A, t_mark);
    fresh = true;
    need_p = scan = true;
    sweep_all = false;   // an edge neither of whose ends had a push did not overlap and still does not
    ++kp;
  }

  if (status) {
    // undo the step: positions and directions from the step start, the
    // triangulation from the undo journal
    phase_start();
    for (int i = tid; i < x.np; i += nth) {
      if (d.ext_id[i] < 0) continue;
      const double2 p0 = d.pos0[i];
      d.pos[i] = p0;
      d.prev[i] = p0;
      d.work[i] = split_pos(p0);
      d.theta[i] = d.theta0[i];
      d.disp[i] = make_double2(0.0, 0.0);
      d.moved[i] = 0;
    }
    // the journaled triangles as they were
    for (int t = tid; t < x.T; t += nth) {
      d.tinv[t] = 0;
      if (d.jmark[t] == x.jstamp) unjournal(d, t);
    }
    if (lead) atomicCAS(&ctl->status, 0, status);
  } else {
    for (int i = tid; i < x.np / 4; i += nth) ((unsigned *)d.moved)[i] = 0u;
  }
  if (lead) {
    if (logging && !status) {
      ctl->log_npairs = log_head;
      ctl->log_npass = log_npass;
      d.log_step_pass[log_step + 1] = log_npass;
    }
    ctl->epoch = epoch + 1;
    ctl->in_move = 0;
    ctl->act_gen = g0 + (unsigned)kp + 3u;
    ctl->st_tri_visits += tri_visits;
    ctl->st_corr_iters += corr_iter;
    ctl->st_overlap_pairs += st_overlap;
    ctl->st_flips += st_flips;
    ctl->st_repair_flips += st_rflips;
    ctl->st_inverted += st_inv;
    ctl->st_flip_rounds += st_rounds;
    ctl->st_barriers += b.gen;
    if (corr_iter > ctl->st_max_corr_iters) ctl->st_max_corr_iters = corr_iter;
    if (!status && mode == 2) ctl->st_substeps += 1;
    else if (!status) ctl->st_steps += 1;
    if (!status && mode == 0) ctl->step_dev += 1;
  }
  leave();
}

template <bool PER, bool QUEUE>
__global__ void __launch_bounds__(BD_DT_THREADS, 3)
    k_triangulation(const __grid_constant__ BdDev d, const __grid_constant__ BdConst c, int mode, int log_step) {
  triangulation_body<PER, false, QUEUE>(d, c, mode, log_step);
}
template <bool PER>
__global__ void __launch_bounds__(BD_DTC_THREADS, 1)
    k_triangulation_cl(const __grid_constant__ BdDev d, const __grid_constant__ BdConst c, int mode, int log_step) {
  triangulation_body<PER, true, false>(d, c, mode, log_step);
}

// Undo a step whose persistent kernel left at a timed-out barrier, or did not
// start because the Verlet lists overflowed (the kernel's own failure path did
// not run).  The launch journaled every
// triangle before its first change to it, and all its blocks have finished
// (this kernel runs after it in stream order), so replaying the journal
// restores the triangulation; positions and directions come from pos0 /
// theta0 (the step start, or the positions before bd_set_state).
// bd_launch_restore_step runs it (the header above the launcher declares it).
__global__ void k_restore_step(BdDev d, BdConst c) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nth = gridDim.x * blockDim.x;
  // a rebuild of the Verlet lists was cut off or ran out of room (the force that
  // follows it takes the request back): references parked far away make the
  // next use of the lists rebuild them
  if (c.any_short && *(volatile const int *)&d.ctl->vl_need)
    for (int i = tid; i < c.np; i += nth) d.vl_ref[i] = make_double2(1e30, 1e30);
  if (!*(volatile const int *)&d.ctl->in_move) return;   // nothing had moved yet
  for (int i = tid; i < c.np; i += nth) {
    if (d.ext_id[i] < 0) continue;
    const double2 p0 = d.pos0[i];
    d.pos[i] = p0;
    d.prev[i] = p0;
    d.work[i] = split_pos(p0);
    d.theta[i] = d.theta0[i];
    d.disp[i] = make_double2(0.0, 0.0);
    d.moved[i] = 0;
  }
  if (!c.overlap_verlet) {
    // the journaled triangles as they were; their marks cleared (the abandoned
    // launch did not publish its epoch, so the next launch takes the same stamp)
    const unsigned jstamp = ((unsigned)d.ctl->epoch << 1) | 1u;
    for (int t = tid; t < c.nt; t += nth) {
      d.tinv[t] = 0;
      if (d.jmark[t] == jstamp) {
        unjournal(d, t);
        d.jmark[t] = 0u;
      }
      // the abandoned launch did not publish the claim epochs it used (the next
      // launch starts from the same ones): clear its claims and owner marks (0
      // matches no epoch)
      d.claim[t] = d.claim[(size_t)c.nt + t] = 0ull;
      d.clmark[t] = 0u;
    }
  }
}

cudaError_t bd_launch_restore_step(const BdDev &d, const BdConst &c, cudaStream_t s) {
  const int work = c.np > c.nt ? c.np : c.nt;
  int blocks = (work + 255) / 256;
  if (blocks < 1) blocks = 1;
  if (blocks > 4096) blocks = 4096;
  k_restore_step<<<blocks, 256, 0, s>>>(d, c);
  return cudaGetLastError();
}

int bd_dt_grid_for(long long work_items, int *grid, int *block) {
  // all co-resident blocks (the phases are latency-bound chains of dependent
  // loads and integer predicates, so more threads in flight help), but no
  // more than about one work item per thread
  int g = 0, b = 0;
  if (bd_dt_grid(&g, &b) != 0) return -1;
  long long want = (work_items + b - 1) / b;
  if (want < 1) want = 1;
  *grid = want < g ? (int)want : g;
  *block = b;
  return 0;
}

int bd_dt_grid(int *grid, int *block) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  const void *fns[4] = {(const void *)k_triangulation<false, false>, (const void *)k_triangulation<true, false>,
                        (const void *)k_triangulation<false, true>, (const void *)k_triangulation<true, true>};
  for (int i = 0; i < 4; ++i) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fns[i], BD_DT_THREADS, 0) != cudaSuccess) return -1;
    per = i == 0 || n < per ? n : per;
  }
  if (per < 1) return -1;
  *grid = sms * per;
  *block = BD_DT_THREADS;
  return 0;
}

// One cluster serves triangulations of up to BD_DTC_TRIS triangles: its barriers
// cost a fraction of the grid's, its threads (8192 in sixteen blocks) are fewer.
// Cluster against grid, us per step: 139 -> 117 with walls at 777 disks coupled
// to a fluid (1985 triangles), 75 -> 67 at 1024 disks (2.6e3), but 172 -> 180 in
// a rollout of 4096 disks with its gradient (8.6e3).
#define BD_DTC_TRIS 4096
int bd_dt_cluster_for(int nt) {
  const char *env = getenv("BD_TRI_CLUSTER");   // 0: never, n: up to n triangles
  const int most = env ? atoi(env) : BD_DTC_TRIS;
  if (nt > most) return 0;
  for (int n = 16; n >= 8; n /= 2) {
    int ok = 1;
    for (int per = 0; per < 2 && ok; ++per) {
      const void *fn = per ? (const void *)k_triangulation_cl<true> : (const void *)k_triangulation_cl<false>;
      if (n > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ok = 0;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(n);
      cfg.blockDim = dim3(BD_DTC_THREADS);
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = n;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int can = 0;
      if (!ok || cudaOccupancyMaxActiveClusters(&can, fn, &cfg) != cudaSuccess || can < 1) ok = 0;
    }
    if (ok) return n;
    cudaGetLastError();
  }
  return 0;
}

// Check passes through the warps' queues from more than BD_DT_QUEUE triangles per
// thread on: first check pass of 2^20 disks (18 per thread) 121 -> 84 us, of 64
// boxes of 350000 disks in all (6) 46 -> 39 us with as much lost in the passes after
// it, of 16384 disks (a third) 10.0 -> 10.3 us.
#define BD_DT_QUEUE 8
int bd_dt_queue_for(int nt, int grid, int block) {
  const char *env = getenv("BD_TRI_QUEUE");   // triangles per thread
  return nt > (long long)(env ? atoi(env) : BD_DT_QUEUE) * grid * block;
}

cudaError_t bd_launch_dt(const BdDev &d, const BdConst &c, int mode, cudaStream_t s, int grid,
                         int block, int log_step) {
  // the barrier words and phase counters were reset by the previous
  // launch's last block (and zeroed at allocation)
  BdDev dd = d;
  BdConst cc = c;
  int m = mode, ls = log_step;
  void *args[] = {&dd, &cc, &m, &ls};
  if (c.tri_cluster) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c.tri_cluster);
    cfg.blockDim = dim3(BD_DTC_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c.tri_cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(
        &cfg, c.any_periodic ? (const void *)k_triangulation_cl<true> : (const void *)k_triangulation_cl<false>, args);
  }
  const void *fn = c.any_periodic
                       ? c.tri_queue ? (const void *)k_triangulation<true, true> : (const void *)k_triangulation<true, false>
                       : c.tri_queue ? (const void *)k_triangulation<false, true> : (const void *)k_triangulation<false, false>;
  return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(block), args, 0, s);
}
