// Symmetric all-pairs sweep: the long-range force of Sec. 2.2,
//   F_i = sum_{j != i} A[s_i][s_j] (r_i - r_j) / |r_i - r_j|^3,
// with the geometric factor g_ij = (r_i - r_j)/|r_ij|^3 = -g_ji evaluated
// once per unordered pair and added to both disks (A[s_i][s_j] g_ij to i,
// -A[s_j][s_i] g_ij to j; the table need not be symmetric).
//
// Disks sit in blocks of BD_SB = 512 consecutive slots (two j tiles), each of
// one species.  A work item pairs block P with a range of groups of 32 disks j:
//  - groups of P itself: the i side only, all ordered pairs inside P;
//  - groups of later blocks: every pair once, both sides.
// Pairs with an earlier group are done by that group's block.  Items are cut in
// groups, not in whole tiles of 256, so that a small system still has several
// items for every resident block.
//
// Inside an item each warp holds a share of the disks i of P in registers
// (four or eight per lane, as packed f32x2 pairs).  A tile of 256 disks j is staged
// in shared memory; a warp takes 32 of them, one per lane, and passes them
// round its lanes by shuffles, each j carrying its own accumulator, so after
// 32 steps every j has met all of the warp's i and returned to its lane.  Per
// unordered pair: 2 sub, 2 FMA (r^2), 1 MUFU rsqrt, 2 mul (r^-3), 2 FMA into
// the i accumulators and 2 FMA into the j accumulator -- 10 FP32 lane
// operations for two ordered pair interactions, against 8 per ordered pair in
// the one-sided sweep.
//
// Partial forces are written, not added: the i side of each item to ipart,
// the j side of each (item, group) to jpart.  k_force_sym_reduce then sums, for
// every disk, its block's i partials and its group's j partials in a fixed
// order, so the force is deterministic.  Coordinates are re-centred on the
// block's integer origin from the (hi, lo) FP32 pair of each FP64 coordinate,
// as in the one-sided sweep; per-tile FP32 sums are added in (hi, lo) pairs
// within an item on the i side, and partials (FP32) in float-float by the
// reduction.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "bd_internal.h"
#include "em.cuh"
#include "f32x2.cuh"

using namespace bdf;

// below this many slots the reduction takes fifteen shares per disk, not four:
// about the slots whose four shares fill the SMs' threads.  Fifteen whether the
// move is in it (with the warp that draws, four blocks of 512 threads fill an SM)
// or not: the shares set the order of the sum, and a step's force is the same
// bits in a graph, in launches of its own, timed, and in a rollout's replay.
#define BD_RED_SMALL 65536
#define BD_RED_SHARES 15
static_assert(BD_MOVE_FUSED < BD_RED_SMALL, "a fused move and the force apart take the same shares");

namespace {

__device__ __forceinline__ float2 recentre(float4 w, float2 org) {
  return make_float2(__fadd_rn(__fsub_rn(w.x, org.x), w.z), __fadd_rn(__fsub_rn(w.y, org.y), w.w));
}

// periodic box: disk j about the integer block origin o as its minimum
// image, from its stored (x_hi, y_hi, x_lo, y_lo) (tiles are copied to
// shared memory as they are): per coordinate the rounded difference
// s = x_hi - o and its error e (TwoSum), s wrapped by L when beyond L/2
// (exact: L/2 < |s| <= L), then (s, e + x_lo) renormalised (Fast2Sum), so
// that the hi part is the rounded minimum image up to the rounding of the lo
// part; L = 0 (walls): no wrap.  The i side takes the same form, which keeps
// the self pair's difference exactly 0.
__device__ __forceinline__ void rel_raw1(float h, float l, float o, float Lf, float hLf, float &hi, float &lo) {
  const float s = __fsub_rn(h, o);
  const float bb = __fsub_rn(s, h);
  const float e = __fsub_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fadd_rn(o, bb));
  const float w = s > hLf ? __fsub_rn(s, Lf) : (s < -hLf ? __fadd_rn(s, Lf) : s);
  const float t = __fadd_rn(e, l);
  hi = __fadd_rn(w, t);
  lo = __fsub_rn(t, __fsub_rn(hi, w));
}
__device__ __forceinline__ float4 rel_raw(float4 w, float2 org, float Lf, float hLf) {
  if (w.x > 1.0e17f) return make_float4(1.0e18f, 1.0e18f, 0.f, 0.f);   // inert slot
  float4 r;
  rel_raw1(w.x, w.z, org.x, Lf, hLf, r.x, r.z);
  rel_raw1(w.y, w.w, org.y, Lf, hLf, r.y, r.w);
  return r;
}

// bounding box (x_min, x_max, y_min, y_max), inert slots (1e18) left out
__device__ __forceinline__ void sbox_add(float4 &bx, float x, float y) {
  if (x > 1.0e17f) return;
  bx.x = fminf(bx.x, x);
  bx.y = fmaxf(bx.y, x);
  bx.z = fminf(bx.z, y);
  bx.w = fmaxf(bx.w, y);
}
__device__ __forceinline__ float4 swarp_box(float4 bx) {
  for (int o = 16; o > 0; o >>= 1) {
    bx.x = fminf(bx.x, __shfl_xor_sync(0xffffffffu, bx.x, o));
    bx.y = fmaxf(bx.y, __shfl_xor_sync(0xffffffffu, bx.y, o));
    bx.z = fminf(bx.z, __shfl_xor_sync(0xffffffffu, bx.z, o));
    bx.w = fmaxf(bx.w, __shfl_xor_sync(0xffffffffu, bx.w, o));
  }
  return bx;
}
__device__ __forceinline__ float4 sempty_box() { return make_float4(3e38f, -3e38f, 3e38f, -3e38f); }

// minimum image of a packed pair of coordinate differences in (-3L/2, 3L/2):
// t = rint(dx / L) by the 1.5 2^23 rounding constant, dx - t L exact (Sterbenz)
__device__ __forceinline__ u64 min_image2(u64 dx, u64 invL2, u64 nL2, u64 M2) {
  const u64 t = sub2(fma2(dx, invL2, M2), M2);
  return fma2(t, nL2, dx);
}
// the same by compares, which leaves the far-away inert slots far away
__device__ __forceinline__ u64 min_image2_cmp(u64 dx, float Lf, float hLf) {
  float a, b;
  up2(dx, a, b);
  a = a > hLf ? __fsub_rn(a, Lf) : (a < -hLf ? __fadd_rn(a, Lf) : a);
  b = b > hLf ? __fsub_rn(b, Lf) : (b < -hLf ? __fadd_rn(b, Lf) : b);
  return pk2(a, b);
}

// lo parts of the disks i, kept in the thread's local memory (read only by
// the rare near tiles, so they hold no registers across the sweep)
__device__ __forceinline__ void st_local4(float4 *p, float4 v) {
  asm volatile("st.local.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_local(p)), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ float4 ld_local4(const float4 *p) {
  float4 v;
  asm volatile("ld.local.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(__cvta_generic_to_local(p)));
  return v;
}

}  // namespace

// NW warps per block, NP packed i pairs (2 NP disks) per lane, one disk j
// carried per lane; NW * 32 * 2 * NP = BD_SB.  Shapes built: (4 warps, 4 disks per
// lane) and (2 warps, 8 disks per lane); the second halves the ring's shuffles
// and register moves per pair.  (Two j per lane, the packed halves of a j
// accumulator folded before it is passed, and deeper unrolling measured within
// 3 % of these.)  A tile of j is copied raw with cp.async (no registers held
// across the tile's arithmetic) and each j re-centred as it is read (walls),
// or, PER, the tile is re-centred in place once it has landed.  The i side's sum
// over an item's tiles is float-float.
//
// PER (periodic boxes, Sec. 2.1): every coordinate is re-centred on the block
// origin as its minimum image, as an FP32 (hi, lo) pair (rel_raw); each warp
// holds a contiguous quarter (half) of the block's disks i.  Per (warp, group
// of 32 disks j) the warp's box of its disks i and the group's box (taken
// about one of its disks, so a group across the antipode is not mistaken for
// one spanning the box) tell which pair form every pair of the two may take
// (pair_mode): hi parts alone; per-pair minimum image on one axis or both;
// the exact vector for boxes closer than 20.
template <int NW, int NP, bool PER>
__device__ __forceinline__ void force_long_sym_body(const BdDev &d, const BdConst &c) {
  if (ctl_failed(d.ctl)) return;
  constexpr int T = NW * 32;         // threads
  constexpr int NQ = 2 * NP;         // disks i per thread
  constexpr int NS = BD_TJ / T;      // j disks each thread stages per tile
  constexpr int NG = BD_TJ / BD_SG;  // groups of 32 disks j per tile
  static_assert(BD_SB == T * NQ, "a block is BD_SB disks");
  __shared__ __align__(16) float4 sraw[2][BD_TJ];   // j as stored (x_hi, y_hi, x_lo, y_lo);
                                                    // PER: re-centred in place (hi, lo)
  __shared__ float2 shw[NW][BD_TJ];  // per-warp j-side sums of the current tile
  __shared__ float4 sgbox[2][PER ? NG : 1];   // PER: per-group boxes of the staged tile
  __shared__ int sgpad[2][PER ? NG : 1];      //      and whether the group holds inert slots
  __shared__ float4 sibox[PER ? NW : 1];      //      per-warp boxes of the block's disks i
  __shared__ int sipad[PER ? NW : 1];         //      and whether they include inert slots
  const int item_id = c.sitem0 + (int)blockIdx.x;   // this launch's share of the plan (force sharding)
  const int4 item = d.sitems[item_id];
  const int P = item.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int base = P * BD_SB;
  const int gsym = (P + 1) * (BD_SB / BD_SG);   // first group met from both sides
  const int2 binfo = d.sblock[P];
  const BdRep &R = d.rep[binfo.x];
  const int a = binfo.y;
  const float2 org = d.sorigin[P];
  bool per = false;                  // this block's replica is periodic
  float Lf = 0.f, hLf = __int_as_float(0x7f800000);
  if (PER && R.periodic) {
    per = true;
    Lf = R.Lf;
    hLf = R.hLf;
  }
  auto rel = [&](int j) -> float4 {
    if (PER) return rel_raw(d.work[j], org, Lf, hLf);
    const float2 v = recentre(d.work[j], org);
    return make_float4(v.x, v.y, 0.f, 0.f);
  };
  // slot (in the block) of this thread's disk i number q
  auto islot = [&](int q) -> int { return PER ? warp * (BD_SB / NW) + q * 32 + lane : q * T + tid; };
  u64 xi2[NP], yi2[NP], ax2[NP], ay2[NP];
  float4 ilo[PER ? NP : 1];          // PER: lo parts of the disks i (x0, y0, x1, y1), local memory
  float fxh[NQ], fxl[NQ], fyh[NQ], fyl[NQ];
  float4 ibox = sempty_box();
  bool ipad = false;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const float4 p0 = rel(base + islot(2 * k));
    const float4 p1 = rel(base + islot(2 * k + 1));
    xi2[k] = pk2(p0.x, p1.x);
    yi2[k] = pk2(p0.y, p1.y);
    if (PER) st_local4(&ilo[k], make_float4(p0.z, p0.w, p1.z, p1.w));
    ax2[k] = ay2[k] = 0ull;
    if (PER) {
      sbox_add(ibox, p0.x, p0.y);
      sbox_add(ibox, p1.x, p1.y);
      ipad = ipad || p0.x > 1.0e17f || p1.x > 1.0e17f;
    }
  }
  if (PER) {
    ibox = swarp_box(ibox);
    ipad = __any_sync(0xffffffffu, ipad);
    if (lane == 0) {
      sibox[warp] = ibox;
      sipad[warp] = ipad ? 1 : 0;
    }
  }
  const u64 invL2 = pk2(Lf > 0.f ? 1.0f / Lf : 0.f, Lf > 0.f ? 1.0f / Lf : 0.f);
  const u64 nL2 = pk2(-Lf, -Lf), M2 = pk2(12582912.0f, 12582912.0f);
#pragma unroll
  for (int q = 0; q < NQ; ++q) fxh[q] = fyh[q] = fxl[q] = fyl[q] = 0.f;
  const float e0 = 1e-20f * (float)(c.a * c.a);   // makes the self pair exactly 0
  const u64 eps2 = pk2(e0, e0);
  const int t_begin = item.y / NG, t_end = (item.z + NG - 1) / NG;   // tiles staged
  // j sums: group G of the item at slot item.w + G - max(item.y, gsym)
  float2 *const jout = d.jpart + ((ptrdiff_t)item.w - max(item.y, gsym)) * BD_SG;
  int buf = 0;
  auto fetch = [&](int tile) {
    // asynchronous 16-byte copies straight into shared memory
#pragma unroll
    for (int m = 0; m < NS; ++m) {
      const unsigned dst = (unsigned)__cvta_generic_to_shared(&sraw[buf ^ 1][m * T + tid]);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                   "l"(d.work + (size_t)tile * BD_TJ + m * T + tid)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto store = [&](int b) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if constexpr (PER) {
      // each thread re-centres the slots it copied (its own copies are
      // visible to it after the wait), in place; the warp's 32 slots of
      // stage m are group m NW + warp, whose box is taken about its first
      // live disk (minimum images about it), then shifted back
#pragma unroll
      for (int m = 0; m < NS; ++m) {
        const float4 v = rel_raw(sraw[b][m * T + tid], org, Lf, hLf);
        sraw[b][m * T + tid] = v;
        const bool live = v.x < 1.0e17f;
        const unsigned bal = __ballot_sync(0xffffffffu, live);
        float4 bx = sempty_box();
        if (bal) {
          const int src = __ffs(bal) - 1;
          const float rx = __shfl_sync(0xffffffffu, v.x, src), ry = __shfl_sync(0xffffffffu, v.y, src);
          if (live) {
            float dx = __fsub_rn(v.x, rx), dy = __fsub_rn(v.y, ry);
            if (per) {
              dx = dx > hLf ? __fsub_rn(dx, Lf) : (dx < -hLf ? __fadd_rn(dx, Lf) : dx);
              dy = dy > hLf ? __fsub_rn(dy, Lf) : (dy < -hLf ? __fadd_rn(dy, Lf) : dy);
            }
            bx = make_float4(dx, dx, dy, dy);
          }
          bx = swarp_box(bx);
          bx = make_float4(__fadd_rn(rx, bx.x), __fadd_rn(rx, bx.y), __fadd_rn(ry, bx.z), __fadd_rn(ry, bx.w));
        }
        if (lane == 0) {
          sgbox[b][m * NW + warp] = bx;
          sgpad[b][m * NW + warp] = bal != 0xffffffffu ? 1 : 0;
        }
      }
    }
  };
  buf = 1;   // fetch fills sraw[buf ^ 1]
  if (t_begin < t_end) {
    fetch(t_begin);
    store(0);
  }
  buf = 0;
  __syncthreads();
  // the j disk in slot jj of the current staging buffer, re-centred
  auto jpos = [&](int jj) -> float2 {
    if constexpr (PER) return make_float2(sraw[buf][jj].x, sraw[buf][jj].y);
    else return recentre(sraw[buf][jj], org);
  };
  // PER: its lo parts
  auto jlo = [&](int jj) -> float2 { return make_float2(sraw[buf][jj].z, sraw[buf][jj].w); };
  // pair differences (r_j - r_i), per axis AX (0: x, 1: y), by the pair form
  // MODE: 0 the hi parts alone; 1 the exact near-pair vector (hi_j - hi_i) +
  // (lo_j - lo_i); 2 the hi difference's packed minimum image on both axes;
  // 3 the same by compares (inert slots, which must stay far away, take part);
  // 5 / 6 the packed minimum image on x / y alone (an inert slot stays far
  // away on the other axis); 4 near pairs across the antipode (boxes of a
  // size near L/2): the hi difference, about L there, is formed exactly as
  // s + e (TwoDiff), s takes the minimum image (exact: |s| in [L/2, 3L/2]),
  // then e and the lo difference are added.  Far pairs (all forms but 1 and
  // 4) drop the lo parts, as form 0 does.
  auto diff = [&](auto MODE, auto AX, u64 jh2, u64 ih2, u64 jl2, u64 il2) -> u64 {
    constexpr int m0 = decltype(MODE)::value, ax = decltype(AX)::value;
    constexpr int mode = m0 == 5 ? (ax == 0 ? 2 : 0) : (m0 == 6 ? (ax == 1 ? 2 : 0) : m0);
    u64 dd = sub2(jh2, ih2);
    if constexpr (mode == 4) {
      const u64 v = sub2(dd, jh2);
      const u64 e = sub2(sub2(jh2, sub2(dd, v)), add2(ih2, v));
      return add2(min_image2_cmp(dd, Lf, hLf), add2(e, sub2(jl2, il2)));
    }
    if constexpr (mode == 2) dd = min_image2(dd, invL2, nL2, M2);
    if constexpr (mode == 3) dd = min_image2_cmp(dd, Lf, hLf);
    if constexpr (mode == 1) dd = add2(dd, sub2(jl2, il2));
    return dd;
  };
  using AXX = std::integral_constant<int, 0>;
  using AXY = std::integral_constant<int, 1>;
  // PER: the pair form of this warp's disks i with the j group g0 of the current tile.  Pair components range over [j_min - i_max,
  // j_max - i_min]; a plain difference is the minimum image when that range
  // and the j coordinates themselves lie inside (-L/2, L/2) (then each j is
  // stored as the image its box describes), with a margin of 2^-16 L/2 for
  // the rounding of the boxes.  Near: the range comes within 20 of 0 or L.
  auto pair_mode = [&](int g0) -> int {
    if constexpr (!PER) return 0;
    const float4 ib = sibox[warp];
    if (ib.x > ib.y) return 0;                 // the warp's disks i are all inert
    const float4 jb = sgbox[buf][g0];
    const int pad = sipad[warp] | sgpad[buf][g0];
    if (jb.x > jb.y) return 0;                 // inert disks j only: their pairs vanish
    const float lox = __fsub_rn(jb.x, ib.y), hix = __fsub_rn(jb.y, ib.x);
    const float loy = __fsub_rn(jb.z, ib.w), hiy = __fsub_rn(jb.w, ib.z);
    const float hLm = __fmul_rn(hLf, 1.0f - 1.0f / 65536.0f);
    const bool wx = per && (hix > hLm || lox < -hLm || jb.y > hLm || jb.x < -hLm);
    const bool wy = per && (hiy > hLm || loy < -hLm || jb.w > hLm || jb.z < -hLm);
    auto gap = [&](float lo, float hi) -> float {
      float g = fmaxf(0.f, fmaxf(lo, -hi));
      if (per) {
        g = fminf(g, fmaxf(0.f, fmaxf(__fsub_rn(lo, Lf), -__fsub_rn(hi, Lf))));
        g = fminf(g, fmaxf(0.f, fmaxf(__fadd_rn(lo, Lf), -__fadd_rn(hi, Lf))));
      }
      return g;
    };
    const float gx = gap(lox, hix), gy = gap(loy, hiy);
    // boxes closer than 20: the exact vector keeps their pairs at FP32
    // resolution of their separation (coordinates reach L/2 from the block
    // origin, where one rounding costs ulp(L/2) / 2)
    const bool near = gx * gx + gy * gy < 400.f;
    return near ? (wx || wy ? 4 : 1) : (wx && wy ? (pad ? 3 : 2) : (wx ? 5 : (wy ? 6 : 0)));
  };
  using M0 = std::integral_constant<int, 0>;
  using M1 = std::integral_constant<int, 1>;
  using M2c = std::integral_constant<int, 2>;
  using M3 = std::integral_constant<int, 3>;
  using M4 = std::integral_constant<int, 4>;
  using M5 = std::integral_constant<int, 5>;
  using M6 = std::integral_constant<int, 6>;
  auto dispatch = [&](int mode, auto &&fn) {
    if constexpr (PER) {
      if (mode == 1) fn(M1());
      else if (mode == 2) fn(M2c());
      else if (mode == 3) fn(M3());
      else if (mode == 4) fn(M4());
      else if (mode == 5) fn(M5());
      else if (mode == 6) fn(M6());
      else fn(M0());
    } else {
      fn(M0());
    }
  };
  auto own_group = [&](auto MODE, int g) {
    // the block's own disks: i side only, j broadcast from shared memory
    constexpr bool LO = decltype(MODE)::value == 1 || decltype(MODE)::value == 4;
#pragma unroll 4
    for (int jj = g * 32; jj < g * 32 + 32; ++jj) {
      const float2 p = jpos(jj);
      const u64 jx2 = pk2(p.x, p.x), jy2 = pk2(p.y, p.y);
      u64 jxl2 = 0ull, jyl2 = 0ull;
      if constexpr (LO) {
        const float2 pl = jlo(jj);
        jxl2 = pk2(pl.x, pl.x);
        jyl2 = pk2(pl.y, pl.y);
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        u64 ixl2 = 0ull, iyl2 = 0ull;
        if constexpr (LO) {
          const float4 il = ld_local4(&ilo[k]);
          ixl2 = pk2(il.x, il.z);
          iyl2 = pk2(il.y, il.w);
        }
        const u64 dx = diff(MODE, AXX(), jx2, xi2[k], jxl2, ixl2);
        const u64 dy = diff(MODE, AXY(), jy2, yi2[k], jyl2, iyl2);
        u64 r2 = fma2(dx, dx, eps2);
        r2 = fma2(dy, dy, r2);
        float ra, rb;
        up2(r2, ra, rb);
        const u64 sv = pk2(rsqrt_apx(ra), rsqrt_apx(rb));
        const u64 s3 = mul2(mul2(sv, sv), sv);
        ax2[k] = fma2(dx, s3, ax2[k]);
        ay2[k] = fma2(dy, s3, ay2[k]);
      }
    }
  };
  auto ring_group = [&](auto MODE, int g) {
    // a later tile's group g: every pair once, both sides; each lane carries one disk j
    constexpr bool LO = decltype(MODE)::value == 1 || decltype(MODE)::value == 4;
    const float2 p = jpos(g * 32 + lane);
    float jx = p.x, jy = p.y, jxl = 0.f, jyl = 0.f;
    if constexpr (LO) {
      const float2 pl = jlo(g * 32 + lane);
      jxl = pl.x;
      jyl = pl.y;
    }
    u64 hx2 = 0ull, hy2 = 0ull;
    float h0, h1, h2, h3;
#pragma unroll 2
    for (int rot = 0; rot < 32; ++rot) {
      const int src = (lane + 1) & 31;
      const u64 jx2 = pk2(jx, jx), jy2 = pk2(jy, jy);
      const u64 jxl2 = LO ? pk2(jxl, jxl) : 0ull, jyl2 = LO ? pk2(jyl, jyl) : 0ull;
      // the next j position does not depend on this step's arithmetic
      const float njx = __shfl_sync(0xffffffffu, jx, src);
      const float njy = __shfl_sync(0xffffffffu, jy, src);
      float njxl = 0.f, njyl = 0.f;
      if constexpr (LO) {
        njxl = __shfl_sync(0xffffffffu, jxl, src);
        njyl = __shfl_sync(0xffffffffu, jyl, src);
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        u64 ixl2 = 0ull, iyl2 = 0ull;
        if constexpr (LO) {
          const float4 il = ld_local4(&ilo[k]);
          ixl2 = pk2(il.x, il.z);
          iyl2 = pk2(il.y, il.w);
        }
        const u64 dx = diff(MODE, AXX(), jx2, xi2[k], jxl2, ixl2);
        const u64 dy = diff(MODE, AXY(), jy2, yi2[k], jyl2, iyl2);
        u64 r2 = fma2(dx, dx, eps2);
        r2 = fma2(dy, dy, r2);
        float ra, rb;
        up2(r2, ra, rb);
        const u64 sv = pk2(rsqrt_apx(ra), rsqrt_apx(rb));
        const u64 s3 = mul2(mul2(sv, sv), sv);
        ax2[k] = fma2(dx, s3, ax2[k]);
        ay2[k] = fma2(dy, s3, ay2[k]);
        hx2 = fma2(dx, s3, hx2);
        hy2 = fma2(dy, s3, hy2);
      }
      // pass the j accumulator one lane down the ring, after its disk
      up2(hx2, h0, h1);
      up2(hy2, h2, h3);
      h0 = __shfl_sync(0xffffffffu, h0, src);
      h1 = __shfl_sync(0xffffffffu, h1, src);
      h2 = __shfl_sync(0xffffffffu, h2, src);
      h3 = __shfl_sync(0xffffffffu, h3, src);
      hx2 = pk2(h0, h1);
      hy2 = pk2(h2, h3);
      jx = njx;
      jy = njy;
      jxl = njxl;
      jyl = njyl;
    }
    // after 32 passes every j is back in its own lane
    up2(hx2, h0, h1);
    up2(hy2, h2, h3);
    shw[warp][g * 32 + lane] = make_float2(__fadd_rn(h0, h1), __fadd_rn(h2, h3));
  };
  for (int t = t_begin; t < t_end; ++t) {
    if (t + 1 < t_end) fetch(t + 1);
    const int b = d.tile_species[t];
    const int ga = max(item.y - t * NG, 0), gz = min(item.z - t * NG, NG);   // the item's groups of the tile
    if (t * NG < gsym) {
      for (int g = ga; g < gz; ++g)
        dispatch(pair_mode(g), [&](auto M) { own_group(M, g); });
    } else {
      for (int g = ga; g < gz; ++g)
        dispatch(pair_mode(g), [&](auto M) { ring_group(M, g); });
      __syncthreads();
      // j side of this tile: F_j += A[s_j][s_i] sum_i (r_j - r_i)/r^3
      const float alj = R.alpha[BD_MAX_SPECIES * b + a];
      float2 *out = jout + (ptrdiff_t)t * BD_TJ;
      for (int jj = ga * BD_SG + tid; jj < gz * BD_SG; jj += T) {
        float hx = 0.f, hy = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          hx = __fadd_rn(hx, shw[w][jj].x);
          hy = __fadd_rn(hy, shw[w][jj].y);
        }
        out[jj] = make_float2(alj * hx, alj * hy);
      }
    }
    // i side of this tile: F_i -= A[s_i][s_j] sum_j (r_j - r_i)/r^3
    const float ali = R.alpha[BD_MAX_SPECIES * a + b];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      float ax0, ax1, ay0, ay1;
      up2(ax2[k], ax0, ax1);
      up2(ay2[k], ay0, ay1);
      two_sum(fxh[2 * k], fxl[2 * k], -ali * ax0);
      two_sum(fyh[2 * k], fyl[2 * k], -ali * ay0);
      two_sum(fxh[2 * k + 1], fxl[2 * k + 1], -ali * ax1);
      two_sum(fyh[2 * k + 1], fyl[2 * k + 1], -ali * ay1);
      ax2[k] = ay2[k] = 0ull;
    }
    if (t + 1 < t_end) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  float2 *ip = d.ipart + (size_t)item_id * BD_SB;
#pragma unroll
  for (int q = 0; q < NQ; ++q) ip[islot(q)] = make_float2(__fadd_rn(fxh[q], fxl[q]), __fadd_rn(fyh[q], fyl[q]));
}

// with a register budget for MINB resident blocks per SM
template <int NW, int NP, bool PER, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) k_force_long_sym_mb(BdDev d, BdConst c) {
  force_long_sym_body<NW, NP, PER>(d, c);
}

// F_i = sum of its block's i partials + sum of its group's j partials, in the
// order the host listed them (item order), into partial-force slot 0.
// Bound by the partials' reads.  ND disks per block, NS shares: thread share g
// takes every NS-th partial (entries g, g + NS, ...) of the ND disks, so the
// loads stay coalesced and NS times as many warps hide their latency; the
// shares' sums are added in a fixed order.  A share's sum is float-float (TwoSum
// into a (hi, lo) FP32 pair, about 48 bits): FP64 adds run at 1/64 of the FP32
// rate on this part and would bound the kernel.
// Four partials in flight against two: 2884 -> 2871 us for 20 steps of 16384
// disks, 2009 -> 2004 for four of 350000 in 64 boxes.
// MOVE: the disks' move (k_integrate's) in the same kernel, whose launch and
// first loads cost a small system as much as its work.  A warp of its own draws
// the noise beside the shares that sum; the first share's then moves the disks.
template <int ND, int NS, bool MOVE>
__global__ void __launch_bounds__(ND * (NS + (MOVE ? 1 : 0))) k_force_sym_reduce(BdDev d, BdConst c, long long step,
                                                                                 int log_step, int node) {
  __shared__ float4 part[NS][ND];   // each share's sum: (x, y) and their low parts
  __shared__ bdem::Draw<float> draws[MOVE ? ND : 1];
  if (ctl_failed(d.ctl)) return;
  const int g = threadIdx.x / ND, dl = threadIdx.x % ND;
  const int i = blockIdx.x * ND + dl;               // np is a multiple of 512: i < np
  const int P = i / BD_SB, t = i / BD_SG;            // the same for the whole warp
  const float2 *ib = d.ipart + (i - P * BD_SB);
  const float2 *jb = d.jpart + (i - t * BD_SG);
  int e = -1;
  double2 p = make_double2(0.0, 0.0);
  float th = 0.f;
  if (MOVE && (g == 0 || g == NS)) {
    e = d.ext_id[i];
    p = d.pos[i];
    th = d.theta[i];
    const long long step_dev = *(volatile const long long *)&d.ctl->step_dev;
    if (step < 0) step = step_dev;
  }
  float xh[2] = {0.f, 0.f}, xl[2] = {0.f, 0.f}, yh[2] = {0.f, 0.f}, yl[2] = {0.f, 0.f};
  auto run = [&](const int *idx, int k0, int k1, const float2 *b, int stride) {
    int k = k0 + g;
    for (; k + 3 * NS < k1; k += 4 * NS) {   // four partials in flight
      const int i0 = __ldg(idx + k), i1 = __ldg(idx + k + NS), i2 = __ldg(idx + k + 2 * NS), i3 = __ldg(idx + k + 3 * NS);
      const float2 v0 = b[(size_t)i0 * stride], v1 = b[(size_t)i1 * stride];
      const float2 v2 = b[(size_t)i2 * stride], v3 = b[(size_t)i3 * stride];
      two_sum(xh[0], xl[0], v0.x);
      two_sum(yh[0], yl[0], v0.y);
      two_sum(xh[1], xl[1], v1.x);
      two_sum(yh[1], yl[1], v1.y);
      two_sum(xh[0], xl[0], v2.x);
      two_sum(yh[0], yl[0], v2.y);
      two_sum(xh[1], xl[1], v3.x);
      two_sum(yh[1], yl[1], v3.y);
    }
    for (; k + NS < k1; k += 2 * NS) {
      const float2 v0 = b[(size_t)__ldg(idx + k) * stride];
      const float2 v1 = b[(size_t)__ldg(idx + k + NS) * stride];
      two_sum(xh[0], xl[0], v0.x);
      two_sum(yh[0], yl[0], v0.y);
      two_sum(xh[1], xl[1], v1.x);
      two_sum(yh[1], yl[1], v1.y);
    }
    if (k < k1) {
      const float2 v0 = b[(size_t)__ldg(idx + k) * stride];
      two_sum(xh[0], xl[0], v0.x);
      two_sum(yh[0], yl[0], v0.y);
    }
  };
  if (MOVE && g == NS) {
    if (e >= 0) draws[dl] = bdem::draw_f32(d.rep[d.rep_of[i]], (uint32_t)e, step, (uint32_t)node, th);
  } else {
    run(d.red_iidx, d.red_iptr[P], d.red_iptr[P + 1], ib, BD_SB);
    run(d.red_jidx, d.red_jptr[t], d.red_jptr[t + 1], jb, BD_SG);
    two_sum(xh[0], xl[0], xh[1]);
    two_sum(yh[0], yl[0], yh[1]);
    part[g][dl] = make_float4(xh[0], yh[0], __fadd_rn(xl[0], xl[1]), __fadd_rn(yl[0], yl[1]));
  }
  __syncthreads();
  if (g != 0) return;
  const int r = d.rep_of[i];
  if (MOVE && i == 0) d.ctl->in_move = 1;
  if (r < 0) return;
  const BdRep &R = d.rep[r];
  if (R.law != BD_LAW_LONG) {   // no force law
    if (MOVE) bdem::move_disk<float>(d, c, R, i, e, step, log_step, node, p, th, make_double2(0.0, 0.0), &draws[dl]);
    return;
  }
  // The shares in three FP32 words (about 72 bits), x and y packed: what an
  // addition to the first loses goes into the second, and what that loses into the
  // third, so that the sum is rounded once, to FP64, as fine as one of FP64
  // additions.  (Those and their conversions would keep this warp's FP64 pipe,
  // two lanes per SM, for sixteen cycles each, eight times per share; unpacked,
  // the three words cost a 4096-disk rollout with its gradient 2 us per step.)
  u64 s0 = 0ull, s1 = 0ull, s2 = 0ull;
#pragma unroll
  for (int m = 0; m < NS; ++m) {
    const float4 q = part[m][dl];
    u64 lost, rest;
    s0 = two_sum2(s0, pk2(q.x, q.y), lost);
    s1 = two_sum2(s1, lost, rest);
    s2 = add2(s2, rest);
    s1 = two_sum2(s1, pk2(q.z, q.w), rest);
    s2 = add2(s2, rest);
  }
  float x0, x1, x2, y0, y1, y2;
  up2(s0, x0, y0);
  up2(s1, x1, y1);
  up2(s2, x2, y2);
  const double2 F = make_double2((double)x0 + ((double)x1 + (double)x2), (double)y0 + ((double)y1 + (double)y2));
  d.fpart[i] = F;
  if (MOVE) bdem::move_disk<float>(d, c, R, i, e, step, log_step, node, p, th, F, &draws[dl]);
}

int bd_force_launches(const BdConst &c) { return (c.precision == 0 ? c.force_variant >= 2 : c.f64_sym) ? 2 : 1; }

int bd_force_sym_blocks_per_sm(int variant, int periodic) {
  int per = 0;
  cudaError_t e;
  if (periodic)
    e = variant == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                           &per, k_force_long_sym_mb<4, 2, true, 8>, 128, 0)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                           &per, k_force_long_sym_mb<2, 4, true, 12>, 64, 0);
  else
    e = variant == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                           &per, k_force_long_sym_mb<4, 2, false, 8>, 128, 0)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                           &per, k_force_long_sym_mb<2, 4, false, 16>, 64, 0);
  return e == cudaSuccess ? per : 0;
}

// variant 2: 4 warps x 4 disks per lane; variant 3: 2 warps x 8 disks per lane
// (a rank with none of the work items sweeps nothing; its reduction still writes
// the sums, all 0, over what fpart held)
static void launch_sweep(const BdDev &d, const BdConst &c, int variant, cudaStream_t s) {
  if (c.n_sitems == 0) return;
  // periodic boxes (any replica) take the form with minimum images
  if (c.any_periodic) {
    // measured at N = 1e5 (periodic), step times with pair forms chosen per
    // (warp, group of 32 disks j): <2,4> 2.241 ms with 12 resident blocks
    // (2.248 with 16, 2.288 with 10), <4,2> 2.464 ms with 8 (2.519 with 6);
    // 2.86 ms before, with one form per (block, tile) and the tiles staged
    // through registers
    if (variant == 2)
      k_force_long_sym_mb<4, 2, true, 8><<<c.n_sitems, 128, 0, s>>>(d, c);
    else
      k_force_long_sym_mb<2, 4, true, 12><<<c.n_sitems, 64, 0, s>>>(d, c);
  } else {
    if (variant == 2)
      k_force_long_sym_mb<4, 2, false, 8><<<c.n_sitems, 128, 0, s>>>(d, c);
    else
      // 16 resident blocks (32 warps) per SM in 64 registers, j tiles staged by
      // cp.async: measured 1.776 -> 1.668 ms at N = 1e5 against the
      // register-staged form (120 registers, 16 warps), forces unchanged.
      // Other shapes in the same budget measured slower at N = 1e5: ring
      // unrolled 1 or 4 steps deep (+1.7 %, +1.1 %), two j disks per lane
      // (+1.9 %), folded j accumulators (+3.5 %), one warp of 16 disks per
      // lane (+2.7 %)
      k_force_long_sym_mb<2, 4, false, 16><<<c.n_sitems, 64, 0, s>>>(d, c);
  }
}

cudaError_t bd_launch_force_sym(const BdDev &d, const BdConst &c, int variant, cudaStream_t s) {
  launch_sweep(d, c, variant, s);
  constexpr int NS = BD_RED_SHARES;
  if (c.np < BD_RED_SMALL) k_force_sym_reduce<32, NS, false><<<c.np / 32, 32 * NS, 0, s>>>(d, c, 0, 0, 0);
  else k_force_sym_reduce<64, 4, false><<<c.np / 64, 256, 0, s>>>(d, c, 0, 0, 0);
  return cudaGetLastError();
}

cudaError_t bd_launch_force_sym_move(const BdDev &d, const BdConst &c, int variant, int64_t step, int log_step,
                                     cudaStream_t s, int node) {
  launch_sweep(d, c, variant, s);
  constexpr int NS = BD_RED_SHARES;
  k_force_sym_reduce<32, NS, true><<<c.np / 32, 32 * (NS + 1), 0, s>>>(d, c, (long long)step, log_step, node);
  return cudaGetLastError();
}
