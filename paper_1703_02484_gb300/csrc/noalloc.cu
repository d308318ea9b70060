// bd_forces_noalloc: the all-pairs long-range force for callers that cannot
// allocate device memory.
//
// Some callers of this library cannot call cudaMalloc: a host framework that
// owns the whole device memory budget through its own allocator and must see
// every byte that is handed out, a latency-critical loop in which the device
// synchronisation implied by cudaMalloc/cudaFree is not acceptable, or a
// deployment that fixes the process's device footprint when the library is
// loaded.  They pass device buffers for the inputs and the output; the only
// scratch this entry point needs lives in the file-scope array below, which
// every GPU that loads the library holds until the process exits.
//
// Scratch layout (BD_NOALLOC_BYTES bytes):
//   double2 partial forces, [chunk][n]
// Every call rewrites every scratch element it reads, so nothing has to be
// cleared between calls.  All calls on a device share the one array: two calls
// whose kernels overlap on the GPU (e.g. on two streams) race on it, and the
// caller must serialise them.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "bd_internal.h"
#include "f32x2.cuh"

using namespace bdf;

#define BD_NOALLOC_MAX_N 65536
#define BD_NOALLOC_MAX_CHUNKS 64
#define BD_NOALLOC_BYTES ((size_t)BD_NOALLOC_MAX_N * 16 * 9)
#define BD_NA_THREADS 128
#define BD_NA_IPT 4
#define BD_NA_TJ 128

static __device__ __align__(256) unsigned char bd_noalloc_scratch[BD_NOALLOC_BYTES];

namespace {

struct NaArgs {
  int n, nchunk;
  const double2 *xy;
  const uint8_t *sp;
  double2 *F;
  double2 *part;
  float A[4];
};

// (hi, lo) FP32 pair of each FP64 coordinate
__device__ __forceinline__ float4 na_split(double2 p) {
  const float xh = __double2float_rn(p.x), yh = __double2float_rn(p.y);
  return make_float4(xh, yh, __double2float_rn(p.x - (double)xh), __double2float_rn(p.y - (double)yh));
}

// Variant of the tiled all-pairs sweep for disks in the caller's order:
// r_j - r_i is formed from the (hi, lo) pairs, which keeps near pairs exact
// without a spatial ordering.  Bound by the FP32 pipe: 12 lane operations per
// ordered pair (6 for the vector, 2 for r^2, 2 for r^-3, 2 into the sums) in
// packed f32x2 instructions, two disks i each.  The disks j of a tile are
// put in species order as they are staged (warp ballots, so the order is
// fixed), and the table's factor is applied once per tile and species instead of
// once per pair.  512 disks i per block of four warps, and as many j chunks as
// fill the SMs with eight blocks each: with few large blocks (two waves of
// one block per SM) the sweep left most issue slots empty.  Measured at 30011
// disks: 812 -> 430 us for the whole call, error against FP64 1.9e-7 -> 1.5e-7.  The split into
// FP32 pairs is done while staging (a kernel and a pass over memory less).
// Tiles of 128 with one double buffer; sums beyond a tile in float-float.
__global__ void __launch_bounds__(BD_NA_THREADS, 8) k_na_force(NaArgs g) {
  constexpr int NP = BD_NA_IPT / 2;
  __shared__ ulonglong2 sh[2][BD_NA_TJ], sl[2][BD_NA_TJ];   // per j: ((xh, xh), (yh, yh)), ((xl, xl), (yl, yl))
  __shared__ unsigned szero[2][BD_NA_TJ / 32];               // per warp: which of its j are species 0
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * BD_NA_THREADS * BD_NA_IPT;
  u64 xh[NP], yh[NP], xl[NP], yl[NP];
  float a0[BD_NA_IPT], a1[BD_NA_IPT], fxh[BD_NA_IPT], fxl[BD_NA_IPT], fyh[BD_NA_IPT], fyl[BD_NA_IPT];
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    float4 w[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = 2 * k + h, i = i0 + q * BD_NA_THREADS + tid;
      w[h] = make_float4(1.0e18f, 1.0e18f, 0.f, 0.f);
      a0[q] = a1[q] = 0.f;
      if (i < g.n) {
        w[h] = na_split(g.xy[i]);
        const int s = g.sp[i] ? 1 : 0;
        a0[q] = g.A[2 * s];
        a1[q] = g.A[2 * s + 1];
      }
      fxh[q] = fxl[q] = fyh[q] = fyl[q] = 0.f;
    }
    xh[k] = pk2(w[0].x, w[1].x);
    yh[k] = pk2(w[0].y, w[1].y);
    xl[k] = pk2(w[0].z, w[1].z);
    yl[k] = pk2(w[0].w, w[1].w);
  }
  const int per = (g.n + g.nchunk - 1) / g.nchunk;
  const int jb = blockIdx.y * per, je = min(g.n, jb + per);
  const u64 eps2 = pk2(1e-20f, 1e-20f);
  double2 pj = make_double2(0.0, 0.0);
  bool in = false, zero = false;
  // this thread's j of the tile at j0; its warp's species 0 lanes
  auto fetch = [&](int j0, int b) {
    const int j = j0 + tid;
    in = j < je;
    zero = false;
    if (in) {
      pj = g.xy[j];
      zero = g.sp[j] == 0;
    }
    const unsigned z = __ballot_sync(0xffffffffu, zero);
    if (lane == 0) szero[b][warp] = z;
  };
  // (after a barrier) into the tile: species 0 in order, then species 1 and
  // the far-away stand-ins past the chunk's end; returns the count of species 0
  auto store = [&](int b) -> int {
    int n0 = 0, before = 0;
#pragma unroll
    for (int w = 0; w < BD_NA_TJ / 32; ++w) {
      const int k = __popc(szero[b][w]);
      if (w < warp) before += k;
      n0 += k;
    }
    before += __popc(szero[b][warp] & ((1u << lane) - 1u));   // species 0 before this thread's j
    const int slot = zero ? before : n0 + (tid - before);
    const float4 w = in ? na_split(pj) : make_float4(1.0e18f, 1.0e18f, 0.f, 0.f);
    sh[b][slot] = make_ulonglong2(pk2(w.x, w.x), pk2(w.y, w.y));
    sl[b][slot] = make_ulonglong2(pk2(w.z, w.z), pk2(w.w, w.w));
    return n0;
  };
  int buf = 0, n0 = 0;
  if (jb < je) {
    fetch(jb, 0);
    __syncthreads();
    n0 = store(0);
  }
  __syncthreads();
  for (int j0 = jb; j0 < je; j0 += BD_NA_TJ) {
    const bool more = j0 + BD_NA_TJ < je;
    if (more) fetch(j0 + BD_NA_TJ, buf ^ 1);
    auto section = [&](int k0, int k1, const float *al) {
      u64 ax[NP], ay[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) ax[k] = ay[k] = 0ull;
#pragma unroll 4
      for (int jj = k0; jj < k1; ++jj) {
        const ulonglong2 ph = sh[buf][jj], pl = sl[buf][jj];
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          const u64 dx = add2(sub2(ph.x, xh[k]), sub2(pl.x, xl[k]));
          const u64 dy = add2(sub2(ph.y, yh[k]), sub2(pl.y, yl[k]));
          const u64 r2 = fma2(dy, dy, fma2(dx, dx, eps2));
          float ra, rb;
          up2(r2, ra, rb);
          const u64 s = pk2(rsqrt_apx(ra), rsqrt_apx(rb));
          const u64 s3 = mul2(mul2(s, s), s);
          ax[k] = fma2(dx, s3, ax[k]);
          ay[k] = fma2(dy, s3, ay[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        float x0, x1, y0, y1;
        up2(ax[k], x0, x1);
        up2(ay[k], y0, y1);
        two_sum(fxh[2 * k], fxl[2 * k], -al[2 * k] * x0);
        two_sum(fyh[2 * k], fyl[2 * k], -al[2 * k] * y0);
        two_sum(fxh[2 * k + 1], fxl[2 * k + 1], -al[2 * k + 1] * x1);
        two_sum(fyh[2 * k + 1], fyl[2 * k + 1], -al[2 * k + 1] * y1);
      }
    };
    section(0, n0, a0);
    section(n0, min(BD_NA_TJ, je - j0), a1);
    __syncthreads();
    if (more) n0 = store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int q = 0; q < BD_NA_IPT; ++q) {
    const int i = i0 + q * BD_NA_THREADS + tid;
    if (i < g.n)
      g.part[(size_t)blockIdx.y * g.n + i] =
          make_double2((double)fxh[q] + (double)fxl[q], (double)fyh[q] + (double)fyl[q]);
  }
}

__global__ void k_na_sum(NaArgs g) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.n) return;
  double fx = 0.0, fy = 0.0;
  for (int k = 0; k < g.nchunk; ++k) {
    double2 f = g.part[(size_t)k * g.n + i];
    fx += f.x;
    fy += f.y;
  }
  g.F[i] = make_double2(fx, fy);
}

std::mutex g_na_mutex;
void *g_na_ptr[256] = {nullptr};
int g_na_sms[256] = {0};

}  // namespace

extern "C" int bd_forces_noalloc(int32_t n, const double *xy, const uint8_t *species,
                                 const double alpha[4], double *F, void *stream) {
  if (n < 1 || n > BD_NOALLOC_MAX_N || !xy || !species || !alpha || !F) return BD_ERR_ARG;
  // positions and forces are read and written as 16-byte double2 pairs
  if (((uintptr_t)xy & 15u) != 0 || ((uintptr_t)F & 15u) != 0) return BD_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return BD_ERR_CUDA;
  void *base = nullptr;
  int sms = 0;
  {
    // once per device, with that device current: the device address of the
    // scratch array (its host-side name is only a stand-in) and the SM count
    std::lock_guard<std::mutex> lk(g_na_mutex);
    if (!g_na_ptr[dev]) {
      void *p = nullptr;
      int k = 0;
      if (cudaGetSymbolAddress(&p, bd_noalloc_scratch) != cudaSuccess || !p) return BD_ERR_CUDA;
      if (cudaDeviceGetAttribute(&k, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || k < 1)
        return BD_ERR_CUDA;
      g_na_sms[dev] = k;
      g_na_ptr[dev] = p;
    }
    base = g_na_ptr[dev];
    sms = g_na_sms[dev];
  }
  NaArgs g;
  g.n = n;
  int iblocks = (n + BD_NA_THREADS * BD_NA_IPT - 1) / (BD_NA_THREADS * BD_NA_IPT);
  // j chunks: at most as many as fill the eight blocks an SM holds (once: a
  // second, partly filled wave would idle SMs) and as the scratch holds partial
  // forces for, at least 64 disks j each; among these the count that leaves the
  // fullest SM the least work, blocks per SM times the chunk (30011 disks: 18
  // chunks, seven blocks on every SM, instead of 19, eight on some)
  int most = 8 * sms / iblocks;
  const int room = (int)(BD_NOALLOC_BYTES / 16 / (size_t)n);
  most = most > room ? room : most;
  most = most > BD_NOALLOC_MAX_CHUNKS ? BD_NOALLOC_MAX_CHUNKS : most;
  most = most > (n + 63) / 64 ? (n + 63) / 64 : most;
  most = most < 1 ? 1 : most;
  int nchunk = most;
  long long best = -1;
  for (int k = most; k >= 1 && 2 * k >= most; --k) {
    const long long load = (long long)((iblocks * k + sms - 1) / sms) * ((n + k - 1) / k);
    if (best < 0 || load < best) {
      best = load;
      nchunk = k;
    }
  }
  g.nchunk = nchunk;
  g.xy = (const double2 *)xy;
  g.sp = species;
  g.F = (double2 *)F;
  g.part = (double2 *)base;
  for (int k = 0; k < 4; ++k) g.A[k] = (float)alpha[k];
  cudaStream_t s = (cudaStream_t)stream;
  k_na_force<<<dim3(iblocks, nchunk), BD_NA_THREADS, 0, s>>>(g);
  k_na_sum<<<(n + 255) / 256, 256, 0, s>>>(g);
  if (cudaGetLastError() != cudaSuccess) return BD_ERR_CUDA;
  return BD_OK;
}
