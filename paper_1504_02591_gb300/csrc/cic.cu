// cic.cu: cloud-in-cell mass assignment and interpolation, the reconstruction shift, reductions.
//
// Mass assignment (Sec. 3 bins tracers on the mesh; this library uses CIC instead of NGP): a
// particle at grid coordinate u = x N / L deposits w (1 - t) and w t on the nodes floor(u) and
// floor(u) + 1 of each axis, t = u - floor(u), with periodic wrap.  The same kernel interpolates
// Psi back to particles for the shift of Sec. 1 (reversing Eq. Lagrange x = q + Psi).
#include <mutex>

#include "../../include/recon.h"
#include "cic.h"
#include "reduce.cuh"

namespace rg {

// Nodes and weights of one particle.  u 2^32 = x times scale 2^32 (exact scaling) rounded down to an
// integer T: floor(u) = T >> 32 and t = (T mod 2^32) 2^-32.  One float64 operation per axis (float64
// runs at a small fraction of the float32 rate on this GPU).
template <typename PT>
__device__ __forceinline__ void cic_setup(const PT* __restrict__ pos, long long p, int n, double scale,
                                          int (&i0)[3], int (&i1)[3], float (&t)[3]) {
  const double scale32 = scale * 4294967296.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const long long T = floor_scaled(widen(pos[3 * p + a]), scale32, 0.0);
    t[a] = (float)(uint32_t)T * 2.3283064365386963e-10f;   // 2^-32
    int c = (int)(T >> 32);
    if (c < 0 || c >= n) c = ((c % n) + n) % n;   // outside [0, L): periodic image
    i0[a] = c;
    i1[a] = (c + 1 == n) ? 0 : c + 1;
  }
}

__device__ __forceinline__ double block_sum_d(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  return r;
}

template <typename PT>
__global__ void __launch_bounds__(256) deposit_kernel(const PT* __restrict__ pos, const float* __restrict__ w,
                                                      long long np, int n, double scale,
                                                      float* __restrict__ rho, double* __restrict__ partials) {
  double wsum = 0.0;
  int count = 0;   // unit weights: a thread's share is far below 2^31
  const size_t nn = (size_t)n;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    int i0[3], i1[3];
    float t[3];
    cic_setup(pos, p, n, scale, i0, i1, t);
    const float wp = w ? w[p] : 1.f;
    if (w) wsum += wp;
    else ++count;
    const float wx0 = wp * (1.f - t[0]), wx1 = wp * t[0];
    const float wy0 = 1.f - t[1], wy1 = t[1];
    const float wz0 = 1.f - t[2], wz1 = t[2];
    const size_t r00 = ((size_t)i0[0] * nn + i0[1]) * nn, r01 = ((size_t)i0[0] * nn + i1[1]) * nn;
    const size_t r10 = ((size_t)i1[0] * nn + i0[1]) * nn, r11 = ((size_t)i1[0] * nn + i1[1]) * nn;
    atomicAdd(rho + r00 + i0[2], wx0 * wy0 * wz0);
    atomicAdd(rho + r00 + i1[2], wx0 * wy0 * wz1);
    atomicAdd(rho + r01 + i0[2], wx0 * wy1 * wz0);
    atomicAdd(rho + r01 + i1[2], wx0 * wy1 * wz1);
    atomicAdd(rho + r10 + i0[2], wx1 * wy0 * wz0);
    atomicAdd(rho + r10 + i1[2], wx1 * wy0 * wz1);
    atomicAdd(rho + r11 + i0[2], wx1 * wy1 * wz0);
    atomicAdd(rho + r11 + i1[2], wx1 * wy1 * wz1);
  }
  const double s = block_sum_d(w ? wsum : (double)count);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// Nearest-grid-point binning (Sec. 3, the paper's scheme): node floor(u + 1/2) per axis, from the
// same 32.32 fixed-point coordinate as the CIC kernel (u 2^32 + 2^31 rounded down).  Four particles'
// positions are read before any is used: floor_scaled's rare branch keeps the compiler from doing so, and one
// at a time the pass waits for memory (3e7 float64 positions with unit weights: 537 us, 657 one at a time).
template <typename PT>
__global__ void __launch_bounds__(256) ngp_deposit_kernel(const PT* __restrict__ pos, const float* __restrict__ w,
                                                          long long np, int n, double scale,
                                                          float* __restrict__ rho, double* __restrict__ partials) {
  constexpr int U = 4;
  double wsum = 0.0;
  int count = 0;
  const size_t nn = (size_t)n;
  const double scale32 = scale * 4294967296.0;
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long p0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; p0 < np; p0 += U * step) {
    PT x[U][3];
    float wp[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long p = p0 + u * step < np ? p0 + u * step : p0;
#pragma unroll
      for (int a = 0; a < 3; ++a) x[u][a] = __ldg(pos + 3 * p + a);
      wp[u] = w ? __ldg(w + p) : 1.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (p0 + u * step >= np) break;
      int c[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const long long T = floor_scaled(widen(x[u][a]), scale32, 2147483648.0);
        int k = (int)(T >> 32);
        if (k < 0 || k >= n) k = ((k % n) + n) % n;
        c[a] = k;
      }
      if (w) wsum += wp[u];
      else ++count;
      atomicAdd(rho + ((size_t)c[0] * nn + c[1]) * nn + c[2], wp[u]);
    }
  }
  const double s = block_sum_d(w ? wsum : (double)count);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// x as the sum of two float32, by integer operations (a float64 conversion or sum costs 16 clocks a warp and
// SM here, and a pass over 3.1e7 float64 positions spent them on little else): hi holds the 24 leading bits of
// x and lo the 24 that follow, so x - hi - lo is less than 2^-47 |x|.  False outside 2^-60 <= |x| < 2^60
// (but true for zero).
__device__ __forceinline__ bool split_pair(double x, float& hi, float& lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const uint32_t h = (uint32_t)(b >> 32), e = (h >> 20) & 0x7ffu;
  const uint32_t top = (uint32_t)(b >> 29) & 0x7fffffu, low = (uint32_t)(b >> 5) & 0xffffffu;
  const uint32_t sign = h & 0x80000000u, e8 = (e - 896u) << 23;     // 1023 - 127 = 896
  hi = __uint_as_float(sign | e8 | top);
  lo = __uint_as_float(sign | (e8 - (47u << 23))) * (float)low;     // 2^(exponent - 47) times an integer below 2^24
  if (b << 1 == 0) hi = lo = 0.f;
  return b << 1 == 0 || e - 963u < 120u;                            // 1023 - 60 = 963
}
__device__ __forceinline__ bool split_pair(float x, float& hi, float& lo) {
  hi = x;
  lo = 0.f;
  return fabsf(x) < 1e18f;
}

// Shell of a particle: floor((r - rmin) inv_dr) clamped to [-1, nbins], r its float64 distance from obs.
// float64 operations cost most of a pass here, so the shell is found in float32 (the offsets from pairs) unless
// the coordinate lies so near a shell's edge that its rounding could matter: the float32 coordinate is off
// by at most 2^-24 (5 r + 2 rmin) inv_dr + 2^-23 |f| (three offsets of two roundings, two fused sums and a
// correctly rounded root, then one difference and one product) and what the pairs leave out, less than
// 2^-46 of |x| and |obs| on each axis; the margin is three times that and more.  Near an edge, and for
// coordinates that are not finite, the float64 expression decides.
struct ShellArgs {
  double3 obs;
  float3 hi, lo;         // obs as pairs
  double rmin, inv_dr;
  int nbins;
  int pairs;             // obs fits them
};

template <typename PT>
__device__ __forceinline__ int shell_of(PT x, PT y, PT z, const ShellArgs& a) {
  float hx, lx, hy, ly, hz, lz;
  const bool ok = split_pair(x, hx, lx) & split_pair(y, hy, ly) & split_pair(z, hz, lz) & (a.pairs != 0);
  const float fx = (hx - a.hi.x) + (lx - a.lo.x), fy = (hy - a.hi.y) + (ly - a.lo.y), fz = (hz - a.hi.z) + (lz - a.lo.z);
  const float r = __fsqrt_rn(fmaf(fx, fx, fmaf(fy, fy, fz * fz)));
  const float rm = (float)a.rmin, inv = (float)a.inv_dr;
  const float f = (r - rm) * inv;
  const float left = 1e-13f * ((fabsf(hx) + fabsf(a.hi.x)) + (fabsf(hy) + fabsf(a.hi.y)) + (fabsf(hz) + fabsf(a.hi.z)));
  const float margin = fmaf(fmaf(1.2e-6f, r + fabsf(rm), left), inv, 6e-7f * fabsf(f));
  const float k = floorf(f);
  if (ok && f - k > margin && k + 1.f - f > margin && r > 1e-15f && r < 1e18f && fabsf(f) < 1e6f)
    return k < 0.f ? -1 : (k >= (float)a.nbins ? a.nbins : (int)k);
  const double dx = (double)x - a.obs.x, dy = (double)y - a.obs.y, dz = (double)z - a.obs.z;
  const double b = floor((sqrt(dx * dx + dy * dy + dz * dz) - a.rmin) * a.inv_dr);
  return b >= 0.0 ? (b < (double)a.nbins ? (int)b : a.nbins) : -1;
}

// Shells of the particles p0 + u step below np, u < U, their positions read before any is used.
template <int U, typename PT, class Fn>
__device__ __forceinline__ void shells(const PT* __restrict__ pos, long long p0, long long step, long long np,
                                       const ShellArgs& a, Fn&& fn) {
  PT x[U][3];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const long long p = p0 + u * step < np ? p0 + u * step : p0;
#pragma unroll
    for (int c = 0; c < 3; ++c) x[u][c] = __ldg(pos + 3 * p + c);
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (p0 + u * step < np) fn(p0 + u * step, shell_of(x[u][0], x[u][1], x[u][2], a));
}

// Radial number density (Sec. 3.2 n(z), in comoving distance from the observer): counts of the
// particles in nbins equal shells of [rmin, rmax), float64 distances; counted per block in shared memory
// (6e5 galaxies in 50 shells: 120 us when every particle went to a global counter).
template <typename PT>
__global__ void __launch_bounds__(256) radial_hist_kernel(const PT* __restrict__ pos, long long np, const ShellArgs a,
                                                          unsigned long long* __restrict__ counts) {
  const int nbins = a.nbins;
  __shared__ unsigned int h[4096];
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) h[b] = 0u;
  __syncthreads();
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long p0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; p0 < np; p0 += 4 * step)
    shells<4>(pos, p0, step, np, a, [&](long long, int b) {
      if (b >= 0 && b < nbins) atomicAdd(h + b, 1u);
    });
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x)
    if (h[b]) atomicAdd(counts + b, (unsigned long long)h[b]);
}

// FKP weights (Sec. 3.2): the table's entry of the particle's shell, its last entry outside the shells.
// A weight depends on the shell alone, so the quotients are formed once per shell on the host.  Bound by the
// positions' bytes: 3.1e7 float64 positions 355 us with float64 offsets, 220 with pairs.
template <typename PT>
__global__ void __launch_bounds__(256) fkp_kernel(const PT* __restrict__ pos, long long np, const ShellArgs a,
                                                  const float* __restrict__ wtab, float* __restrict__ w) {
  const long long step = (long long)gridDim.x * blockDim.x;
  for (long long p0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; p0 < np; p0 += 4 * step)
    shells<4>(pos, p0, step, np, a, [&](long long p, int b) { w[p] = __ldg(wtab + (b < 0 ? a.nbins : b)); });
}

static ShellArgs shell_args(double3 obs, double rmin, double inv_dr, int nbins) {
  ShellArgs a{};
  a.obs = obs;
  a.rmin = rmin;
  a.inv_dr = inv_dr;
  a.nbins = nbins;
  const double o[3] = {obs.x, obs.y, obs.z};
  float hi[3], lo[3];
  a.pairs = 1;
  for (int c = 0; c < 3; ++c) {
    hi[c] = (float)o[c];
    lo[c] = (float)(o[c] - (double)hi[c]);
    if (!(o[c] > -1e18 && o[c] < 1e18)) a.pairs = 0;
  }
  a.hi = make_float3(hi[0], hi[1], hi[2]);
  a.lo = make_float3(lo[0], lo[1], lo[2]);
  return a;
}

__global__ void __launch_bounds__(256) pack_psi_kernel(const float4* __restrict__ x, const float4* __restrict__ y,
                                                       const float4* __restrict__ z, float4* __restrict__ out, size_t n4) {
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n4; i += (size_t)gridDim.x * 256) {
    const float4 a = x[i], b = y[i], c = z[i];
    out[4 * i] = make_float4(a.x, b.x, c.x, 0.f);
    out[4 * i + 1] = make_float4(a.y, b.y, c.y, 0.f);
    out[4 * i + 2] = make_float4(a.z, b.z, c.z, 0.f);
    out[4 * i + 3] = make_float4(a.w, b.w, c.w, 0.f);
  }
}

// The shift of each particle by itself.  Gathers of particles in no order are bound by the L1's look-ups, one
// per lane and load: 24 of them from three fields, 8 from nodes packed as float4 (PACKED).
template <typename PT, bool PACKED>
__global__ void __launch_bounds__(256) shift_kernel(const PT* __restrict__ pos, long long np, ShiftArgs a) {
  __shared__ double slots_sm[8][96];
  double* slots = slots_sm[threadIdx.x >> 5];
  const size_t nn = (size_t)a.n;
  // whole warps stay in the loop: the stores go through the warp's slots
  for (long long p0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); p0 < np;
       p0 += (long long)gridDim.x * blockDim.x) {
    const long long pl = p0 + (threadIdx.x & 31), p = pl < np ? pl : np - 1;
    int i0[3], i1[3];
    float t[3];
    cic_setup(pos, p, a.n, a.scale, i0, i1, t);
    const size_t r00 = ((size_t)i0[0] * nn + i0[1]) * nn, r01 = ((size_t)i0[0] * nn + i1[1]) * nn;
    const size_t r10 = ((size_t)i1[0] * nn + i0[1]) * nn, r11 = ((size_t)i1[0] * nn + i1[1]) * nn;
    const float wx0 = 1.f - t[0], wx1 = t[0], wy0 = 1.f - t[1], wy1 = t[1], wz0 = 1.f - t[2], wz1 = t[2];
    const size_t idx[8] = {r00 + i0[2], r00 + i1[2], r01 + i0[2], r01 + i1[2],
                           r10 + i0[2], r10 + i1[2], r11 + i0[2], r11 + i1[2]};
    const float cw[8] = {wx0 * wy0 * wz0, wx0 * wy0 * wz1, wx0 * wy1 * wz0, wx0 * wy1 * wz1,
                         wx1 * wy0 * wz0, wx1 * wy0 * wz1, wx1 * wy1 * wz0, wx1 * wy1 * wz1};
    float ps[3] = {0.f, 0.f, 0.f};
    if (PACKED) {
      float4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldg(a.psi4 + idx[k]);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        ps[0] = fmaf(cw[k], v[k].x, ps[0]);
        ps[1] = fmaf(cw[k], v[k].y, ps[1]);
        ps[2] = fmaf(cw[k], v[k].z, ps[2]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc = fmaf(cw[k], __ldg(a.psi[c] + idx[k]), acc);
        ps[c] = acc;
      }
    }
    float d[3];
    if (a.is_galaxy) {
      float rx, ry, rz;
      if (a.los_mode == 1) {
        rx = a.los.x; ry = a.los.y; rz = a.los.z;
      } else {
        // offset of the particle's image in [0, L) from the observer, as the brick-sorted path forms it
        const int n = a.n;
        const float dx = fmaf(t[0], a.H, a.off[i0[0]]), dy = fmaf(t[1], a.H, a.off[n + i0[1]]),
                    dz = fmaf(t[2], a.H, a.off[2 * n + i0[2]]);
        const float q = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float ir = q > 0.f ? rsqrtf(q) : 0.f;
        rx = dx * ir; ry = dy * ir; rz = dz * ir;
      }
      const float u = a.f * fmaf(ps[0], rx, fmaf(ps[1], ry, ps[2] * rz));
      d[0] = -fmaf(u, rx, ps[0]);
      d[1] = -fmaf(u, ry, ps[1]);
      d[2] = -fmaf(u, rz, ps[2]);
    } else {
      d[0] = -ps[0]; d[1] = -ps[1]; d[2] = -ps[2];
    }
    warp_store3(a.shift, p0, np, d, reinterpret_cast<float*>(slots));
    if (a.pos_out) {
      double y[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        y[c] = widen(pos[3 * p + c]) + d[c];
        if (a.periodic) y[c] = wrap_box(y[c], a.L);
      }
      warp_store3(a.pos_out, p0, np, y, slots);
    }
  }
}

// Sums the per-block partials (nq <= 4 quantities, interleaved): red[dst + q] (=|+=) sum_b partials[b * nq + q].
// 4.3 us for up to 1024 partials (8.1 with 1024 threads).
__global__ void __launch_bounds__(kReduceThreads) finalize_kernel(const double* __restrict__ partials, int nblocks, int nq,
                                                                  double* __restrict__ red, int dst, int accumulate,
                                                                  double* __restrict__ bsum, unsigned int* __restrict__ counter) {
  double t[4];
  if (reduce_partials(partials, nblocks, nq, bsum, counter, t))
    for (int q = 0; q < nq; ++q) red[dst + q] = accumulate ? red[dst + q] + t[q] : t[q];
}

__global__ void add_scalar_kernel(float* __restrict__ x, size_t n, float v) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    x[i] += v;
}

cudaError_t launch_deposit(const void* pos, int dtype, const float* w, long long np, int n, double L,
                           float* rho, double* partials, int blocks, cudaStream_t st, int ngp) {
  if (np <= 0) return cudaSuccess;
  const double scale = (double)n / L;
  if (ngp) {
    if (dtype == 0)
      ngp_deposit_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, w, np, n, scale, rho, partials);
    else
      ngp_deposit_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, w, np, n, scale, rho, partials);
    return cudaGetLastError();
  }
  if (dtype == 0)
    deposit_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, w, np, n, scale, rho, partials);
  else
    deposit_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, w, np, n, scale, rho, partials);
  return cudaGetLastError();
}

cudaError_t launch_pack_psi(const float* const psi[3], float4* psi4, size_t n, cudaStream_t st) {
  const size_t want = (n / 4 + 255) / 256;
  const int blocks = (int)(want < 152 * 16 ? want : 152 * 16);
  pack_psi_kernel<<<blocks, 256, 0, st>>>(reinterpret_cast<const float4*>(psi[0]), reinterpret_cast<const float4*>(psi[1]),
                                          reinterpret_cast<const float4*>(psi[2]), psi4, n / 4);
  return cudaGetLastError();
}

template <typename PT>
static void shift_launch(const void* pos, long long np, const ShiftArgs& a, int blocks, cudaStream_t st) {
  if (a.psi4) shift_kernel<PT, true><<<blocks, 256, 0, st>>>((const PT*)pos, np, a);
  else shift_kernel<PT, false><<<blocks, 256, 0, st>>>((const PT*)pos, np, a);
}

cudaError_t launch_shift(const void* pos, int dtype, long long np, const ShiftArgs& a, cudaStream_t st) {
  if (np <= 0) return cudaSuccess;
  long long want = (np + 255) / 256;
  const int blocks = (int)(want < 152 * 16 ? want : 152 * 16);
  if (dtype == 0) shift_launch<double>(pos, np, a, blocks, st);
  else shift_launch<float>(pos, np, a, blocks, st);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const double* partials, int nblocks, int nq, double* red, int dst, int accumulate,
                            cudaStream_t st, double* bsum, unsigned int* counter) {
  if (nq < 1 || nq > 4) return cudaErrorInvalidValue;
  const int blocks = bsum && counter ? reduce_blocks(nblocks, kFinalizeBlocks) : 1;
  finalize_kernel<<<blocks, kReduceThreads, 0, st>>>(partials, nblocks, nq, red, dst, accumulate, bsum, counter);
  return cudaGetLastError();
}

cudaError_t launch_add_scalar(float* x, size_t n, float v, cudaStream_t st) {
  add_scalar_kernel<<<152 * 8, 256, 0, st>>>(x, n, v);
  return cudaGetLastError();
}

// One ratio into the running statistics (float64; the decision at the cut is taken in float64 on
// the float32 inputs).
__device__ __forceinline__ void ratio_acc(float num, float den, double lo, double hi, double (&acc)[4]) {
  acc[3] += 1.0;
  if (den != 0.f) {
    const double r = (double)num / (double)den;
    if (r >= lo && r <= hi) {
      acc[0] += 1.0;
      acc[1] += r;
      acc[2] += r * r;
    }
  }
}

__device__ __forceinline__ void ratio_flush(double (&acc)[4], double* partials) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const double s = block_sum_d(acc[q]);
    if (threadIdx.x == 0) partials[4 * blockIdx.x + q] = s;
  }
}

template <typename PT>
__global__ void __launch_bounds__(256) radial_ratio_kernel(const PT* __restrict__ pos, long long np, RatioArgs a) {
  const size_t nn = (size_t)a.n;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    int i0[3], i1[3];
    float t[3];
    cic_setup(pos, p, a.n, a.scale, i0, i1, t);
    const size_t r00 = ((size_t)i0[0] * nn + i0[1]) * nn, r01 = ((size_t)i0[0] * nn + i1[1]) * nn;
    const size_t r10 = ((size_t)i1[0] * nn + i0[1]) * nn, r11 = ((size_t)i1[0] * nn + i1[1]) * nn;
    const float wx0 = 1.f - t[0], wx1 = t[0], wy0 = 1.f - t[1], wy1 = t[1], wz0 = 1.f - t[2], wz1 = t[2];
    const size_t idx[8] = {r00 + i0[2], r00 + i1[2], r01 + i0[2], r01 + i1[2],
                           r10 + i0[2], r10 + i1[2], r11 + i0[2], r11 + i1[2]};
    const float cw[8] = {wx0 * wy0 * wz0, wx0 * wy0 * wz1, wx0 * wy1 * wz0, wx0 * wy1 * wz1,
                         wx1 * wy0 * wz0, wx1 * wy0 * wz1, wx1 * wy1 * wz0, wx1 * wy1 * wz1};
    float rv[3];
    if (a.los_mode == 1) {
      rv[0] = a.los.x; rv[1] = a.los.y; rv[2] = a.los.z;
    } else {
      const int n = a.n;
      const float dx = fmaf(t[0], a.H, a.off[i0[0]]), dy = fmaf(t[1], a.H, a.off[n + i0[1]]),
                  dz = fmaf(t[2], a.H, a.off[2 * n + i0[2]]);
      const float q = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      const float ir = q > 0.f ? rsqrtf(q) : 0.f;
      rv[0] = dx * ir; rv[1] = dy * ir; rv[2] = dz * ir;
    }
    float un = 0.f, ud = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float gn = 0.f, gd = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        gn = fmaf(cw[k], __ldg(a.num[c] + idx[k]), gn);
        gd = fmaf(cw[k], __ldg(a.den[c] + idx[k]), gd);
      }
      un = fmaf(gn, rv[c], un);
      ud = fmaf(gd, rv[c], ud);
    }
    ratio_acc(un, ud, a.lo, a.hi, acc);
  }
  ratio_flush(acc, a.partials);
}

__global__ void __launch_bounds__(256) ratio_kernel(const float* __restrict__ num, const float* __restrict__ den,
                                                    size_t n, double lo, double hi, double* __restrict__ partials) {
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    ratio_acc(num[i], den[i], lo, hi, acc);
  ratio_flush(acc, partials);
}

cudaError_t launch_radial_ratio(const void* pos, int dtype, long long np, const RatioArgs& a, int blocks,
                                cudaStream_t st) {
  if (dtype == 0)
    radial_ratio_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, np, a);
  else
    radial_ratio_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, np, a);
  return cudaGetLastError();
}

cudaError_t launch_radial_hist(const void* pos, int dtype, long long np, double3 obs, double rmin, double rmax,
                               int nbins, unsigned long long* counts, cudaStream_t st) {
  if (np <= 0) return cudaSuccess;
  const double inv_dr = nbins / (rmax - rmin);
  const int blocks = (int)((np + 255) / 256 < 152 * 16 ? (np + 255) / 256 : 152 * 16);
  const ShellArgs sa = shell_args(obs, rmin, inv_dr, nbins);
  if (dtype == 0)
    radial_hist_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, np, sa, counts);
  else
    radial_hist_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, np, sa, counts);
  return cudaGetLastError();
}

cudaError_t launch_fkp(const void* pos, int dtype, long long np, double3 obs, double rmin, double rmax, int nbins,
                       const float* wtab, float* w, cudaStream_t st) {
  if (np <= 0) return cudaSuccess;
  const double inv_dr = nbins / (rmax - rmin);
  const int blocks = (int)((np + 255) / 256 < 152 * 16 ? (np + 255) / 256 : 152 * 16);
  const ShellArgs sa = shell_args(obs, rmin, inv_dr, nbins);
  if (dtype == 0)
    fkp_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, np, sa, wtab, w);
  else
    fkp_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, np, sa, wtab, w);
  return cudaGetLastError();
}

cudaError_t launch_ratio(const float* num, const float* den, size_t n, double lo, double hi, double* partials,
                         int blocks, cudaStream_t st) {
  ratio_kernel<<<blocks, 256, 0, st>>>(num, den, n, lo, hi, partials);
  return cudaGetLastError();
}

}  // namespace rg

// ------------------------------------------------------------------------------------------------
// CIC deposit that allocates nothing (recon_cic_deposit_noalloc).  The only scratch it needs, the
// per-block partial sums of the weights, lives in a fixed file-scope device array; every device
// that loads the library holds these 32 KB until the process exits.
// ------------------------------------------------------------------------------------------------
namespace rg {
namespace {

constexpr int kNoAllocMaxBlocks = 4096;                    // partial sums in the static scratch
constexpr long long kNoAllocPerThread = 64;                // particles per thread at most
constexpr long long kNoAllocMaxParticles = (long long)kNoAllocMaxBlocks * 256 * kNoAllocPerThread;
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) double g_noalloc_partials[kNoAllocMaxBlocks];

std::mutex g_noalloc_mu;
double* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of the scratch array for the current device, looked up once per device.  The
// host-side name of a __device__ array is only a stand-in: kernels must be given this address.
cudaError_t noalloc_scratch(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_partials);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace
}  // namespace rg

extern "C" recon_status recon_cic_deposit_noalloc(const void* pos, int dtype, const float* w, int64_t n,
                                                  int nmesh, double box, float* rho, double* sum_w,
                                                  void* stream) {
  using namespace rg;
  if (n < 0 || (n > 0 && !pos) || !rho || !sum_w || nmesh < 2 || nmesh > 2048 || !(box > 0))
    return RECON_ERR_INVALID_ARG;
  if (dtype != RECON_F64 && dtype != RECON_F32) return RECON_ERR_INVALID_ARG;
  if (n > kNoAllocMaxParticles) return RECON_ERR_INVALID_ARG;
  double* scratch = nullptr;
  if (noalloc_scratch(&scratch) != cudaSuccess) {
    cudaGetLastError();
    return RECON_ERR_CUDA;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const size_t cells = (size_t)nmesh * nmesh * nmesh;
  if (cudaMemsetAsync(rho, 0, cells * sizeof(float), st) != cudaSuccess) return RECON_ERR_CUDA;
  if (n == 0) return cudaMemsetAsync(sum_w, 0, sizeof(double), st) == cudaSuccess ? RECON_OK : RECON_ERR_CUDA;
  long long blocks = (n + 255) / 256;
  if (blocks > kNoAllocMaxBlocks) blocks = kNoAllocMaxBlocks;
  if (launch_deposit(pos, dtype == RECON_F64 ? 0 : 1, w, n, nmesh, box, rho, scratch, (int)blocks, st) != cudaSuccess)
    return RECON_ERR_CUDA;
  if (launch_finalize(scratch, (int)blocks, 1, sum_w, 0, 0, st) != cudaSuccess) return RECON_ERR_CUDA;
  return RECON_OK;
}
