// unet.cu: the learned warm start — a small periodic 3-D U-Net with its own forward, backward and
// AdamW kernels (float32 accumulation; activations stored as bfloat16 or float32).
//
// Network (3 levels, widths c1/2c1/4c1): two 3x3x3 conv+ReLU per level, 2x2x2 average pooling down,
// nearest-neighbour 2x upsampling up, skip connections by channel concatenation, and a 1x1x1 head
// whose output is added to the last input channel (the radial displacement of the Eq. approx2
// start), so the network predicts the correction that brings the start to the converged solution
// of Eq. Nusser.  Tensors are channels-last [voxel][channel] on a periodic n^3 grid; a 3x3x3 kernel
// w[tap][cin][cout] computes y[v][co] = b[co] + sum_tap sum_ci x[v + d(tap)][ci] w[tap][ci][co].
#include <cuda_bf16.h>

#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/recon.h"
#include "unet_tc.h"

namespace rg {
namespace {

typedef __nv_bfloat16 bf16;

template <typename T>
__device__ __forceinline__ float tof(T v);
template <>
__device__ __forceinline__ float tof<float>(float v) { return v; }
template <>
__device__ __forceinline__ float tof<bf16>(bf16 v) { return __bfloat162float(v); }
template <typename T>
__device__ __forceinline__ T fromf(float v);
template <>
__device__ __forceinline__ float fromf<float>(float v) { return v; }
template <>
__device__ __forceinline__ bf16 fromf<bf16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ int wrapc(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ void tap_offset(int t, int ntap, int& dx, int& dy, int& dz) {
  if (ntap == 27) {
    dx = t / 9 - 1;
    dy = (t / 3) % 3 - 1;
    dz = t % 3 - 1;
  } else {
    dx = dy = dz = 0;
  }
}

// Eight channels of one voxel as float32 (16-byte loads of bfloat16, two of float32).
__device__ __forceinline__ void load8(const bf16* p, float (&v)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
  v[4] = __uint_as_float(u.z << 16); v[5] = __uint_as_float(u.z & 0xffff0000u);
  v[6] = __uint_as_float(u.w << 16); v[7] = __uint_as_float(u.w & 0xffff0000u);
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// ---- convolution forward: y = act(b + conv(concat(xa, xb))) (+ res for the head) ----------------
// VPT voxels per thread (blockDim apart, so loads stay contiguous), all COUT channels of each in
// registers; the weights of TG taps at a time in shared memory, read as broadcasts shared by the
// thread's voxels; activations as 8-channel loads through the L1 (ca and cb multiples of 8; cin counts
// the channels of xa that have weights, ca its stride).  Per output the sum runs over the taps and,
// inside a tap, over the channels, one fused multiply-add each from the bias: the order that fixes
// which way a stored bfloat16 rounds.
template <typename T, int COUT>
struct ConvFwd {
  static constexpr int VPT = COUT >= 32 ? 1 : 2;
  static constexpr int TG = 3;
};
template <typename T, int COUT>
__global__ void __launch_bounds__(256) conv_fwd_kernel(const T* __restrict__ xa, int ca, int cina, int up,
                                                       const T* __restrict__ xb, int cb, const T* __restrict__ w,
                                                       const float* __restrict__ bias, int n, T* __restrict__ y) {
  constexpr int VPT = ConvFwd<T, COUT>::VPT, TG = ConvFwd<T, COUT>::TG;
  extern __shared__ float4 wsm4[];
  float* wsm = reinterpret_cast<float*>(wsm4);
  const int cin = cina + cb;
  const int nv = n * n * n;   // below 2^31 (ensure)
  float2 acc[VPT][COUT / 2];
  int vx[VPT], vy[VPT], vz[VPT], vv[VPT];
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    vv[k] = blockIdx.x * (256 * VPT) + k * 256 + threadIdx.x;
    const int v = vv[k] < nv ? vv[k] : 0;
    vx[k] = v / (n * n);
    vy[k] = (v / n) % n;
    vz[k] = v % n;
#pragma unroll
    for (int c = 0; c < COUT / 2; ++c) acc[k][c] = make_float2(bias[2 * c], bias[2 * c + 1]);
  }
  for (int t0 = 0; t0 < 27; t0 += TG) {
    __syncthreads();
    for (int e = threadIdx.x; e < TG * cin * COUT; e += 256) wsm[e] = tof(w[(size_t)t0 * cin * COUT + e]);
    __syncthreads();
    for (int tt = 0; tt < TG; ++tt) {
      int dx, dy, dz;
      tap_offset(t0 + tt, 27, dx, dy, dz);
      int u[VPT], ua[VPT];   // voxel in the fine grid, and in xa's (the coarse one: nearest upsampling)
#pragma unroll
      for (int k = 0; k < VPT; ++k) {
        const int x = wrapc(vx[k] + dx, n), y = wrapc(vy[k] + dy, n), z = wrapc(vz[k] + dz, n);
        u[k] = (x * n + y) * n + z;
        ua[k] = up ? ((x >> 1) * (n >> 1) + (y >> 1)) * (n >> 1) + (z >> 1) : u[k];
      }
      const float* wt = wsm + tt * cin * COUT;
      for (int c0 = 0; c0 < cin; c0 += 8) {
        float xv[VPT][8];
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
          if (c0 < cina) load8(xa + (size_t)ua[k] * ca + c0, xv[k]);
          else load8(xb + (size_t)u[k] * cb + (c0 - cina), xv[k]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (c0 + i < cin) {   // uniform
            const float4* w4 = reinterpret_cast<const float4*>(wt + (c0 + i) * COUT);
#pragma unroll
            for (int c = 0; c < COUT / 4; ++c) {
              const float4 ww = w4[c];
#pragma unroll
              for (int k = 0; k < VPT; ++k) {
                const float2 xx = make_float2(xv[k][i], xv[k][i]);
                acc[k][2 * c] = __ffma2_rn(xx, make_float2(ww.x, ww.y), acc[k][2 * c]);
                acc[k][2 * c + 1] = __ffma2_rn(xx, make_float2(ww.z, ww.w), acc[k][2 * c + 1]);
              }
            }
          }
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    if (vv[k] < nv) {
      T* o = y + (size_t)vv[k] * COUT;
#pragma unroll
      for (int c = 0; c < COUT; c += 8) {
        __align__(16) T t8[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          t8[2 * i] = fromf<T>(fmaxf(acc[k][c / 2 + i].x, 0.f));
          t8[2 * i + 1] = fromf<T>(fmaxf(acc[k][c / 2 + i].y, 0.f));
        }
#pragma unroll
        for (int b = 0; b < (int)sizeof(T) / 2; ++b)
          reinterpret_cast<uint4*>(o + c)[b] = reinterpret_cast<const uint4*>(t8)[b];
      }
    }
  }
}

// The 1x1x1 head: y = res + (b + sum_c x[c] w[c]).
template <typename T, int CIN>
__global__ void __launch_bounds__(256) head_fwd_kernel(const T* __restrict__ x, const T* __restrict__ w,
                                                       const float* __restrict__ bias, const float* __restrict__ res,
                                                       int res_stride, long long nv, float* __restrict__ y) {
  const long long v = (long long)blockIdx.x * 256 + threadIdx.x;
  if (v >= nv) return;
  float acc = bias[0];
#pragma unroll
  for (int c0 = 0; c0 < CIN; c0 += 8) {
    float xv[8];
    load8(x + v * CIN + c0, xv);
#pragma unroll
    for (int i = 0; i < 8; ++i) acc = fmaf(xv[i], tof(w[c0 + i]), acc);
  }
  y[v] = acc + res[v * res_stride];
}

// ---- tiles of the backward convolutions: 4 x 4 x 32 voxels with a halo of one --------------------
constexpr int kBX = 4, kBY = 4, kBZ = 32;
constexpr int kHX = kBX + 2, kHY = kBY + 2, kHZ = kBZ + 2;
struct TileGrid {
  int nx, ny, nz;
  __host__ __device__ explicit TileGrid(int n)
      : nx((n + kBX - 1) / kBX), ny((n + kBY - 1) / kBY), nz((n + kBZ - 1) / kBZ) {}
  __host__ __device__ int count() const { return nx * ny * nz; }
  __device__ void origin(int t, int& x, int& y, int& z) const {
    z = (t % nz) * kBZ;
    y = (t / nz) % ny * kBY;
    x = t / (nz * ny) * kBX;
  }
};
__device__ __forceinline__ int wrapm(int i, int n) { return ((i % n) + n) % n; }   // any i: tiles may pass the grid

// ---- gradient w.r.t. the input: gx[v][ci] = sum_t sum_co gy[v - d(t)][co] w[t][ci][co] ---------
// A block of 128 threads owns one tile and 8 input channels, a thread 4 voxels along z (32 sums).
// Per 8 output channels it stages gy's halo as float4 planes (4 channels a plane; z skewed by one
// word in four, so the eight z runs of a quarter warp read distinct banks) and the 27 x 8 x 8 weights
// (read as broadcasts).  A thread slides over z: six staged positions serve three taps of four voxels,
// 384 multiply-adds per 30 shared loads.  The one-voxel-per-thread form spent its time on its loads:
// 6.6 ms of a 128^3 training step for what is 1.2 ms of multiply-adds.
// With mask the result is zeroed where the activation mask (same layout) is not positive (the ReLU).
constexpr int kDZ = kHZ + (kHZ >> 2);
constexpr int kDPlane = kHX * kHY * kDZ;
template <typename T>
__global__ void __launch_bounds__(128) conv_dgrad_kernel(const float* __restrict__ gy, int cout,
                                                         const T* __restrict__ w, int ca, int cb, int n,
                                                         float* __restrict__ gxa, float* __restrict__ gxb,
                                                         const T* __restrict__ mask) {
  extern __shared__ float4 dsm[];
  float4* pl = dsm;                                           // [2][kHX][kHY][kDZ]
  float* ws = reinterpret_cast<float*>(dsm + 2 * kDPlane);    // [27][8 co][8 ci], taps reversed
  const int cin = ca + cb, c0 = blockIdx.y * 8;
  const TileGrid tg(n);
  int X, Y, Z;
  tg.origin(blockIdx.x, X, Y, Z);
  const int run = threadIdx.x & 7, ty = (threadIdx.x >> 3) & 3, tx = threadIdx.x >> 5;
  float2 acc[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[k][c] = make_float2(0.f, 0.f);
  for (int o0 = 0; o0 < cout; o0 += 8) {
    __syncthreads();
    for (int e = threadIdx.x; e < kHX * kHY * kHZ; e += 128) {
      const int hz = e % kHZ, hy = (e / kHZ) % kHY, hx = e / (kHZ * kHY);
      const int u = (wrapm(X + hx - 1, n) * n + wrapm(Y + hy - 1, n)) * n + wrapm(Z + hz - 1, n);
      const float4* g = reinterpret_cast<const float4*>(gy + (size_t)u * cout + o0);
      const int p = (hx * kHY + hy) * kDZ + hz + (hz >> 2);
      pl[p] = g[0];
      pl[kDPlane + p] = g[1];
    }
    for (int e = threadIdx.x; e < 27 * 64; e += 128) {
      const int ci = e & 7, co = (e >> 3) & 7, t = e >> 6;
      ws[e] = tof(w[((size_t)(26 - t) * cin + c0 + ci) * cout + o0 + co]);
    }
    __syncthreads();
#pragma unroll 1
    for (int dxy = 0; dxy < 9; ++dxy) {
      const int p0 = ((tx + dxy / 3) * kHY + ty + dxy % 3) * kDZ + 5 * run;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4 g[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) g[k] = pl[h * kDPlane + p0 + k + (k >> 2)];
#pragma unroll
        for (int dz = 0; dz < 3; ++dz) {
          const float4* w4 = reinterpret_cast<const float4*>(ws + ((dxy * 3 + dz) * 8 + 4 * h) * 8);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 wa = w4[2 * i], wb = w4[2 * i + 1];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 gv = g[k + dz];
              const float s = i == 0 ? gv.x : (i == 1 ? gv.y : (i == 2 ? gv.z : gv.w));
              const float2 ss = make_float2(s, s);
              acc[k][0] = __ffma2_rn(ss, make_float2(wa.x, wa.y), acc[k][0]);
              acc[k][1] = __ffma2_rn(ss, make_float2(wa.z, wa.w), acc[k][1]);
              acc[k][2] = __ffma2_rn(ss, make_float2(wb.x, wb.y), acc[k][2]);
              acc[k][3] = __ffma2_rn(ss, make_float2(wb.z, wb.w), acc[k][3]);
            }
          }
        }
      }
    }
  }
  const int x = X + tx, y = Y + ty;
  if (x >= n || y >= n) return;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int z = Z + 4 * run + k;
    if (z < n) {
      const size_t v = ((size_t)x * n + y) * n + z;
      if (mask) {
        float mv[8];
        load8(mask + v * ca + c0, mv);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (!(mv[2 * c] > 0.f)) acc[k][c].x = 0.f;
          if (!(mv[2 * c + 1] > 0.f)) acc[k][c].y = 0.f;
        }
      }
      float4* o = reinterpret_cast<float4*>(c0 < ca ? gxa + v * ca + c0 : gxb + v * cb + (c0 - ca));
      o[0] = make_float4(acc[k][0].x, acc[k][0].y, acc[k][1].x, acc[k][1].y);
      o[1] = make_float4(acc[k][2].x, acc[k][2].y, acc[k][3].x, acc[k][3].y);
    }
  }
}
constexpr size_t kDSmem = 2 * kDPlane * sizeof(float4) + 27 * 64 * sizeof(float);

// ---- gradients w.r.t. the weights and the bias: gw[t][ci][co] += sum_v x[v + d(t)][ci] gy[v][co] ----
// A block owns one group of 8 input and one of 8 output channels (blockIdx.y) and walks over tiles.
// Lane t < 27 of every warp is a tap and holds its 8 x 8 sums; the warp's lanes read the same gy
// voxel (a broadcast) and their own shifted x voxel, one 16-byte load each for 64 multiply-adds (row
// and plane strides of 3 and 1 mod 8 units put any eight consecutive taps in distinct banks).  Lane 27
// multiplies by one instead: the bias gradient.  The 8 warps take the tile's rows and are summed at
// the end, one atomic per block and weight.  The form before (one weight per thread and pass, both
// factors reloaded from shared memory for every multiply-add) took 40 of a step's 52 ms.
constexpr int kWRow = 35, kWPlane = 217;                     // voxel strides of the staged x (units of 8 channels)
template <typename T>
__global__ void __launch_bounds__(256, 2) conv_wgrad_kernel(const T* __restrict__ xa, int ca, int cina, int up,
                                                            const T* __restrict__ xb, int cb,
                                                            const float* __restrict__ gy, int cout, int n,
                                                            float* __restrict__ gw, float* __restrict__ gb) {
  constexpr int U = (int)sizeof(T) / 2;                      // 16-byte units per 8 channels
  extern __shared__ float4 gsm[];
  uint4* xs = reinterpret_cast<uint4*>(gsm);                 // [U][kHX][kHY][kHZ] (padded strides)
  float4* gs = gsm + U * kHX * kWPlane;                      // [512][2]
  const int cin = cina + cb, og = cout / 8;
  const int cg = blockIdx.y / og, o0 = (blockIdx.y % og) * 8, c0 = cg * 8;
  const bool from_a = c0 < cina;
  const T* src = from_a ? xa + c0 : xb + (c0 - cina);
  const int cs = from_a ? ca : cb, sh = from_a ? up : 0, m = n >> sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = lane < 27 ? lane : 26;
  const int toff = (t / 9) * kWPlane + (t / 3 % 3) * kWRow + t % 3;
  const bool ones = lane == 27;
  const TileGrid tg(n);
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = make_float2(0.f, 0.f);
  for (int tile = blockIdx.x; tile < tg.count(); tile += gridDim.x) {
    int X, Y, Z;
    tg.origin(tile, X, Y, Z);
    __syncthreads();
    for (int e = threadIdx.x; e < kHX * kHY * kHZ; e += 256) {
      const int hz = e % kHZ, hy = (e / kHZ) % kHY, hx = e / (kHZ * kHY);
      const int x = wrapm(X + hx - 1, n) >> sh, y = wrapm(Y + hy - 1, n) >> sh, z = wrapm(Z + hz - 1, n) >> sh;
      const uint4* p = reinterpret_cast<const uint4*>(src + (size_t)((x * m + y) * m + z) * cs);
#pragma unroll
      for (int b = 0; b < U; ++b) xs[b * kHX * kWPlane + hx * kWPlane + hy * kWRow + hz] = p[b];
    }
    for (int e = threadIdx.x; e < kBX * kBY * kBZ; e += 256) {
      const int z = Z + e % kBZ, y = Y + (e / kBZ) % kBY, x = X + e / (kBZ * kBY);
      float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;   // voxels past the grid add nothing
      if (x < n && y < n && z < n) {
        const float4* g = reinterpret_cast<const float4*>(gy + ((size_t)(x * n + y) * n + z) * cout + o0);
        g0 = g[0];
        g1 = g[1];
      }
      gs[2 * e] = g0;
      gs[2 * e + 1] = g1;
    }
    __syncthreads();
    for (int row = warp; row < kBX * kBY; row += 8) {
      const uint4* xr = xs + (row / kBY) * kWPlane + (row % kBY) * kWRow + toff;
      const float4* gr = gs + 2 * row * kBZ;
#pragma unroll 4
      for (int z = 0; z < kBZ; ++z) {
        float xv[8];
        if (U == 1) {
          const uint4 q = xr[z];
          xv[0] = __uint_as_float(q.x << 16); xv[1] = __uint_as_float(q.x & 0xffff0000u);
          xv[2] = __uint_as_float(q.y << 16); xv[3] = __uint_as_float(q.y & 0xffff0000u);
          xv[4] = __uint_as_float(q.z << 16); xv[5] = __uint_as_float(q.z & 0xffff0000u);
          xv[6] = __uint_as_float(q.w << 16); xv[7] = __uint_as_float(q.w & 0xffff0000u);
        } else {
          const uint4 q = xr[z], q2 = xr[z + (U - 1) * kHX * kWPlane];
          xv[0] = __uint_as_float(q.x); xv[1] = __uint_as_float(q.y); xv[2] = __uint_as_float(q.z); xv[3] = __uint_as_float(q.w);
          xv[4] = __uint_as_float(q2.x); xv[5] = __uint_as_float(q2.y); xv[6] = __uint_as_float(q2.z); xv[7] = __uint_as_float(q2.w);
        }
        if (ones) xv[0] = 1.f;
        const float4 ga = gr[2 * z], gc = gr[2 * z + 1];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float2 xx = make_float2(xv[i], xv[i]);
          acc[i][0] = __ffma2_rn(xx, make_float2(ga.x, ga.y), acc[i][0]);
          acc[i][1] = __ffma2_rn(xx, make_float2(ga.z, ga.w), acc[i][1]);
          acc[i][2] = __ffma2_rn(xx, make_float2(gc.x, gc.y), acc[i][2]);
          acc[i][3] = __ffma2_rn(xx, make_float2(gc.z, gc.w), acc[i][3]);
        }
      }
    }
  }
  __syncthreads();
  float* red = reinterpret_cast<float*>(gsm);                // [28][64], padded to 65
  for (int k = 0; k < 8; ++k) {
    if (warp == k && lane < 28) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float* d = red + lane * 65 + 8 * i + 2 * c;
          d[0] = k ? d[0] + acc[i][c].x : acc[i][c].x;
          d[1] = k ? d[1] + acc[i][c].y : acc[i][c].y;
        }
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < 28 * 64; e += 256) {
    const int tt = e >> 6, i = (e >> 3) & 7, c = e & 7;
    const float v = red[tt * 65 + (e & 63)];
    if (tt < 27) {
      if (c0 + i < cin) atomicAdd(gw + ((size_t)tt * cin + c0 + i) * cout + o0 + c, v);
    } else if (cg == 0 && i == 0) {
      atomicAdd(gb + o0 + c, v);
    }
  }
}
template <typename T>
constexpr size_t wgrad_smem() {
  return (size_t)(sizeof(T) / 2) * kHX * kWPlane * 16 + (size_t)kBX * kBY * kBZ * 32;
}

// ---- loss and head backward in one pass: d = y - t, loss += d^2 / m, g = 2 d / m; the head's weight and
// bias gradients; gd = g w masked by the ReLU of its input --------------------------------------------
template <typename T, int CIN>
__global__ void __launch_bounds__(256) head_back_kernel(const float* __restrict__ y, const float* __restrict__ t,
                                                        const T* __restrict__ x, const T* __restrict__ w, long long m,
                                                        float* __restrict__ gx, float* __restrict__ gw,
                                                        float* __restrict__ gb, double* __restrict__ loss) {
  double s = 0.0;
  const float sc = 2.f / (float)m;
  float aw[CIN], ab = 0.f, wv[CIN];
#pragma unroll
  for (int c = 0; c < CIN; ++c) {
    aw[c] = 0.f;
    wv[c] = tof(w[c]);
  }
  for (long long v = (long long)blockIdx.x * 256 + threadIdx.x; v < m; v += (long long)gridDim.x * 256) {
    const float d = y[v] - t[v], g = sc * d;
    s += (double)d * d;
    ab += g;
#pragma unroll
    for (int c0 = 0; c0 < CIN; c0 += 8) {
      float xv[8];
      load8(x + v * CIN + c0, xv);
      float o[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        aw[c0 + i] = fmaf(xv[i], g, aw[c0 + i]);
        o[i] = xv[i] > 0.f ? g * wv[c0 + i] : 0.f;
      }
      float4* p = reinterpret_cast<float4*>(gx + v * CIN + c0);
      p[0] = make_float4(o[0], o[1], o[2], o[3]);
      p[1] = make_float4(o[4], o[5], o[6], o[7]);
    }
  }
  __shared__ double sh[8];
  __shared__ float shf[8][CIN + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    ab += __shfl_down_sync(0xffffffffu, ab, o);
#pragma unroll
    for (int c = 0; c < CIN; ++c) aw[c] += __shfl_down_sync(0xffffffffu, aw[c], o);
  }
  if (lane == 0) {
    sh[warp] = s;
    shf[warp][CIN] = ab;
#pragma unroll
    for (int c = 0; c < CIN; ++c) shf[warp][c] = aw[c];
  }
  __syncthreads();
  if (threadIdx.x <= CIN) {
    float r = 0.f;
    for (int k = 0; k < 8; ++k) r += shf[k][threadIdx.x];
    atomicAdd(threadIdx.x < CIN ? gw + threadIdx.x : gb, r);
  }
  if (threadIdx.x == 32) {
    double r = 0.0;
    for (int k = 0; k < 8; ++k) r += sh[k];
    atomicAdd(loss, r / (double)m);
  }
}

// 2x2x2 average pooling: coarse n/2 grid
template <typename T>
__global__ void pool_kernel(const T* __restrict__ x, int c, int n, T* __restrict__ y) {
  const int m = n / 2;
  const long long tot = (long long)m * m * m * c;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
    const int ch = (int)(i % c);
    const long long cv = i / c;
    const int X = (int)(cv / ((long long)m * m)), Y = (int)((cv / m) % m), Z = (int)(cv % m);
    float s = 0.f;
    for (int a = 0; a < 8; ++a) {
      const long long f = ((long long)(2 * X + (a >> 2)) * n + (2 * Y + ((a >> 1) & 1))) * n + (2 * Z + (a & 1));
      s += tof(x[f * c + ch]);
    }
    y[i] = fromf<T>(0.125f * s);
  }
}

// gx += pooled gradient / 8, then the ReLU of the pooled activation (c a multiple of 4)
template <typename T>
__global__ void pool_backward_kernel(const float* __restrict__ g, int c, int n, float* __restrict__ gx,
                                     const T* __restrict__ mask) {
  const int m = n / 2, c4 = c / 4;
  const long long tot = (long long)n * n * n * c4;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
    const int ch = (int)(i % c4);
    const int f = (int)(i / c4), x = f / (n * n), y = (f / n) % n, z = f % n;
    const float4 p = reinterpret_cast<const float4*>(g)[(((long long)(x >> 1) * m + (y >> 1)) * m + (z >> 1)) * c4 + ch];
    float4 v = reinterpret_cast<const float4*>(gx)[i];
    v = make_float4(v.x + 0.125f * p.x, v.y + 0.125f * p.y, v.z + 0.125f * p.z, v.w + 0.125f * p.w);
    const T* k = mask + 4 * i;
    if (!(tof(k[0]) > 0.f)) v.x = 0.f;
    if (!(tof(k[1]) > 0.f)) v.y = 0.f;
    if (!(tof(k[2]) > 0.f)) v.z = 0.f;
    if (!(tof(k[3]) > 0.f)) v.w = 0.f;
    reinterpret_cast<float4*>(gx)[i] = v;
  }
}

// sum over the 8 upsampled copies, then the ReLU of the coarse activation (c a multiple of 4)
template <typename T>
__global__ void up_backward_kernel(const float* __restrict__ g, int c, int n, float* __restrict__ gx,
                                   const T* __restrict__ mask) {
  const int m = n / 2, c4 = c / 4;
  const long long tot = (long long)m * m * m * c4;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
    const int ch = (int)(i % c4);
    const int cv = (int)(i / c4), X = cv / (m * m), Y = (cv / m) % m, Z = cv % m;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const long long f = ((long long)(2 * X + (a >> 2)) * n + (2 * Y + ((a >> 1) & 1))) * n + (2 * Z + (a & 1));
      const float4 p = reinterpret_cast<const float4*>(g)[f * c4 + ch];
      s = make_float4(s.x + p.x, s.y + p.y, s.z + p.z, s.w + p.w);
    }
    const T* k = mask + 4 * i;
    if (!(tof(k[0]) > 0.f)) s.x = 0.f;
    if (!(tof(k[1]) > 0.f)) s.y = 0.f;
    if (!(tof(k[2]) > 0.f)) s.z = 0.f;
    if (!(tof(k[3]) > 0.f)) s.w = 0.f;
    reinterpret_cast<float4*>(gx)[i] = s;
  }
}

template <typename T>
__global__ void to_t_kernel(const float* __restrict__ x, T* __restrict__ y, long long m) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (long long)gridDim.x * blockDim.x)
    y[i] = fromf<T>(x[i]);
}

// network input: 5 float32 channels -> 8 stored channels a voxel, the last ones zero
template <typename T>
__global__ void to_x8_kernel(const float* __restrict__ x, int cin, long long nv, T* __restrict__ y) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += (long long)gridDim.x * blockDim.x) {
    __align__(16) T o[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) o[c] = fromf<T>(c < cin ? x[v * cin + c] : 0.f);
#pragma unroll
    for (int b = 0; b < (int)sizeof(T) / 2; ++b)
      reinterpret_cast<uint4*>(y + v * 8)[b] = reinterpret_cast<const uint4*>(o)[b];
  }
}

// decoupled weight decay Adam on the float32 master weights; refreshes the stored-type copy
template <typename T>
__global__ void adamw_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                             float* __restrict__ m2, const unsigned char* __restrict__ decay, T* __restrict__ pt,
                             long long np, float lr, float wd, float c1, float c2) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = 0.9f * m1[i] + 0.1f * gi;
    const float b = 0.999f * m2[i] + 0.001f * gi * gi;
    m1[i] = a;
    m2[i] = b;
    float w = p[i] - lr * ((a / c1) / (sqrtf(b / c2) + 1e-8f) + (decay[i] ? wd * p[i] : 0.f));
    p[i] = w;
    pt[i] = fromf<T>(w);
  }
}

int grid_for(long long m, int threads = 256) {
  long long b = (m + threads - 1) / threads;
  return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

struct Spec {
  const char* name;
  int cin, cout, ntap;
};

}  // namespace
}  // namespace rg

using namespace rg;

struct recon_unet {
  int c1 = 16, cin = 5, bf16 = 1, n_alloc = 0, step = 0;
  cudaStream_t st = nullptr;
  std::vector<Spec> spec;
  std::vector<size_t> woff, boff;
  size_t np = 0;
  float *p = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;
  unsigned char* decay = nullptr;
  void* pt = nullptr;                  // stored-type copy of the parameters
  void* acts = nullptr;                // activations (stored type) for n_alloc
  float* grads = nullptr;              // activation gradients for n_alloc
  float* y = nullptr;                  // network output (float)
  double* loss = nullptr;
  std::string err;
  // tensor-core forward
  int use_tc = 1;
  int* dev_err = nullptr;              // set by a tensor-core kernel whose wait timed out
  void* wpack = nullptr;               // packed weight tiles of the layers on the tensor-core path
  size_t wpack_cap = 0;
  rg::tc::ConvPlan plan[10];
  bool plan_ok[10] = {};
  size_t pack_off[10] = {};
  int plan_n = 0;
  unsigned pver = 1, packed_ver = 0;   // parameter version, version the packed tiles were made from
  int last_n = 0;                      // side of the last forward
  long long launches = 0;              // kernels launched by recon_unet_forward (all calls)
  bool head_fused = false;             // last forward fused the head into layer 9 (d1b not stored)
};

namespace {

void make_spec(recon_unet* u) {
  const int c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1, ci = u->cin;
  u->spec = {{"enc1a", ci, c1, 27}, {"enc1b", c1, c1, 27}, {"enc2a", c1, c2, 27}, {"enc2b", c2, c2, 27},
             {"bota", c2, c3, 27},  {"botb", c3, c3, 27},  {"dec2a", c3 + c2, c2, 27}, {"dec2b", c2, c2, 27},
             {"dec1a", c2 + c1, c1, 27}, {"dec1b", c1, c1, 27}, {"head", c1, 1, 1}};
  u->woff.clear();
  u->boff.clear();
  size_t o = 0;
  for (auto& s : u->spec) {
    u->woff.push_back(o);
    o += (size_t)s.ntap * s.cin * s.cout;
    u->boff.push_back(o);
    o += s.cout;
  }
  u->np = o;
}

// activation layout for one grid of side n (offsets in elements of the stored type)
struct Acts {
  size_t a1a, a1b, p1, a2a, a2b, p2, a3a, a3b, d2a, d2b, d1a, d1b, x8, total;
};
Acts act_layout(const recon_unet* u, int n) {
  const size_t V1 = (size_t)n * n * n, V2 = V1 / 8, V3 = V1 / 64;
  const size_t c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1;
  Acts a{};
  size_t o = 0;
  auto take = [&](size_t k) { size_t r = o; o += (k + 127) & ~(size_t)127; return r; };
  a.a1a = take(V1 * c1); a.a1b = take(V1 * c1); a.p1 = take(V2 * c1);
  a.a2a = take(V2 * c2); a.a2b = take(V2 * c2); a.p2 = take(V3 * c2);
  a.a3a = take(V3 * c3); a.a3b = take(V3 * c3);
  a.d2a = take(V2 * c2); a.d2b = take(V2 * c2);
  a.d1a = take(V1 * c1); a.d1b = take(V1 * c1);
  a.x8 = take(V1 * 8);
  a.total = o;
  return a;
}
struct Grads {
  size_t gd1b, gd1a, gu2, gs1, gd2b, gd2a, gu3, gs2, ga3b, ga3a, gp2, ga2a, gp1, ga1a, total;
};
Grads grad_layout(const recon_unet* u, int n) {
  const size_t V1 = (size_t)n * n * n, V2 = V1 / 8, V3 = V1 / 64;
  const size_t c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1;
  Grads g{};
  size_t o = 0;
  auto take = [&](size_t k) { size_t r = o; o += (k + 63) & ~(size_t)63; return r; };
  g.gd1b = take(V1 * c1); g.gd1a = take(V1 * c1); g.gu2 = take(V1 * c2); g.gs1 = take(V1 * c1);
  g.gd2b = take(V2 * c2); g.gd2a = take(V2 * c2); g.gu3 = take(V2 * c3); g.gs2 = take(V2 * c2);
  g.ga3b = take(V3 * c3); g.ga3a = take(V3 * c3); g.gp2 = take(V3 * c2); g.ga2a = take(V2 * c2);
  g.gp1 = take(V2 * c1); g.ga1a = take(V1 * c1);
  g.total = o;
  return g;
}

#define UN_CUDA(call)                                                   \
  do {                                                                  \
    cudaError_t e_ = (call);                                            \
    if (e_ != cudaSuccess) {                                            \
      u->err = std::string(#call) + ": " + cudaGetErrorString(e_);      \
      return RECON_ERR_CUDA;                                            \
    }                                                                   \
  } while (0)

recon_status ensure(recon_unet* u, int n, bool train) {
  if (n < 8 || n % 8 != 0) return RECON_ERR_INVALID_ARG;
  // The layers index voxels in 32 bits.  Only the narrowest network's inference at sides 1296 to 1312 would fit
  // 288 GB beyond that.
  if ((long long)n * n * n > INT_MAX) return RECON_ERR_OOM;
  if (n <= u->n_alloc && (!train || u->grads)) return RECON_OK;
  const int nn = n > u->n_alloc ? n : u->n_alloc;
  if (u->acts) cudaFree(u->acts);
  if (u->grads) cudaFree(u->grads);
  if (u->y) cudaFree(u->y);
  u->acts = nullptr;
  u->grads = nullptr;
  u->y = nullptr;
  u->n_alloc = 0;   // until all of them are there: a call after one that ran out of memory allocates again
  const size_t es = u->bf16 ? 2 : 4;
  if (cudaMalloc(&u->acts, act_layout(u, nn).total * es) != cudaSuccess ||
      cudaMalloc(&u->y, (size_t)nn * nn * nn * sizeof(float)) != cudaSuccess ||
      (train && cudaMalloc(&u->grads, grad_layout(u, nn).total * sizeof(float)) != cudaSuccess)) {
    cudaGetLastError();
    return RECON_ERR_OOM;
  }
  u->n_alloc = nn;
  return RECON_OK;
}

// One 3x3x3 layer on the CUDA cores: xa holds ca channels a voxel, cina of them with weights; up: xa is
// read from the coarse grid of half the side (nearest upsampling).
template <typename T>
cudaError_t conv_fwd(recon_unet* u, int li, const T* xa, int ca, int cina, int up, const T* xb, int cb, int n, T* y) {
  const Spec& s = u->spec[li];
  const T* w = static_cast<const T*>(u->pt) + u->woff[li];
  const float* b = u->p + u->boff[li];
  const long long nv = (long long)n * n * n;
  cudaError_t e = cudaSuccess;
  switch (s.cout) {
#define UN_CASE(C)                                                                                              \
  case C: {                                                                                                     \
    using F = ConvFwd<T, C>;                                                                                    \
    const size_t smem = sizeof(float) * F::TG * s.cin * C;                                                      \
    e = cudaFuncSetAttribute((const void*)conv_fwd_kernel<T, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    if (e != cudaSuccess) return e;                                                                             \
    conv_fwd_kernel<T, C><<<(unsigned)((nv + 256 * F::VPT - 1) / (256 * F::VPT)), 256, smem, u->st>>>(          \
        xa, ca, cina, up, xb, cb, w, b, n, y);                                                                      \
    break;                                                                                                      \
  }
    UN_CASE(8) UN_CASE(16) UN_CASE(32) UN_CASE(64)
#undef UN_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t head_fwd(recon_unet* u, const T* x, const float* res, int res_stride, int n, float* y) {
  const T* w = static_cast<const T*>(u->pt) + u->woff[10];
  const float* b = u->p + u->boff[10];
  const long long nv = (long long)n * n * n;
  const unsigned blocks = (unsigned)((nv + 255) / 256);
  if (u->c1 == 8) head_fwd_kernel<T, 8><<<blocks, 256, 0, u->st>>>(x, w, b, res, res_stride, nv, y);
  else head_fwd_kernel<T, 16><<<blocks, 256, 0, u->st>>>(x, w, b, res, res_stride, nv, y);
  return cudaGetLastError();
}

// Gradients of one 3x3x3 layer: weights and bias, and (gxa, gxb not null) its inputs.  up: xa is read
// from the coarse grid of half the side (nearest upsampling).
template <typename T>
cudaError_t conv_back(recon_unet* u, int li, const T* xa, int ca, int cina, int up, const T* xb, int cb, const float* gy,
                      int n, float* gxa, float* gxb, const T* mask) {
  const Spec& s = u->spec[li];
  const T* w = static_cast<const T*>(u->pt) + u->woff[li];
  const int tiles = TileGrid(n).count();
  cudaError_t e = cudaFuncSetAttribute((const void*)conv_wgrad_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)wgrad_smem<T>());
  if (e != cudaSuccess) return e;
  const int groups = ((s.cin + 7) / 8) * (s.cout / 8);
  // two blocks per SM over all channel groups together, at least one tile each
  int per = (2 * 152 + groups - 1) / groups;
  if (per > tiles) per = tiles;
  conv_wgrad_kernel<T><<<dim3(per, groups), 256, wgrad_smem<T>(), u->st>>>(xa, ca, cina, up, xb, cb, gy, s.cout, n,
                                                                          u->g + u->woff[li], u->g + u->boff[li]);
  if (gxa) {
    e = cudaFuncSetAttribute((const void*)conv_dgrad_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDSmem);
    if (e != cudaSuccess) return e;
    conv_dgrad_kernel<T><<<dim3(tiles, s.cin / 8), 128, kDSmem, u->st>>>(gy, s.cout, w, ca, cb, n, gxa, gxb, mask);
  }
  return cudaGetLastError();
}

template <typename T>
recon_status forward_t(recon_unet* u, const float* x, int n, float* out) {
  const Acts A = act_layout(u, n);
  T* a = static_cast<T*>(u->acts);
  const int c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1, n2 = n / 2, n4 = n / 4;
  const long long V1 = (long long)n * n * n;
  to_x8_kernel<T><<<grid_for(V1), 256, 0, u->st>>>(x, u->cin, V1, a + A.x8);
  UN_CUDA(conv_fwd<T>(u, 0, a + A.x8, 8, u->cin, 0, nullptr, 0, n, a + A.a1a));
  UN_CUDA(conv_fwd<T>(u, 1, a + A.a1a, c1, c1, 0, nullptr, 0, n, a + A.a1b));
  pool_kernel<T><<<grid_for(V1 / 8 * c1), 256, 0, u->st>>>(a + A.a1b, c1, n, a + A.p1);
  UN_CUDA(conv_fwd<T>(u, 2, a + A.p1, c1, c1, 0, nullptr, 0, n2, a + A.a2a));
  UN_CUDA(conv_fwd<T>(u, 3, a + A.a2a, c2, c2, 0, nullptr, 0, n2, a + A.a2b));
  pool_kernel<T><<<grid_for(V1 / 64 * c2), 256, 0, u->st>>>(a + A.a2b, c2, n2, a + A.p2);
  UN_CUDA(conv_fwd<T>(u, 4, a + A.p2, c2, c2, 0, nullptr, 0, n4, a + A.a3a));
  UN_CUDA(conv_fwd<T>(u, 5, a + A.a3a, c3, c3, 0, nullptr, 0, n4, a + A.a3b));
  UN_CUDA(conv_fwd<T>(u, 6, a + A.a3b, c3, c3, 1, a + A.a2b, c2, n2, a + A.d2a));
  UN_CUDA(conv_fwd<T>(u, 7, a + A.d2a, c2, c2, 0, nullptr, 0, n2, a + A.d2b));
  UN_CUDA(conv_fwd<T>(u, 8, a + A.d2b, c2, c2, 1, a + A.a1b, c1, n, a + A.d1a));
  UN_CUDA(conv_fwd<T>(u, 9, a + A.d1a, c1, c1, 0, nullptr, 0, n, a + A.d1b));
  UN_CUDA(head_fwd<T>(u, a + A.d1b, x + (u->cin - 1), u->cin, n, out));
  return RECON_OK;
}

// Tensor-core plans for the ten 3x3x3 layers at grid side n (levels n, n/2, n/4), and the packed
// weight tiles; a layer whose level does not fit the tensor-core tiling stays on the CUDA cores.
recon_status tc_prepare(recon_unet* u, int n) {
  const int c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1, n2 = n / 2, n4 = n / 4;
  if (u->plan_n != n) {
    struct L {
      int n, c0, up0, c1, cin, cout;
    };
    const L ls[10] = {{n, 8, 0, 0, u->cin, c1},      {n, c1, 0, 0, c1, c1},         {n2, c1, 0, 0, c1, c2},
                      {n2, c2, 0, 0, c2, c2},        {n4, c2, 0, 0, c2, c3},        {n4, c3, 0, 0, c3, c3},
                      {n2, c3, 1, c2, c3 + c2, c2},  {n2, c2, 0, 0, c2, c2},        {n, c2, 1, c1, c2 + c1, c1},
                      {n, c1, 0, 0, c1, c1}};
    size_t off = 0;
    for (int l = 0; l < 10; ++l) {
      u->plan_ok[l] = tc::plan_conv(ls[l].n, ls[l].c0, ls[l].up0, ls[l].c1, ls[l].cin, ls[l].cout, &u->plan[l]);
      u->pack_off[l] = off;
      if (u->plan_ok[l]) off += (u->plan[l].packed_elems + 127) / 128 * 128;
    }
    if (off * sizeof(bf16) > u->wpack_cap) {
      cudaFree(u->wpack);
      u->wpack = nullptr;
      u->wpack_cap = 0;
      if (cudaMalloc(&u->wpack, off * sizeof(bf16)) != cudaSuccess) {
        cudaGetLastError();
        u->plan_n = 0;
        return RECON_ERR_OOM;
      }
      u->wpack_cap = off * sizeof(bf16);
    }
    u->plan_n = n;
    u->packed_ver = 0;
  }
  if (u->packed_ver != u->pver) {
    const bf16* w = static_cast<const bf16*>(u->pt);
    for (int l = 0; l < 10; ++l)
      if (u->plan_ok[l]) {
        ++u->launches;
        UN_CUDA(tc::pack_weights(u->plan[l], w + u->woff[l], static_cast<bf16*>(u->wpack) + u->pack_off[l], u->st));
      }
    u->packed_ver = u->pver;
  }
  return RECON_OK;
}

// Inference forward with bf16 storage: the same network and rounding points as forward_t<bf16>,
// with the convolutions on the tensor cores where the level allows, the upsampling folded into the
// loads of the decoder convolutions and the 1x1 head folded into the last convolution.
recon_status forward_tc(recon_unet* u, const float* x, int n, float* out) {
  recon_status rs = tc_prepare(u, n);
  if (rs != RECON_OK) return rs;
  const Acts A = act_layout(u, n);
  bf16* a = static_cast<bf16*>(u->acts);
  const bf16* wp = static_cast<const bf16*>(u->wpack);
  const int c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1, n2 = n / 2, n4 = n / 4;
  const long long V1 = (long long)n * n * n;
  auto run = [&](int l, const bf16* s0, const bf16* s1, bf16* y) -> cudaError_t {
    ++u->launches;
    tc::ConvIO io;
    io.src0 = s0;
    io.src1 = s1;
    io.wpack = wp + u->pack_off[l];
    io.bias = u->p + u->boff[l];
    io.out = y;
    io.err = u->dev_err;
    return tc::conv_forward(u->plan[l], io, u->st);
  };
  auto plain = [&](int l, const bf16* s0, int ca, bf16* y, int nl) -> cudaError_t {
    if (u->plan_ok[l]) return run(l, s0, nullptr, y);
    ++u->launches;
    return conv_fwd<bf16>(u, l, s0, ca, ca, 0, nullptr, 0, nl, y);
  };
  u->launches += 3;   // input conversion and the two poolings
  to_x8_kernel<bf16><<<grid_for(V1), 256, 0, u->st>>>(x, u->cin, V1, a + A.x8);
  if (u->plan_ok[0]) UN_CUDA(run(0, a + A.x8, nullptr, a + A.a1a));
  else UN_CUDA(conv_fwd<bf16>(u, 0, a + A.x8, 8, u->cin, 0, nullptr, 0, n, a + A.a1a));
  UN_CUDA(plain(1, a + A.a1a, c1, a + A.a1b, n));
  pool_kernel<bf16><<<grid_for(V1 / 8 * c1), 256, 0, u->st>>>(a + A.a1b, c1, n, a + A.p1);
  UN_CUDA(plain(2, a + A.p1, c1, a + A.a2a, n2));
  UN_CUDA(plain(3, a + A.a2a, c2, a + A.a2b, n2));
  pool_kernel<bf16><<<grid_for(V1 / 64 * c2), 256, 0, u->st>>>(a + A.a2b, c2, n2, a + A.p2);
  UN_CUDA(plain(4, a + A.p2, c2, a + A.a3a, n4));
  UN_CUDA(plain(5, a + A.a3a, c3, a + A.a3b, n4));
  if (u->plan_ok[6]) {
    UN_CUDA(run(6, a + A.a3b, a + A.a2b, a + A.d2a));
  } else {
    ++u->launches;
    UN_CUDA(conv_fwd<bf16>(u, 6, a + A.a3b, c3, c3, 1, a + A.a2b, c2, n2, a + A.d2a));
  }
  UN_CUDA(plain(7, a + A.d2a, c2, a + A.d2b, n2));
  if (u->plan_ok[8]) {
    UN_CUDA(run(8, a + A.d2b, a + A.a1b, a + A.d1a));
  } else {
    ++u->launches;
    UN_CUDA(conv_fwd<bf16>(u, 8, a + A.d2b, c2, c2, 1, a + A.a1b, c1, n, a + A.d1a));
  }
  u->head_fused = u->plan_ok[9] && u->plan[9].orient == 0;
  if (u->head_fused) {
    tc::ConvIO io;
    io.src0 = a + A.d1a;
    io.wpack = wp + u->pack_off[9];
    io.bias = u->p + u->boff[9];
    io.head_w = static_cast<const bf16*>(u->pt) + u->woff[10];
    io.head_b = u->p + u->boff[10];
    io.res = x + (u->cin - 1);
    io.res_stride = u->cin;
    io.yout = out;
    io.err = u->dev_err;
    ++u->launches;
    UN_CUDA(tc::conv_forward(u->plan[9], io, u->st));
  } else {
    ++u->launches;
    UN_CUDA(plain(9, a + A.d1a, c1, a + A.d1b, n));
    UN_CUDA(head_fwd<bf16>(u, a + A.d1b, x + (u->cin - 1), u->cin, n, out));
  }
  int flag = 0;
  UN_CUDA(cudaMemcpyAsync(&flag, u->dev_err, sizeof(int), cudaMemcpyDeviceToHost, u->st));
  UN_CUDA(cudaStreamSynchronize(u->st));
  if (flag) {
    cudaMemsetAsync(u->dev_err, 0, sizeof(int), u->st);
    u->err = "tensor-core convolution: a pipeline wait timed out";
    return RECON_ERR_CUDA;
  }
  return RECON_OK;
}

template <typename T>
recon_status backward_t(recon_unet* u, const float* x, const float* target, int n, double* loss) {
  recon_status rs = forward_t<T>(u, x, n, u->y);
  if (rs != RECON_OK) return rs;
  const Acts A = act_layout(u, n);
  const Grads G = grad_layout(u, n);
  const T* a = static_cast<const T*>(u->acts);
  float* g = u->grads;
  const int c1 = u->c1, c2 = 2 * c1, c3 = 4 * c1, n2 = n / 2, n4 = n / 4;
  const long long V1 = (long long)n * n * n, V2 = V1 / 8, V3 = V1 / 64;
  UN_CUDA(cudaMemsetAsync(u->g, 0, u->np * sizeof(float), u->st));
  UN_CUDA(cudaMemsetAsync(u->loss, 0, sizeof(double), u->st));
  const int hb = grid_for(V1) < 608 ? grid_for(V1) : 608;
  float *gw10 = u->g + u->woff[10], *gb10 = u->g + u->boff[10];
  const T* w10 = static_cast<const T*>(u->pt) + u->woff[10];
  if (c1 == 8) head_back_kernel<T, 8><<<hb, 256, 0, u->st>>>(u->y, target, a + A.d1b, w10, V1, g + G.gd1b, gw10, gb10, u->loss);
  else head_back_kernel<T, 16><<<hb, 256, 0, u->st>>>(u->y, target, a + A.d1b, w10, V1, g + G.gd1b, gw10, gb10, u->loss);
  const T* none = nullptr;
  UN_CUDA(conv_back<T>(u, 9, a + A.d1a, c1, c1, 0, none, 0, g + G.gd1b, n, g + G.gd1a, nullptr, a + A.d1a));
  UN_CUDA(conv_back<T>(u, 8, a + A.d2b, c2, c2, 1, a + A.a1b, c1, g + G.gd1a, n, g + G.gu2, g + G.gs1, none));
  up_backward_kernel<T><<<grid_for(V2 * c2 / 4), 256, 0, u->st>>>(g + G.gu2, c2, n, g + G.gd2b, a + A.d2b);
  UN_CUDA(conv_back<T>(u, 7, a + A.d2a, c2, c2, 0, none, 0, g + G.gd2b, n2, g + G.gd2a, nullptr, a + A.d2a));
  UN_CUDA(conv_back<T>(u, 6, a + A.a3b, c3, c3, 1, a + A.a2b, c2, g + G.gd2a, n2, g + G.gu3, g + G.gs2, none));
  up_backward_kernel<T><<<grid_for(V3 * c3 / 4), 256, 0, u->st>>>(g + G.gu3, c3, n2, g + G.ga3b, a + A.a3b);
  UN_CUDA(conv_back<T>(u, 5, a + A.a3a, c3, c3, 0, none, 0, g + G.ga3b, n4, g + G.ga3a, nullptr, a + A.a3a));
  UN_CUDA(conv_back<T>(u, 4, a + A.p2, c2, c2, 0, none, 0, g + G.ga3a, n4, g + G.gp2, nullptr, none));
  pool_backward_kernel<T><<<grid_for(V2 * c2 / 4), 256, 0, u->st>>>(g + G.gp2, c2, n2, g + G.gs2, a + A.a2b);
  UN_CUDA(conv_back<T>(u, 3, a + A.a2a, c2, c2, 0, none, 0, g + G.gs2, n2, g + G.ga2a, nullptr, a + A.a2a));
  UN_CUDA(conv_back<T>(u, 2, a + A.p1, c1, c1, 0, none, 0, g + G.ga2a, n2, g + G.gp1, nullptr, none));
  pool_backward_kernel<T><<<grid_for(V1 * c1 / 4), 256, 0, u->st>>>(g + G.gp1, c1, n, g + G.gs1, a + A.a1b);
  UN_CUDA(conv_back<T>(u, 1, a + A.a1a, c1, c1, 0, none, 0, g + G.gs1, n, g + G.ga1a, nullptr, a + A.a1a));
  UN_CUDA(conv_back<T>(u, 0, a + A.x8, 8, u->cin, 0, none, 0, g + G.ga1a, n, nullptr, nullptr, none));
  UN_CUDA(cudaGetLastError());
  if (loss) {
    UN_CUDA(cudaMemcpyAsync(loss, u->loss, sizeof(double), cudaMemcpyDeviceToHost, u->st));
    UN_CUDA(cudaStreamSynchronize(u->st));
  }
  return RECON_OK;
}

}  // namespace

extern "C" {

recon_status recon_unet_param_count(int c1, size_t* count) {
  if ((c1 != 8 && c1 != 16) || !count) return RECON_ERR_INVALID_ARG;
  recon_unet tmp;
  tmp.c1 = c1;
  make_spec(&tmp);
  *count = tmp.np;
  return RECON_OK;
}

recon_status recon_unet_create(int c1, int bf16_storage, void* stream, recon_unet** out) {
  if (!out || (c1 != 8 && c1 != 16)) return RECON_ERR_INVALID_ARG;
  *out = nullptr;
  recon_unet* u = new recon_unet();
  u->c1 = c1;
  u->bf16 = bf16_storage ? 1 : 0;
  u->st = (cudaStream_t)stream;
  make_spec(u);
  const size_t es = u->bf16 ? 2 : 4;
  if (cudaMalloc(&u->p, u->np * 4) != cudaSuccess || cudaMalloc(&u->g, u->np * 4) != cudaSuccess ||
      cudaMalloc(&u->m1, u->np * 4) != cudaSuccess || cudaMalloc(&u->m2, u->np * 4) != cudaSuccess ||
      cudaMalloc(&u->decay, u->np) != cudaSuccess || cudaMalloc(&u->pt, u->np * es) != cudaSuccess ||
      cudaMalloc(&u->loss, sizeof(double)) != cudaSuccess || cudaMalloc(&u->dev_err, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    recon_unet_destroy(u);
    return RECON_ERR_OOM;
  }
  std::vector<unsigned char> dec(u->np, 0);
  for (size_t l = 0; l < u->spec.size(); ++l)
    for (size_t i = u->woff[l]; i < u->boff[l]; ++i) dec[i] = 1;
  if (cudaMemcpy(u->decay, dec.data(), u->np, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(u->p, 0, u->np * 4) != cudaSuccess || cudaMemset(u->pt, 0, u->np * es) != cudaSuccess ||
      cudaMemset(u->m1, 0, u->np * 4) != cudaSuccess || cudaMemset(u->m2, 0, u->np * 4) != cudaSuccess ||
      cudaMemset(u->dev_err, 0, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    recon_unet_destroy(u);
    return RECON_ERR_CUDA;
  }
  *out = u;
  return RECON_OK;
}

recon_status recon_unet_set_params(recon_unet* u, const float* host, size_t count) {
  if (!u || !host || count != u->np) return RECON_ERR_INVALID_ARG;
  UN_CUDA(cudaMemcpyAsync(u->p, host, u->np * 4, cudaMemcpyHostToDevice, u->st));
  if (u->bf16)
    to_t_kernel<bf16><<<grid_for((long long)u->np), 256, 0, u->st>>>(u->p, static_cast<bf16*>(u->pt), (long long)u->np);
  else
    UN_CUDA(cudaMemcpyAsync(u->pt, u->p, u->np * 4, cudaMemcpyDeviceToDevice, u->st));
  UN_CUDA(cudaMemsetAsync(u->m1, 0, u->np * 4, u->st));
  UN_CUDA(cudaMemsetAsync(u->m2, 0, u->np * 4, u->st));
  u->step = 0;
  ++u->pver;
  UN_CUDA(cudaStreamSynchronize(u->st));
  return RECON_OK;
}

recon_status recon_unet_get_params(recon_unet* u, float* host, size_t count) {
  if (!u || !host || count != u->np) return RECON_ERR_INVALID_ARG;
  UN_CUDA(cudaMemcpyAsync(host, u->p, u->np * 4, cudaMemcpyDeviceToHost, u->st));
  UN_CUDA(cudaStreamSynchronize(u->st));
  return RECON_OK;
}

recon_status recon_unet_get_grads(recon_unet* u, float* host, size_t count) {
  if (!u || !host || count != u->np) return RECON_ERR_INVALID_ARG;
  UN_CUDA(cudaMemcpyAsync(host, u->g, u->np * 4, cudaMemcpyDeviceToHost, u->st));
  UN_CUDA(cudaStreamSynchronize(u->st));
  return RECON_OK;
}

recon_status recon_unet_forward(recon_unet* u, const float* x, int n, float* y) {
  if (!u || !x || !y) return RECON_ERR_INVALID_ARG;
  recon_status rs = ensure(u, n, false);
  if (rs != RECON_OK) return rs;
  u->last_n = n;
  u->head_fused = false;
  if (u->bf16 && u->use_tc) return forward_tc(u, x, n, y);
  return u->bf16 ? forward_t<bf16>(u, x, n, y) : forward_t<float>(u, x, n, y);
}

recon_status recon_unet_backward(recon_unet* u, const float* x, const float* target, int n, double* loss) {
  if (!u || !x || !target) return RECON_ERR_INVALID_ARG;
  recon_status rs = ensure(u, n, true);
  if (rs != RECON_OK) return rs;
  u->last_n = n;
  u->head_fused = false;
  return u->bf16 ? backward_t<bf16>(u, x, target, n, loss) : backward_t<float>(u, x, target, n, loss);
}

recon_status recon_unet_adamw(recon_unet* u, float lr, float wd) {
  if (!u || !(lr > 0) || !(wd >= 0)) return RECON_ERR_INVALID_ARG;
  u->step += 1;
  ++u->pver;
  const float c1 = 1.f - powf(0.9f, (float)u->step), c2 = 1.f - powf(0.999f, (float)u->step);
  if (u->bf16)
    adamw_kernel<bf16><<<grid_for((long long)u->np), 256, 0, u->st>>>(u->p, u->g, u->m1, u->m2, u->decay,
                                                                       static_cast<bf16*>(u->pt), (long long)u->np, lr,
                                                                       wd, c1, c2);
  else
    adamw_kernel<float><<<grid_for((long long)u->np), 256, 0, u->st>>>(u->p, u->g, u->m1, u->m2, u->decay,
                                                                        static_cast<float*>(u->pt), (long long)u->np, lr,
                                                                        wd, c1, c2);
  UN_CUDA(cudaGetLastError());
  return RECON_OK;
}

recon_status recon_unet_destroy(recon_unet* u) {
  if (!u) return RECON_OK;
  if (u->st) cudaStreamSynchronize(u->st);
  cudaFree(u->p);
  cudaFree(u->g);
  cudaFree(u->m1);
  cudaFree(u->m2);
  cudaFree(u->decay);
  cudaFree(u->pt);
  cudaFree(u->loss);
  cudaFree(u->acts);
  cudaFree(u->grads);
  cudaFree(u->y);
  cudaFree(u->dev_err);
  cudaFree(u->wpack);
  delete u;
  return RECON_OK;
}

recon_status recon_unet_set_option(recon_unet* u, int option, int value) {
  if (!u) return RECON_ERR_INVALID_ARG;
  if (option == RECON_UNET_OPT_TENSOR_CORES) {
    u->use_tc = value ? 1 : 0;
    return RECON_OK;
  }
  return RECON_ERR_INVALID_ARG;
}

recon_status recon_unet_launch_count(recon_unet* u, long long* count) {
  if (!u || !count) return RECON_ERR_INVALID_ARG;
  *count = u->launches;
  return RECON_OK;
}

recon_status recon_unet_get_layer(recon_unet* u, int layer, float* host, size_t count) {
  if (!u || !host || layer < 0 || layer > 9 || !u->last_n || !u->acts) return RECON_ERR_INVALID_ARG;
  if (layer == 9 && u->head_fused) return RECON_ERR_STATE;
  static const int level[10] = {0, 0, 1, 1, 2, 2, 1, 1, 0, 0};
  const long long side = u->last_n >> level[layer];
  const size_t m = (size_t)(side * side * side) * u->spec[layer].cout;
  if (count != m) return RECON_ERR_INVALID_ARG;
  const Acts A = act_layout(u, u->last_n);
  const size_t offs[10] = {A.a1a, A.a1b, A.a2a, A.a2b, A.a3a, A.a3b, A.d2a, A.d2b, A.d1a, A.d1b};
  UN_CUDA(cudaStreamSynchronize(u->st));
  if (u->bf16) {
    std::vector<unsigned short> raw(m);
    UN_CUDA(cudaMemcpy(raw.data(), static_cast<const bf16*>(u->acts) + offs[layer], m * 2, cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < m; ++i) {
      const unsigned int bits = (unsigned int)raw[i] << 16;
      std::memcpy(host + i, &bits, 4);
    }
  } else {
    UN_CUDA(cudaMemcpy(host, static_cast<const float*>(u->acts) + offs[layer], m * 4, cudaMemcpyDeviceToHost));
  }
  return RECON_OK;
}

const char* recon_unet_last_error(recon_unet* u) { return u ? u->err.c_str() : ""; }

}  // extern "C"
