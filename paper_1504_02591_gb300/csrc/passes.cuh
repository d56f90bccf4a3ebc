// passes.cuh: the three kinds of FFT pass of the reconstruction, each with its pointwise work fused.
//
// A 3-D r2c transform is three passes over the field: Z (contiguous rows, real <-> half complex),
// Y and X (strided lines, one [N x C] tile of C adjacent columns per CTA).  Work that is pointwise
// in configuration space rides on the Z pass (delta formation, the radial projection (Psi.r)r of
// Eq. Nusser); work that is pointwise in Fourier space rides on the X pass, between its forward
// and inverse transforms (Z[s] = i k s / k^2 of Eq. Zeldovich, the source update of Eq. iterative
// with its convergence norms).
#pragma once
#include <cuda.h>

#include "fft_core.cuh"
#include "types.h"

namespace rg {
inline namespace RG_KNS {   // the radix order's namespace (fft_core.cuh)

constexpr int kZThreads = 256;

template <int N, int MODE = 0, int NARROW = 0>
struct SCols {  // adjacent columns in one strided tile (the 3-component k-space tiles are narrower)
  static constexpr bool kK = (MODE == S_DELTA || MODE == S_ITER);
  static constexpr int kWide = ((N / 2) % 16 == 0 && N < 1024 && !NARROW) ? 16 : 8;   // must divide N / 2
  // k-space (y) tiles: 4 adjacent kz (one 32-byte sector per row); 8 on the 256 mesh, whose lines leave room
  static constexpr int v = kK ? (N == 256 ? 8 : 4) : kWide;
  static_assert((N / 2) % v == 0 && N % v == 0, "tile columns must divide the half-grid rows");
};

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += sh[i];
  return r;  // valid in thread 0
}

// ------------------------------------------------------------------------------------------------
// Z pass: real rows of N floats <-> N/2+1 complex values (kz = 0..N/2).
// A real row is packed as N/2 complex z_m = x_2m + i x_2m+1 and transformed with an N/2-point FFT;
// the split into even/odd spectra with the exp(-2 pi i k / N) twiddles completes the r2c (and the
// reverse for c2r, which returns N times the inverse transform of the row).
// Each warp owns one row (all of its components) at a time and synchronises only with itself, so
// the CTA never waits at a block-wide barrier inside the row loop.
// ------------------------------------------------------------------------------------------------
template <int N, int NCOL>
__device__ __forceinline__ void r2c_split(float2* s, float2* qv, const float2* tw, int lane) {
  constexpr int L = N / 2;
  using Lay = RowLayout<L>;
  // every line: pairs (k, L - k) for k = 1..L/2, and k = 0 (which also gives the Nyquist value)
  for (int e = lane; e < NCOL * (L / 2 + 1); e += 32) {
    const int col = e / (L / 2 + 1), k = e % (L / 2 + 1);
    if (k == 0) {
      float2 z0 = s[Lay::phys(0, col)];
      s[Lay::phys(0, col)] = make_float2(z0.x + z0.y, 0.f);
      qv[col] = make_float2(z0.x - z0.y, 0.f);
    } else {
      const float2 zk = s[Lay::phys(k, col)], zm = s[Lay::phys(L - k, col)];
      const float2 wk = tw[k], wm = tw[L - k];
      // X[k] = (Zk + conj Zm)/2 - i w^k (Zk - conj Zm)/2
      float2 ev = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
      float2 o = make_float2(0.5f * (zk.x - zm.x), 0.5f * (zk.y + zm.y));
      float2 xk = cadd(ev, cmul(make_float2(o.y, -o.x), wk));
      float2 ev2 = make_float2(0.5f * (zm.x + zk.x), 0.5f * (zm.y - zk.y));
      float2 o2 = make_float2(0.5f * (zm.x - zk.x), 0.5f * (zm.y + zk.y));
      float2 xm = cadd(ev2, cmul(make_float2(o2.y, -o2.x), wm));
      s[Lay::phys(k, col)] = xk;
      s[Lay::phys(L - k, col)] = xm;
    }
  }
}

template <int N, int NCOL>
__device__ __forceinline__ void c2r_merge(float2* s, const float2* qv, const float2* tw, int lane) {
  constexpr int L = N / 2;
  using Lay = RowLayout<L>;
  for (int e = lane; e < NCOL * (L / 2 + 1); e += 32) {
    const int col = e / (L / 2 + 1), k = e % (L / 2 + 1);
    if (k == 0) {
      const float2 x0 = s[Lay::phys(0, col)], xl = qv[col];
      // E = X0 + conj XL, O = X0 - conj XL, Z0 = E + i O
      float2 ev = make_float2(x0.x + xl.x, x0.y - xl.y);
      float2 o = make_float2(x0.x - xl.x, x0.y + xl.y);
      s[Lay::phys(0, col)] = cadd(ev, mul_i(o));
    } else {
      const float2 xk = s[Lay::phys(k, col)], xm = s[Lay::phys(L - k, col)];
      const float2 wk = cconj(tw[k]), wm = cconj(tw[L - k]);
      float2 ev = make_float2(xk.x + xm.x, xk.y - xm.y);
      float2 o = cmul(make_float2(xk.x - xm.x, xk.y + xm.y), wk);
      float2 ev2 = make_float2(xm.x + xk.x, xm.y - xk.y);
      float2 o2 = cmul(make_float2(xm.x - xk.x, xm.y + xk.y), wm);
      s[Lay::phys(k, col)] = cadd(ev, mul_i(o));
      s[Lay::phys(L - k, col)] = cadd(ev2, mul_i(o2));
    }
  }
}

constexpr int kZWarps = kZThreads / 32;

template <int N, int MODE>
struct ZWarpSmem {  // float2 slots of one warp's private region
  static constexpr int NF = (MODE == Z_DELTA) ? 1 : 3;
  static constexpr int kLines = (NF * RowLayout<N / 2>::kStride + 1) & ~1;   // even: keeps raw 16-B aligned
  static constexpr int kQ = 4;                                  // Nyquist values (padded)
  static constexpr int kRaw = (MODE == Z_DELTA) ? N : (MODE == Z_WARM ? N / 4 : 0);   // raw rows / coarse row
  static constexpr int v = kLines + kQ + kRaw + ((kLines + kQ + kRaw) & 1);
};

// 1024-point lines hold twice the butterflies per thread: two CTAs per SM (128 registers) there;
// the radix-3 and 64-point rows of N = 384 and 128 spill at 64 registers, so three CTAs (85)
template <int N>
constexpr int kZMinBlocks = N >= 1024 ? 2 : ((N == 384 || N == 128) ? 3 : 4);

template <int N, int MODE, int NC>
__global__ void __launch_bounds__(kZThreads, kZMinBlocks<N>) zpass_kernel(const ZArgs a) {
  constexpr int L = N / 2;
  constexpr int NF = (MODE == Z_DELTA) ? 1 : NC;   // lines transformed per row
  using Lay = RowLayout<L>;
  constexpr int WS = ZWarpSmem<N, MODE>::v;
  constexpr int TABZ = (Plan<L>::kTab + 1) & ~1;
  extern __shared__ float4 zsm[];
  float2* tw = reinterpret_cast<float2*>(zsm);                       // exp(-2 pi i k / N), k <= L
  float2* tab = tw + L + 2;                                          // stage twiddles of the L-point FFT
  float* taps = reinterpret_cast<float*>(tab + TABZ);                // N floats (Z_DELTA)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* s = tab + TABZ + N / 2 + warp * WS;                        // this warp's lines
  float2* qv = s + ZWarpSmem<N, MODE>::kLines;
  float* raw = reinterpret_cast<float*>(qv + ZWarpSmem<N, MODE>::kQ);
  __shared__ double red_sh[kZWarps];

  for (int m = threadIdx.x; m <= L; m += kZThreads) tw[m] = a.tw[m];
  for (int m = threadIdx.x; m < Plan<L>::kTab; m += kZThreads) tab[m] = a.tab[m];
  if (MODE == Z_DELTA)
    for (int j = threadIdx.x; j < a.ntap; j += kZThreads) taps[j] = a.taps[j];
  __syncthreads();

  float acc0 = 0.f, acc1 = 0.f;
  constexpr bool kInverse = (MODE == Z_INV || MODE == Z_PROJ || MODE == Z_FINAL || MODE == Z_RADIAL);
  // device-driven iteration: once the loop flag says converged, this pass writes the real Psi
  const bool fin = (MODE == Z_PROJ) && a.loop_flag && *a.loop_flag == 1;
  float inv_alpha = 0.f, thr = 0.f;
  const int nin = a.uniform ? 1 : 2;
  if (MODE == Z_DELTA) {
    const double* red = a.red;
    inv_alpha = a.uniform ? (float)((double)N * N * N / red[RED_SUM_WG]) : (float)(red[RED_SUM_WR] / red[RED_SUM_WG]);
    thr = a.uniform ? 0.f : (float)(a.mask_frac * red[RED_SUM_WR] / red[RED_CNT_RPOS]);
  }

  for (size_t row = (size_t)blockIdx.x * kZWarps + warp; row < (size_t)N * N; row += (size_t)gridDim.x * kZWarps) {
    if (kInverse) {
      // half-complex rows (L values) and Nyquist values of every component
      for (int e = lane; e < NC * (L / 2); e += 32) {
        const int q = e / (L / 2), m2 = e % (L / 2);
        const float4 v = reinterpret_cast<const float4*>(a.f[q].M + row * L)[m2];
        s[Lay::phys(2 * m2, q)] = make_float2(v.x, v.y);
        s[Lay::phys(2 * m2 + 1, q)] = make_float2(v.z, v.w);
      }
      if (lane < NC) qv[lane] = a.f[lane].Q[row];
      __syncwarp();
      if ((MODE == Z_PROJ || MODE == Z_RADIAL) && NC == 3 && !fin) {
        // the projection needs only C = dx Psi_x + dy Psi_y and Psi_z (dx and dy are constant along
        // the row), so two rows are transformed each way: C into line 0, Psi_z into line 1
        const Geometry& g = a.g;
        const float dx = g.los_mode == 1 ? g.los.x : g.off[row / N];
        const float dy = g.los_mode == 1 ? g.los.y : g.off[N + row % N];
        for (int m = lane; m < L; m += 32) {
          const float2 p0 = s[Lay::phys(m, 0)], p1 = s[Lay::phys(m, 1)], p2 = s[Lay::phys(m, 2)];
          s[Lay::phys(m, 0)] = make_float2(fmaf(dx, p0.x, dy * p1.x), fmaf(dx, p0.y, dy * p1.y));
          s[Lay::phys(m, 1)] = p2;
        }
        if (lane == 0) {
          const float2 q0 = qv[0], q1 = qv[1];
          qv[0] = make_float2(fmaf(dx, q0.x, dy * q1.x), fmaf(dx, q0.y, dy * q1.y));
          qv[1] = qv[2];
        }
        __syncwarp();
        c2r_merge<N, 2>(s, qv, tw, lane);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 2; ++q) Plan<L>::template run<1, 32, true, Lay, true>(s + q * Lay::kStride, tab);
      } else {
        c2r_merge<N, NF>(s, qv, tw, lane);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NF; ++q) Plan<L>::template run<1, 32, true, Lay, true>(s + q * Lay::kStride, tab);
      }
    } else if (MODE == Z_USTART || MODE == Z_WARM) {
      // a radial displacement u: P = u r on the row, then its forward r2c.  Z_WARM adds to
      // u the trilinear (periodic) upsampling of a coarse correction: the coarse node J of level l
      // sits at fine index (J + 1/2) 2^l - 1/2 along each axis.
      const Geometry& g = a.g;
      const int ix = (int)(row / N), iy = (int)(row % N);
      const float dx = g.los_mode == 1 ? 0.f : g.off[ix], dy = g.los_mode == 1 ? 0.f : g.off[N + iy];
      const float* ur = a.u_in + row * N;
      float* crow = raw;   // Z_WARM: the correction bilinearly interpolated to this (x, y) row
      int nc = 0, fl = 0;
      float inv_f = 0.f;
      if (MODE == Z_WARM) {
        fl = a.clevel;
        nc = N >> fl;
        inv_f = 1.f / (float)(1 << fl);
        const float tx = ((float)ix + 0.5f) * inv_f - 0.5f, ty = ((float)iy + 0.5f) * inv_f - 0.5f;
        const float fx = floorf(tx), fy = floorf(ty);
        const float wx = tx - fx, wy = ty - fy;
        int x0 = (int)fx, y0 = (int)fy;
        x0 = x0 < 0 ? x0 + nc : x0;
        y0 = y0 < 0 ? y0 + nc : y0;
        const int x1 = x0 + 1 == nc ? 0 : x0 + 1, y1 = y0 + 1 == nc ? 0 : y0 + 1;
        const size_t r00 = ((size_t)x0 * nc + y0) * nc, r01 = ((size_t)x0 * nc + y1) * nc;
        const size_t r10 = ((size_t)x1 * nc + y0) * nc, r11 = ((size_t)x1 * nc + y1) * nc;
        for (int j = lane; j < nc; j += 32) {
          const float c00 = a.corr[r00 + j] - a.ucoarse[r00 + j], c01 = a.corr[r01 + j] - a.ucoarse[r01 + j];
          const float c10 = a.corr[r10 + j] - a.ucoarse[r10 + j], c11 = a.corr[r11 + j] - a.ucoarse[r11 + j];
          crow[j] = (1.f - wx) * ((1.f - wy) * c00 + wy * c01) + wx * ((1.f - wy) * c10 + wy * c11);
        }
        __syncwarp();
      }
      for (int m = lane; m < L; m += 32) {
        float2 uu = reinterpret_cast<const float2*>(ur)[m];
        if (MODE == Z_WARM) {
          float add[2];
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const float tz = ((float)(2 * m + h2) + 0.5f) * inv_f - 0.5f;
            const float fz = floorf(tz);
            const float wz = tz - fz;
            int z0 = (int)fz;
            z0 = z0 < 0 ? z0 + nc : z0;
            const int z1 = z0 + 1 == nc ? 0 : z0 + 1;
            add[h2] = (1.f - wz) * crow[z0] + wz * crow[z1];
          }
          uu.x += add[0];
          uu.y += add[1];
        }
        // P = u r = d psi with psi = w u (radial: w = 1/|d|; fixed LOS: d = the LOS, w = 1): line 0
        // takes psi, line 1 dz psi (the forward pass below writes dx psi^, dy psi^ and (dz psi)^)
        float dz0, dz1, w0, w1;
        if (g.los_mode == 1) {
          dz0 = dz1 = g.los.z;
          w0 = w1 = 1.f;
        } else {
          dz0 = g.off[2 * N + 2 * m];
          dz1 = g.off[2 * N + 2 * m + 1];
          const float q0 = fmaf(dx, dx, fmaf(dy, dy, dz0 * dz0));
          const float q1 = fmaf(dx, dx, fmaf(dy, dy, dz1 * dz1));
          w0 = q0 > 0.f ? rsqrtf(q0) : 0.f;
          w1 = q1 > 0.f ? rsqrtf(q1) : 0.f;
        }
        const float p0 = uu.x * w0, p1 = uu.y * w1;
        s[Lay::phys(m, 0)] = make_float2(p0, p1);
        s[Lay::phys(m, 1)] = make_float2(dz0 * p0, dz1 * p1);
      }
      __syncwarp();
    } else if (MODE == Z_DELTA) {
      // rows of rho_g (and rho_r) smoothed along x and y: z factor of the Gaussian as a periodic
      // convolution, then delta (Sec. 3.2) node by node
      for (int e = lane; e < nin * (N / 4); e += 32) {
        const int q = e / (N / 4), m4 = e % (N / 4);
        reinterpret_cast<float4*>(raw + q * N)[m4] = reinterpret_cast<const float4*>(a.f[q].M + row * L)[m4];
      }
      __syncwarp();
      const float* rg = raw;
      const float* rr = raw + N;
      for (int z = lane; z < N; z += 32) {
        int idx = z + a.t0;
        if (idx < 0) idx += N;
        float g = 0.f, r = 0.f;
        if (nin == 1) {
          for (int j = 0; j < a.ntap; ++j) {
            g = fmaf(taps[j], rg[idx], g);
            if (++idx == N) idx = 0;
          }
        } else {
          for (int j = 0; j < a.ntap; ++j) {
            g = fmaf(taps[j], rg[idx], g);
            r = fmaf(taps[j], rr[idx], r);
            if (++idx == N) idx = 0;
          }
        }
        // q = 1 + delta as the density ratio itself: the logarithm takes q, not 1 + (q - 1), which
        // in float32 would lose the digits of a low-density node to cancellation
        float q;
        if (nin == 1) {
          q = g * inv_alpha;
        } else {
          const bool in = r > thr;
          q = in ? g * inv_alpha / r : 1.f;
          acc1 += in ? 1.f : 0.f;
        }
        float d = q - 1.f;
        if (a.lognormal) {
          d = logf(fmaxf(q, 1e-6f));
          acc0 += d;
        }
        if (a.delta_real) a.delta_real[row * N + z] = d;
        reinterpret_cast<float*>(s + Lay::phys(z >> 1, 0))[z & 1] = d;
      }
      __syncwarp();
    } else {
      // real rows of N floats as L packed complex values
      for (int e = lane; e < NC * (L / 2); e += 32) {
        const int q = e / (L / 2), m2 = e % (L / 2);
        const float4 v = reinterpret_cast<const float4*>(a.f[q].M + row * L)[m2];
        s[Lay::phys(2 * m2, q)] = make_float2(v.x, v.y);
        s[Lay::phys(2 * m2 + 1, q)] = make_float2(v.z, v.w);
      }
      __syncwarp();
    }

    if (MODE == Z_RADIAL) {
      // s holds C and Psi_z (as in the projection): the start's radial displacement
      // u = coef w (C + dz Psi_z) = coef (Psi.r), as a real row
      const Geometry& g = a.g;
      const int ix = (int)(row / N), iy = (int)(row % N);
      const float dx = g.los_mode == 1 ? 0.f : g.off[ix], dy = g.los_mode == 1 ? 0.f : g.off[N + iy];
      for (int m = lane; m < L; m += 32) {
        const float2 c = s[Lay::phys(m, 0)], pz = s[Lay::phys(m, 1)];
        float dz0, dz1, w0, w1;
        if (g.los_mode == 1) {
          dz0 = dz1 = g.los.z;
          w0 = w1 = 1.f;
        } else {
          dz0 = g.off[2 * N + 2 * m];
          dz1 = g.off[2 * N + 2 * m + 1];
          const float q0 = fmaf(dx, dx, fmaf(dy, dy, dz0 * dz0));
          const float q1 = fmaf(dx, dx, fmaf(dy, dy, dz1 * dz1));
          w0 = q0 > 0.f ? rsqrtf(q0) : 0.f;
          w1 = q1 > 0.f ? rsqrtf(q1) : 0.f;
        }
        const float u0 = a.coef * (w0 * fmaf(dz0, pz.x, c.x));
        const float u1 = a.coef * (w1 * fmaf(dz1, pz.y, c.y));
        reinterpret_cast<float2*>(a.u_out + row * N)[m] = make_float2(u0, u1);
      }
      __syncwarp();
      continue;
    }

    if (MODE == Z_PROJ && NC == 3 && !fin) {
      // s holds C and Psi_z at z = 2m (.x) and 2m + 1 (.y); with r = w d (radial: w = 1/|d|; fixed
      // LOS: d = the LOS, w = 1), u = coef w (C + dz Psi_z) = coef (Psi.r) and P = u r = d psi with
      // psi = w u (Eq. Nusser): line 0 takes psi, line 1 dz psi
      const Geometry& g = a.g;
      const float dx = g.los_mode == 1 ? g.los.x : g.off[row / N];
      const float dy = g.los_mode == 1 ? g.los.y : g.off[N + row % N];
      for (int m = lane; m < L; m += 32) {
        const float2 c = s[Lay::phys(m, 0)], pz = s[Lay::phys(m, 1)];
        float dz0, dz1, w0, w1;
        if (g.los_mode == 1) {
          dz0 = dz1 = g.los.z;
          w0 = w1 = 1.f;
        } else {
          dz0 = g.off[2 * N + 2 * m];
          dz1 = g.off[2 * N + 2 * m + 1];
          const float q0 = fmaf(dx, dx, fmaf(dy, dy, dz0 * dz0));
          const float q1 = fmaf(dx, dx, fmaf(dy, dy, dz1 * dz1));
          w0 = q0 > 0.f ? rsqrtf(q0) : 0.f;
          w1 = q1 > 0.f ? rsqrtf(q1) : 0.f;
        }
        const float p0 = a.coef * (w0 * fmaf(dz0, pz.x, c.x)) * w0;
        const float p1 = a.coef * (w1 * fmaf(dz1, pz.y, c.y)) * w1;
        s[Lay::phys(m, 0)] = make_float2(p0, p1);
        s[Lay::phys(m, 1)] = make_float2(dz0 * p0, dz1 * p1);
      }
      __syncwarp();
    } else if (MODE == Z_PROJ && !fin) {
      // s holds Psi_j(x, y, z), z = 2m (.x) and 2m + 1 (.y): P = coef (Psi.r) r (Eq. Nusser)
      const Geometry& g = a.g;
      const int ix = (int)(row / N), iy = (int)(row % N);
      float dx = 0.f, dy = 0.f;
      if (g.los_mode != 1) {
        dx = g.off[ix];
        dy = g.off[N + iy];
      }
      for (int m = lane; m < L; m += 32) {
        const float2 p0 = s[Lay::phys(m, 0)], p1 = s[Lay::phys(m, 1)], p2 = s[Lay::phys(m, 2)];
        float rx0, ry0, rz0, rx1, ry1, rz1;
        if (g.los_mode == 1) {
          rx0 = rx1 = g.los.x; ry0 = ry1 = g.los.y; rz0 = rz1 = g.los.z;
        } else {
          const float dz0 = g.off[2 * N + 2 * m], dz1 = g.off[2 * N + 2 * m + 1];
          const float q0 = fmaf(dx, dx, fmaf(dy, dy, dz0 * dz0));
          const float q1 = fmaf(dx, dx, fmaf(dy, dy, dz1 * dz1));
          const float i0 = q0 > 0.f ? rsqrtf(q0) : 0.f;
          const float i1 = q1 > 0.f ? rsqrtf(q1) : 0.f;
          rx0 = dx * i0; ry0 = dy * i0; rz0 = dz0 * i0;
          rx1 = dx * i1; ry1 = dy * i1; rz1 = dz1 * i1;
        }
        const float u0 = a.coef * fmaf(p0.x, rx0, fmaf(p1.x, ry0, p2.x * rz0));
        const float u1 = a.coef * fmaf(p0.y, rx1, fmaf(p1.y, ry1, p2.y * rz1));
        s[Lay::phys(m, 0)] = make_float2(u0 * rx0, u1 * rx1);
        s[Lay::phys(m, 1)] = make_float2(u0 * ry0, u1 * ry1);
        s[Lay::phys(m, 2)] = make_float2(u0 * rz0, u1 * rz1);
      }
      __syncwarp();
    }

    if (MODE == Z_INV || MODE == Z_FINAL || (MODE == Z_PROJ && fin)) {
      for (int e = lane; e < NC * (L / 2); e += 32) {
        const int q = e / (L / 2), m2 = e % (L / 2);
        const float2 v0 = s[Lay::phys(2 * m2, q)], v1 = s[Lay::phys(2 * m2 + 1, q)];
        reinterpret_cast<float4*>(a.f[q].M + row * L)[m2] = make_float4(v0.x, v0.y, v1.x, v1.y);
      }
    } else if ((MODE == Z_PROJ || MODE == Z_USTART || MODE == Z_WARM) && NC == 3) {
      // psi^ and (dz psi)^; P_x = dx psi^ and P_y = dy psi^ are scaled copies
#pragma unroll
      for (int q = 0; q < 2; ++q) Plan<L>::template run<1, 32, false, Lay, true>(s + q * Lay::kStride, tab);
      r2c_split<N, 2>(s, qv, tw, lane);
      __syncwarp();
      const Geometry& g = a.g;
      const float dx = g.los_mode == 1 ? g.los.x : g.off[row / N];
      const float dy = g.los_mode == 1 ? g.los.y : g.off[N + row % N];
      for (int m2 = lane; m2 < L / 2; m2 += 32) {
        const float2 v0 = s[Lay::phys(2 * m2, 0)], v1 = s[Lay::phys(2 * m2 + 1, 0)];
        const float2 z0 = s[Lay::phys(2 * m2, 1)], z1 = s[Lay::phys(2 * m2 + 1, 1)];
        reinterpret_cast<float4*>(a.f[0].M + row * L)[m2] = make_float4(dx * v0.x, dx * v0.y, dx * v1.x, dx * v1.y);
        reinterpret_cast<float4*>(a.f[1].M + row * L)[m2] = make_float4(dy * v0.x, dy * v0.y, dy * v1.x, dy * v1.y);
        reinterpret_cast<float4*>(a.f[2].M + row * L)[m2] = make_float4(z0.x, z0.y, z1.x, z1.y);
      }
      if (lane == 0) {
        a.f[0].Q[row] = cscale(qv[0], dx);
        a.f[1].Q[row] = cscale(qv[0], dy);
        a.f[2].Q[row] = qv[1];
      }
    } else {
#pragma unroll
      for (int q = 0; q < NF; ++q) Plan<L>::template run<1, 32, false, Lay, true>(s + q * Lay::kStride, tab);
      r2c_split<N, NF>(s, qv, tw, lane);
      __syncwarp();
      for (int e = lane; e < NF * (L / 2); e += 32) {
        const int q = e / (L / 2), m2 = e % (L / 2);
        const float2 v0 = s[Lay::phys(2 * m2, q)], v1 = s[Lay::phys(2 * m2 + 1, q)];
        float2* dst = (MODE == Z_DELTA) ? a.dout.M : a.f[q].M;
        reinterpret_cast<float4*>(dst + row * L)[m2] = make_float4(v0.x, v0.y, v1.x, v1.y);
      }
      if (lane < NF) ((MODE == Z_DELTA) ? a.dout.Q : a.f[lane].Q)[row] = qv[lane];
    }
    __syncwarp();   // the stores above read s before the next row overwrites it
  }

  if (MODE == Z_DELTA) {
    double r0 = block_sum((double)acc0, red_sh);
    double r1 = block_sum((double)acc1, red_sh);
    if (threadIdx.x == 0) {
      a.partials[2 * blockIdx.x + 0] = r0;
      a.partials[2 * blockIdx.x + 1] = r1;
    }
  }
}

// ------------------------------------------------------------------------------------------------
// The register-fused family (N = 256, 384, 512, 1024): transforms whose first stage takes its inputs
// straight from global memory (or from the previous transform's last stage) and whose last stage's
// outputs go straight on, in registers, so that shared memory carries only what changes hands between
// stages.  That needs plans whose last stage leaves on a thread exactly the points its first stage
// reads:
//   lines of N (k-space and x passes):  8 x N/64 x 8, butterfly j at the points j + (N/8) r
//   rows of L = N/2 (z pass):           E x G with G lanes a row and E points a lane, lane l at the
//                                       points l + G r: one exchange per transform
// The other mesh sides, and the alternative radix order, use the staged kernels above and below.
// ------------------------------------------------------------------------------------------------
template <int N>
constexpr bool kFusedMesh = RG_RADIX_ORDER == 0 && (N == 256 || N == 384 || N == 512 || N == 1024);

// The z passes of the family.  A group of G lanes transforms one row of L = G E complex points, E a
// lane; a warp holds RPW = 32 / G rows: the two fields (C, Psi_z) of RPW / 2 mesh rows (x, y), field q
// of a mesh row on lane group 2 p + q.  Stage 1 is a radix-E butterfly per lane on its own points
// l + G r; one exchange through shared memory (the row's buffer, one pad word per E so that writes at
// stride E and reads fall in distinct banks); stage 2 is E / G radix-G butterflies per lane, which
// leave the points l + G r again.  The c2r merge pairs point m with L - m on lane G - l (lane 0 with
// itself and the Nyquist value), so it and the r2c split run on shuffles.
// The pass is bound by the L1's shared-memory pipe (the three-stage warp-per-row form used it 80% of
// the time): one exchange instead of two and twiddles shared by the warp's rows cut its wavefronts.
template <int N>
struct ZRow {
  static constexpr int L = N / 2;
  static constexpr int G = (N >= 512) ? 16 : 8;
  static constexpr int E = L / G;              // 16, 24, 16, 32
  static constexpr int Q = E / G;              // stage-2 butterflies a lane
  static_assert(E % G == 0, "stage 2 divides evenly over the row's lanes");
  static constexpr int RPW = 32 / G;           // rows a warp
  static constexpr int PPW = RPW / 2;          // mesh rows (two fields each) a warp
  static constexpr int kRow = (E + 1) * G;     // float2 of one row's buffer
  static constexpr int kTab = (G - 1) * E;     // stage-2 twiddles
  static constexpr int kHead = (L + 1 + kTab + 1) & ~1;
  static constexpr size_t smem = sizeof(float2) * ((size_t)kHead + (size_t)kZWarps * RPW * kRow);
  // CTAs per SM that the points a lane holds leave registers for (measured: 512 at 2, 3, 4 CTAs 576,
  // 534, 529 us; 384 at 2, 3 304, 275 us)
  static constexpr int kMinBlocks = E == 16 ? 4 : (E == 24 ? 3 : 2);
};

// Twiddles of the pass: tw[m] = exp(-2 pi i m / N), m <= L, and the stage-2 table [r - 1][j] =
// exp(-2 pi i r j / L).
template <int N>
__device__ __forceinline__ void zrow_tables(const ZArgs& a, float2* tw, float2* tab) {
  using Z = ZRow<N>;
  for (int m = threadIdx.x; m <= Z::L; m += kZThreads) tw[m] = a.tw[m];
  for (int e = threadIdx.x; e < Z::kTab; e += kZThreads) tab[e] = a.tw[2 * (1 + e / Z::E) * (e % Z::E)];
  __syncthreads();
}

// The L-point transforms of the warp's rows: v[r] = x[l + G r] in, X[l + G r] out; s is the row's buffer.
template <bool INV, int N>
__device__ __forceinline__ void zrow_fft(float2 (&v)[ZRow<N>::E], float2* __restrict__ s,
                                         const float2* __restrict__ tab, int l) {
  using Z = ZRow<N>;
  constexpr int E = Z::E, G = Z::G;
  Dft<E, INV>::run(v);
#pragma unroll
  for (int r = 0; r < E; ++r) s[(E + 1) * l + r] = v[r];
  __syncwarp();
#pragma unroll
  for (int h = 0; h < Z::Q; ++h) {
    const int j = l + G * h;
    float2 u[G];
#pragma unroll
    for (int r = 0; r < G; ++r) u[r] = s[(E + 1) * r + j];
#pragma unroll
    for (int r = 1; r < G; ++r) {
      float2 w = tab[(r - 1) * E + j];
      if (INV) w.y = -w.y;
      u[r] = cmul(u[r], w);
    }
    Dft<G, INV>::run(u);
#pragma unroll
    for (int r = 0; r < G; ++r) v[h + Z::Q * r] = u[r];
  }
  __syncwarp();                                            // s is reused by the next transform
}

template <int N>
__device__ __forceinline__ void zrow_load(const Field& f, size_t row, int l, float2 (&x)[ZRow<N>::E], float2& xl) {
  const float2* src = f.M + row * ZRow<N>::L;
#pragma unroll
  for (int r = 0; r < ZRow<N>::E; ++r) x[r] = src[l + ZRow<N>::G * r];
  xl = f.Q[row];
}

__device__ __forceinline__ float2 shfl2(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ float2 shfl2_xor(float2 v, int m) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

// Walk the mirror pairs of a row in place: fn(r, x[r], mirror) for every point, both values original.
// Point r of lane l >= 1 mirrors point E - 1 - r of lane G - l; on lane 0 point r mirrors E - r, and
// point 0's mirror is xl.
template <int N, class Fn>
__device__ __forceinline__ void zrow_mirror(float2 (&x)[ZRow<N>::E], float2 xl, int l, int partner, Fn&& fn) {
  constexpr int E = ZRow<N>::E;
  float2 prev = xl;                     // lane 0: the original x[E - r]
#pragma unroll
  for (int r = 0; r < E / 2; ++r) {
    const float2 a = x[r], b = x[E - 1 - r];
    float2 am = shfl2(b, partner), bm = shfl2(a, partner);
    if (l == 0) {
      am = prev;
      bm = r + 1 < E / 2 ? x[r + 1] : b;
    }
    prev = b;
    fn(r, x[r], a, am);
    fn(E - 1 - r, x[E - 1 - r], b, bm);
  }
}

// c2r merge of the rows in registers: X[m], the Nyquist value -> the inverse transform's inputs.
template <int N>
__device__ __forceinline__ void zrow_merge(float2 (&x)[ZRow<N>::E], float2 xl, int l, int partner,
                                           const float2* __restrict__ tw) {
  zrow_mirror<N>(x, xl, l, partner, [&](int r, float2& out, float2 xk, float2 xm) {
    const float2 w = cconj(tw[l + ZRow<N>::G * r]);
    const float2 ev = make_float2(xk.x + xm.x, xk.y - xm.y);
    const float2 o = cmul(make_float2(xk.x - xm.x, xk.y + xm.y), w);
    out = cadd(ev, mul_i(o));
  });
}

// r2c split of the transformed rows, stored as a half-complex row and its Nyquist value.
template <int N>
__device__ __forceinline__ void zrow_split_store(float2 (&y)[ZRow<N>::E], const Field& f, size_t row, int l, int partner,
                                                 const float2* __restrict__ tw) {
  float2* dst = f.M + row * ZRow<N>::L;
  zrow_mirror<N>(y, y[0], l, partner, [&](int r, float2&, float2 zk, float2 zm) {
    const int k = l + ZRow<N>::G * r;
    float2 xk;
    if (r == 0 && l == 0) {
      xk = make_float2(zk.x + zk.y, 0.f);
      f.Q[row] = make_float2(zk.x - zk.y, 0.f);
    } else {
      const float2 ev = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
      const float2 o = make_float2(0.5f * (zk.x - zm.x), 0.5f * (zk.y + zm.y));
      xk = cadd(ev, cmul(make_float2(o.y, -o.x), tw[k]));
    }
    dst[k] = xk;
  });
}

// The observer offset d = (dx, dy, dz) of a node and w with r = w d the line of sight (radial: w =
// 1/|d|, zero at the observer; fixed LOS: d = the LOS vector, w = 1), at the real points 2m and
// 2m + 1 of a row; dx and dy are the row's.
__device__ __forceinline__ void zrow_dw(const Geometry& g, float dx, float dy, int m, float& dz0, float& dz1,
                                        float& w0, float& w1) {
  if (g.los_mode == 1) {
    dz0 = dz1 = g.los.z;
    w0 = w1 = 1.f;
    return;
  }
  const float2 dz = reinterpret_cast<const float2*>(g.off + 2 * g.n)[m];   // n is even, the table 256-byte aligned
  dz0 = dz.x;
  dz1 = dz.y;
  const float q0 = fmaf(dx, dx, fmaf(dy, dy, dz0 * dz0));
  const float q1 = fmaf(dx, dx, fmaf(dy, dy, dz1 * dz1));
  w0 = q0 > 0.f ? rsqrtf(q0) : 0.f;
  w1 = q1 > 0.f ? rsqrtf(q1) : 0.f;
}

// With r = w d, the projection P = coef (Psi.r) r needs only C = dx Psi_x + dy Psi_y and Psi_z (dx,
// dy are constant along a z row; the inverse x pass forms C):  u = coef w (C + dz Psi_z) and
// P_j = d_j psi with psi = w u.  So the pass transforms two rows each way and leaves
// psi^ = r2c(psi) and Z^ = r2c(dz psi) (P_x = dx psi^ and P_y = dy psi^ are formed by the forward x
// pass).
//   Z_PROJ:   c2r x2 of C (f[0]) and Psi_z (wf), P, r2c x2; once the device loop has converged,
//             c2r x3 and the real Psi.
//   Z_FINAL:  c2r x3 and the real Psi.
//   Z_RADIAL: c2r x2, u as a real row.
//   Z_WARM:   u from the real row plus the upsampled coarse correction, r2c x2.
//   Z_USTART: u from the real row, r2c x2.
template <int N, int MODE>
__global__ void __launch_bounds__(kZThreads, ZRow<N>::kMinBlocks) zfused_kernel(const ZArgs a) {
  using Z = ZRow<N>;
  constexpr int L = Z::L, E = Z::E, G = Z::G;
  extern __shared__ float4 zsm[];
  float2* tw = reinterpret_cast<float2*>(zsm);                        // exp(-2 pi i m / N), m <= L
  float2* tab = tw + L + 1;                                           // stage-2 twiddles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = lane % G, grp = lane / G, q = grp & 1, pr = grp >> 1;
  float2* sw = tw + Z::kHead + warp * Z::RPW * Z::kRow;
  float2* s = sw + grp * Z::kRow;
  zrow_tables<N>(a, tw, tab);
  const bool fin = MODE == Z_FINAL || (MODE == Z_PROJ && a.loop_flag && *a.loop_flag == 1);
  const int partner = grp * G + (G - l) % G;
  const Geometry& g = a.g;
  // rows (ix, iy) of every y-plane, or of the planes [ybeg, ybeg + ycount)
  const int nrows = a.ycount ? N * a.ycount : N * N;
  auto row_of = [&](int lr) { return a.ycount ? (lr / a.ycount) * N + a.ybeg + lr % a.ycount : lr; };

  if (fin) {
    // the real Psi: RPW rows of one component at a time
    for (int it = blockIdx.x * kZWarps + warp; it < 3 * (nrows / Z::RPW); it += gridDim.x * kZWarps) {
      const Field f = a.f[it / (nrows / Z::RPW)];
      const size_t row = row_of((it % (nrows / Z::RPW)) * Z::RPW + grp);
      float2 x[E], xl;
      zrow_load<N>(f, row, l, x, xl);
      zrow_merge<N>(x, xl, l, partner, tw);
      zrow_fft<true, N>(x, s, tab, l);
      float2* dst = f.M + row * L;
#pragma unroll
      for (int r = 0; r < E; ++r) dst[l + G * r] = x[r];
    }
    return;
  }
  if (MODE == Z_FINAL) return;
  for (int it = blockIdx.x * kZWarps + warp; it < nrows / Z::PPW; it += gridDim.x * kZWarps) {
    const int row = row_of(it * Z::PPW + pr);
    const int ix = row / N, iy = row % N;
    const float dx = g.los_mode == 1 ? g.los.x : g.off[ix], dy = g.los_mode == 1 ? g.los.y : g.off[N + iy];
    float2 v[E];   // C or Psi_z, then psi or dz psi, at the points l + G r
    if (MODE == Z_WARM || MODE == Z_USTART) {
      float* crow = reinterpret_cast<float*>(sw + 2 * pr * Z::kRow);   // Z_WARM: the mesh row's coarse correction
      float inv_f = 1.f;
      int nc = 1;
      if (MODE == Z_WARM) {
        // u = u_s + U[corr - ucoarse] (see the generic pass)
        const int fl = a.clevel;
        nc = N >> fl;
        inv_f = 1.f / (float)(1 << fl);
        const float tx = ((float)ix + 0.5f) * inv_f - 0.5f, ty = ((float)iy + 0.5f) * inv_f - 0.5f;
        const float fx = floorf(tx), fy = floorf(ty);
        const float wx = tx - fx, wy = ty - fy;
        int x0 = (int)fx, y0 = (int)fy;
        x0 = x0 < 0 ? x0 + nc : x0;
        y0 = y0 < 0 ? y0 + nc : y0;
        const int x1 = x0 + 1 == nc ? 0 : x0 + 1, y1 = y0 + 1 == nc ? 0 : y0 + 1;
        const size_t r00 = ((size_t)x0 * nc + y0) * nc, r01 = ((size_t)x0 * nc + y1) * nc;
        const size_t r10 = ((size_t)x1 * nc + y0) * nc, r11 = ((size_t)x1 * nc + y1) * nc;
        for (int jz = q * G + l; jz < nc; jz += 2 * G) {
          const float c00 = a.corr[r00 + jz] - a.ucoarse[r00 + jz], c01 = a.corr[r01 + jz] - a.ucoarse[r01 + jz];
          const float c10 = a.corr[r10 + jz] - a.ucoarse[r10 + jz], c11 = a.corr[r11 + jz] - a.ucoarse[r11 + jz];
          crow[jz] = (1.f - wx) * ((1.f - wy) * c00 + wy * c01) + wx * ((1.f - wy) * c10 + wy * c11);
        }
        __syncwarp();
      }
      const float2* ur = reinterpret_cast<const float2*>(a.u_in + (size_t)row * N);
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int m = l + G * r;
        float2 uu = ur[m];
        if (MODE == Z_WARM) {
          float add[2];
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const float tz = ((float)(2 * m + h2) + 0.5f) * inv_f - 0.5f;
            const float fz = floorf(tz);
            const float wz = tz - fz;
            int z0 = (int)fz;
            z0 = z0 < 0 ? z0 + nc : z0;
            const int z1 = z0 + 1 == nc ? 0 : z0 + 1;
            add[h2] = (1.f - wz) * crow[z0] + wz * crow[z1];
          }
          uu.x += add[0];
          uu.y += add[1];
        }
        float dz0, dz1, w0, w1;
        zrow_dw(g, dx, dy, m, dz0, dz1, w0, w1);
        const float p0 = uu.x * w0, p1 = uu.y * w1;
        v[r] = q ? make_float2(dz0 * p0, dz1 * p1) : make_float2(p0, p1);
      }
      if (MODE == Z_WARM) __syncwarp();   // crow shares the rows' buffers
    } else {
      float2 xl;
      zrow_load<N>(q ? a.wf : a.f[0], row, l, v, xl);
      zrow_merge<N>(v, xl, l, partner, tw);
      zrow_fft<true, N>(v, s, tab, l);
      // u = coef (Psi . r) at the real points 2m, 2m + 1 of the complex point m (Eq. Nusser).  The two
      // lane groups of a mesh row share the work: field 0's lanes form the points r < E/2 and field 1's
      // the rest, and they swap what the other needs.
#pragma unroll
      for (int r = 0; r < E / 2; ++r) {
        const int rm = q ? r + E / 2 : r, m = l + G * rm;
        const float2 mine = q ? v[r + E / 2] : v[r];
        const float2 other = shfl2_xor(q ? v[r] : v[r + E / 2], G);
        const float2 c = q ? other : mine, pz = q ? mine : other;
        float dz0, dz1, w0, w1;
        zrow_dw(g, dx, dy, m, dz0, dz1, w0, w1);
        const float u0 = a.coef * (w0 * fmaf(dz0, pz.x, c.x));
        const float u1 = a.coef * (w1 * fmaf(dz1, pz.y, c.y));
        if (MODE == Z_RADIAL) {
          reinterpret_cast<float2*>(a.u_out + (size_t)row * N)[m] = make_float2(u0, u1);
        } else {
          const float p0 = u0 * w0, p1 = u1 * w1;
          const float2 psi = make_float2(p0, p1), zpsi = make_float2(dz0 * p0, dz1 * p1);
          const float2 back = shfl2_xor(q ? psi : zpsi, G);   // the other field's value at this point
          // field 0 keeps psi at r (own) and r + E/2 (from field 1); field 1 keeps dz psi likewise
          v[r] = q ? back : psi;
          v[r + E / 2] = q ? zpsi : back;
        }
      }
      if (MODE == Z_RADIAL) continue;
    }
    zrow_fft<false, N>(v, s, tab, l);
    zrow_split_store<N>(v, q ? a.f[2] : a.f[0], row, l, partner, tw);   // psi^ and Z^ = (dz psi)^
  }
}

// Z_DELTA of the family (at most 64 smoothing taps): each warp stages its row of rho_g, then of rho_r, with
// the periodic continuation the z convolution reads; each lane convolves V consecutive nodes with V taps at a
// time in registers (a staged value is read once per V outputs and V taps; one pad word per V, so the lanes'
// windows fall in distinct banks), forms delta (mask, lognormal) exactly as the generic pass, stores the
// real copy, and runs the r2c of the fused passes.  The generic pass reads every value once per tap:
// 67 us against 182 at 256, 219 / 625 at 384, 518 / 637 at 512 (which had a form of 32 taps with both
// rows staged) and 4430 / 11540 at 1024, one field.  Both fields staged at once leave fewer CTAs: 384 256,
// 512 602, 1024 8830 us.
template <int N>
struct ZDeltaRow {
  using ZR = ZRow<N>;
  static constexpr int KT = 64, V = N <= 512 ? N / 32 : 16, PARTS = N / (32 * V);
  static constexpr int kTaps = (KT + V - 1) / V * V;            // taps, zero beyond the last
  static constexpr int kExt = N + kTaps;                        // staged entries per row
  static constexpr int kExtPad = (kExt + kExt / V + 2) & ~1;    // with one pad word per V
  static constexpr int kWarp = ZR::RPW * ZR::kRow + kExtPad / 2;   // float2: FFT buffers + a staged row
  static constexpr size_t smem = sizeof(float2) * ((size_t)ZR::kHead + (size_t)kZWarps * kWarp) + sizeof(float) * kTaps;
  static constexpr int kMinBlocks = N == 256 ? 4 : (N <= 512 ? 3 : 2);   // 512 at 2: 580 us
  __device__ __forceinline__ static int pad(int p) { return p + p / V; }
};

template <int N>
__global__ void __launch_bounds__(kZThreads, ZDeltaRow<N>::kMinBlocks) zdelta_kernel(const ZArgs a) {
  using Z = ZDeltaRow<N>;
  using ZR = ZRow<N>;
  constexpr int L = ZR::L, V = Z::V, PARTS = Z::PARTS, G = ZR::G, E = ZR::E;
  extern __shared__ float4 zsm[];
  float2* tw = reinterpret_cast<float2*>(zsm);
  float2* tab = tw + L + 1;
  float* taps = reinterpret_cast<float*>(tw + ZR::kHead + kZWarps * Z::kWarp);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % G, grp = lane / G;
  float2* sw = tw + ZR::kHead + warp * Z::kWarp;                 // the rows' FFT buffers
  float* x = reinterpret_cast<float*>(sw + ZR::RPW * ZR::kRow);  // the staged row
  __shared__ double red_sh[kZWarps];
  for (int j = threadIdx.x; j < Z::kTaps; j += kZThreads) taps[j] = j < a.ntap ? a.taps[j] : 0.f;
  zrow_tables<N>(a, tw, tab);
  const double* red = a.red;
  const int nin = a.uniform ? 1 : 2;
  const float inv_alpha = a.uniform ? (float)((double)N * N * N / red[RED_SUM_WG]) : (float)(red[RED_SUM_WR] / red[RED_SUM_WG]);
  const float thr = a.uniform ? 0.f : (float)(a.mask_frac * red[RED_SUM_WR] / red[RED_CNT_RPOS]);
  const int partner = grp * G + (G - l) % G;
  const int chunks = (a.ntap + V - 1) / V;
  float acc0 = 0.f, acc1 = 0.f;

  for (int it = blockIdx.x * kZWarps + warp; it < N * N / ZR::RPW; it += gridDim.x * kZWarps) {
#pragma unroll 1
    for (int i = 0; i < ZR::RPW; ++i) {
      const size_t row = (size_t)it * ZR::RPW + i;
      float ag[PARTS][V], ar[PARTS][V];
      auto smooth = [&](const float2* M, float (&acc)[PARTS][V]) {
        const float* src = reinterpret_cast<const float*>(M) + row * N;
#pragma unroll 8
        for (int p = lane; p < Z::kExt; p += 32) {   // |t0| <= 32: one wrap at most
          const int k = p + a.t0;
          x[Z::pad(p)] = src[k < 0 ? k + N : (k >= N ? k - N : k)];
        }
        __syncwarp();
#pragma unroll
        for (int part = 0; part < PARTS; ++part) {
#pragma unroll
          for (int v = 0; v < V; ++v) acc[part][v] = 0.f;
#pragma unroll 1
          for (int c = 0; c < chunks; ++c) {
            float tp[V];
#pragma unroll
            for (int j = 0; j < V; ++j) tp[j] = taps[V * c + j];
            const float* xo = x + (lane + 32 * part + c) * (V + 1);   // pad(V (lane + 32 part + c))
#pragma unroll
            for (int w = 0; w < 2 * V - 1; ++w) {
              const float xv = xo[w + w / V];
#pragma unroll
              for (int v = 0; v < V; ++v)
                if (w - v >= 0 && w - v < V) acc[part][v] = fmaf(tp[w - v], xv, acc[part][v]);
            }
          }
        }
        __syncwarp();                     // the staged row is rewritten by the next one
      };
      smooth(a.f[0].M, ag);
      if (nin == 2) smooth(a.f[1].M, ar);
#pragma unroll
      for (int part = 0; part < PARTS; ++part) {
        const int z0 = V * (lane + 32 * part);
        float d[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          float q;   // 1 + delta, kept as the ratio for the logarithm (see the generic pass)
          if (nin == 1) {
            q = ag[part][v] * inv_alpha;
          } else {
            const bool in = ar[part][v] > thr;
            q = in ? ag[part][v] * inv_alpha / ar[part][v] : 1.f;
            acc1 += in ? 1.f : 0.f;
          }
          float dv = q - 1.f;
          if (a.lognormal) {
            dv = logf(fmaxf(q, 1e-6f));
            acc0 += dv;
          }
          d[v] = dv;
        }
        if (a.delta_real) {
          float4* dr = reinterpret_cast<float4*>(a.delta_real + row * N + z0);
#pragma unroll
          for (int v4 = 0; v4 < V / 4; ++v4) dr[v4] = make_float4(d[4 * v4], d[4 * v4 + 1], d[4 * v4 + 2], d[4 * v4 + 3]);
        }
#pragma unroll
        for (int k = 0; k < V / 2; ++k) sw[i * ZR::kRow + z0 / 2 + k] = make_float2(d[2 * k], d[2 * k + 1]);
      }
    }
    __syncwarp();
    float2 y[E];
#pragma unroll
    for (int r = 0; r < E; ++r) y[r] = sw[grp * ZR::kRow + l + G * r];
    __syncwarp();
    zrow_fft<false, N>(y, sw + grp * ZR::kRow, tab, l);
    zrow_split_store<N>(y, a.dout, (size_t)it * ZR::RPW + grp, l, partner, tw);
  }
  const double r0 = block_sum((double)acc0, red_sh);
  const double r1 = block_sum((double)acc1, red_sh);
  if (threadIdx.x == 0) {
    a.partials[2 * blockIdx.x + 0] = r0;
    a.partials[2 * blockIdx.x + 1] = r1;
  }
}

template <int N, int NC>
constexpr size_t zpass_smem(int mode) {
  return sizeof(float2) * ((size_t)N / 2 + 2 + ((Plan<N / 2>::kTab + 1) & ~1) + N / 2 +
                           (size_t)kZWarps * (mode == Z_DELTA  ? ZWarpSmem<N, Z_DELTA>::v
                                              : mode == Z_WARM ? ZWarpSmem<N, Z_WARM>::v
                                                               : ZWarpSmem<N, Z_PROJ>::v));
}

// ------------------------------------------------------------------------------------------------
// Strided passes (Y and X).  A tile is N lines x C adjacent columns.  Tiles over the main array M:
//   Y: lines along y at fixed x, columns kz0..kz0+C-1      (offset (x N + y) N/2 + kz)
//   X: lines along x at fixed ky, columns kz0..kz0+C-1     (offset (x N + ky) N/2 + kz)
// and over the Nyquist plane Q [kx][ky] (the k-space passes, which need all three components of
// P at once, run along y; the plain passes run along either axis):
//   Y: lines along y (contiguous), columns are C values of x
//   X: lines along x (stride N), columns are C adjacent ky
// ------------------------------------------------------------------------------------------------
struct Tile {
  size_t base;
  int ls, cs;      // line stride, column stride (complex elements)
  int isQ;
  int a;           // x (Y pass) or ky (X pass) of an M tile
  int c0;          // first kz (M) or first column (Q)
};

template <int N, int C, int AXIS>
__device__ __forceinline__ Tile tile_of(int t) {
  constexpr int H = N / 2;
  constexpr int MT = N * (H / C);
  Tile r;
  if (t < MT) {
    r.isQ = 0;
    r.a = t / (H / C);
    r.c0 = (t % (H / C)) * C;
    r.base = (AXIS == AX_Y) ? (size_t)r.a * N * H + r.c0 : (size_t)r.a * H + r.c0;
    r.ls = (AXIS == AX_Y) ? H : N * H;
    r.cs = 1;
  } else {
    r.isQ = 1;
    r.a = 0;
    r.c0 = (t - MT) * C;
    r.base = (AXIS == AX_Y) ? (size_t)r.c0 * N : (size_t)r.c0;
    r.ls = (AXIS == AX_Y) ? 1 : N;
    r.cs = (AXIS == AX_Y) ? N : 1;
  }
  return r;
}

template <int N, int C, int T>
__device__ __forceinline__ void tile_load(float2* s, const float2* __restrict__ P, const Tile& t) {
  using Lay = ColLayout<C>;
  if (t.cs == 1) {
#pragma unroll 4
    for (int e = threadIdx.x; e < N * (C / 2); e += T) {
      const int i = e / (C / 2), cp = e % (C / 2);
      const float4 v = *reinterpret_cast<const float4*>(P + t.base + (size_t)i * t.ls + 2 * cp);
      s[Lay::phys(i, 2 * cp)] = make_float2(v.x, v.y);
      s[Lay::phys(i, 2 * cp + 1)] = make_float2(v.z, v.w);
    }
  } else {
    for (int e = threadIdx.x; e < N * C; e += T) {
      const int c = e / N, i = e % N;
      s[Lay::phys(i, c)] = P[t.base + (size_t)c * t.cs + (size_t)i * t.ls];
    }
  }
}

template <int N, int C, int T>
__device__ __forceinline__ void tile_store(const float2* s, float2* __restrict__ P, const Tile& t) {
  using Lay = ColLayout<C>;
  if (t.cs == 1) {
    for (int e = threadIdx.x; e < N * (C / 2); e += T) {
      const int i = e / (C / 2), cp = e % (C / 2);
      const float2 v0 = s[Lay::phys(i, 2 * cp)], v1 = s[Lay::phys(i, 2 * cp + 1)];
      *reinterpret_cast<float4*>(P + t.base + (size_t)i * t.ls + 2 * cp) = make_float4(v0.x, v0.y, v1.x, v1.y);
    }
  } else {
    for (int e = threadIdx.x; e < N * C; e += T) {
      const int c = e / N, i = e % N;
      P[t.base + (size_t)c * t.cs + (size_t)i * t.ls] = s[Lay::phys(i, c)];
    }
  }
}

// Stores of the k-space passes along y: the tile of G = iS/k^2 (one slot) goes out twice, scaled by
// kdx into Psi_x and by kdz into Psi_z (kx and kz are constant along a y line; M tiles: kx = t.a,
// kz = column; Nyquist tiles: kx = column, kz = N/2, whose derivative wavenumber is zero).
template <int N, int C, int T>
__device__ __forceinline__ void tile_store_xz(const float2* s, float2* __restrict__ Px, float2* __restrict__ Pz,
                                              const Tile& t, float kf) {
  using Lay = ColLayout<C>;
  constexpr int H = N / 2;
  auto kd = [&](int c, float& kdx, float& kdz) {
    const int ix = t.isQ ? t.c0 + c : t.a, kz = t.isQ ? H : t.c0 + c;
    kdx = (ix == H) ? 0.f : kf * (float)(ix < H ? ix : ix - N);
    kdz = (kz == H) ? 0.f : kf * (float)kz;
  };
  if (t.cs == 1) {
    for (int e = threadIdx.x; e < N * (C / 2); e += T) {
      const int i = e / (C / 2), cp = e % (C / 2);
      const float2 v0 = s[Lay::phys(i, 2 * cp)], v1 = s[Lay::phys(i, 2 * cp + 1)];
      float ax0, az0, ax1, az1;
      kd(2 * cp, ax0, az0);
      kd(2 * cp + 1, ax1, az1);
      const size_t gi = t.base + (size_t)i * t.ls + 2 * cp;
      *reinterpret_cast<float4*>(Px + gi) = make_float4(ax0 * v0.x, ax0 * v0.y, ax1 * v1.x, ax1 * v1.y);
      *reinterpret_cast<float4*>(Pz + gi) = make_float4(az0 * v0.x, az0 * v0.y, az1 * v1.x, az1 * v1.y);
    }
  } else {
    for (int e = threadIdx.x; e < N * C; e += T) {
      const int c = e / N, i = e % N;
      float ax, az;
      kd(c, ax, az);
      const float2 v = s[Lay::phys(i, c)];
      const size_t gi = t.base + (size_t)c * t.cs + (size_t)i * t.ls;
      Px[gi] = cscale(v, ax);
      Pz[gi] = cscale(v, az);
    }
  }
}

// Threads of a strided CTA.  The plain passes move one component per CTA in 16-column (128-byte)
// tiles with 512 threads; the 3-component k-space passes use 4-column (32-byte) tiles with 256
// threads so that three components fit three CTAs per SM.  The k-space passes run along y, whose
// lines are 2 KB strided, so narrow tiles still stream well; the 1 MB-strided x lines get the
// wide tiles.
template <int N, int MODE, int NARROW = 0>
struct SThreads {
  static constexpr bool kK = (MODE == S_DELTA || MODE == S_ITER);
  // 1024-point lines: 128 registers a thread (their butterflies and prefetched values spill at 64),
  // and the k-space passes on 512 threads so that each prefetches 8 values of delta(k) and S
  static constexpr int v = (N >= 1024 && kK) ? 512 : ((!kK && SCols<N, MODE, NARROW>::v == 16) ? 512 : 256);
  static constexpr int minb = N >= 1024 ? (kK ? 1 : 2) : (kK ? 3 : (v == 512 ? 2 : 4));
};

template <int N, int MODE, int NC, int AXIS, int NARROW = 0>
__global__ void __launch_bounds__(SThreads<N, MODE, NARROW>::v, SThreads<N, MODE, NARROW>::minb)
    spass_kernel(const SArgs a) {
  constexpr int T = SThreads<N, MODE, NARROW>::v;
  constexpr int C = SCols<N, MODE, NARROW>::v;
  constexpr int H = N / 2;
  constexpr int NS = (MODE == S_DELTA || MODE == S_ITER) ? 3 : NC;   // smem slots
  using Lay = ColLayout<C>;
  constexpr int TABS = (Plan<N>::kTab + 1) & ~1;
  extern __shared__ float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);   // stage twiddles of the N-point FFT
  float2* s = tw + TABS;
  __shared__ double red_sh[T / 32];
  const int q0 = blockIdx.y;   // plain passes: the component this CTA transforms
  // k-space passes along y: kx and kz are constant along the line, so the x and z components of
  // k . P travel as A = kdx P_x + kdz P_z (one forward transform for two) and Psi_x, Psi_z leave as
  // kdx G and kdz G of one inverse transform of G = iS/k^2
  constexpr bool RED = (MODE == S_ITER || MODE == S_DELTA) && AXIS == AX_Y;

  if ((MODE == S_FWD || MODE == S_INV) && a.skip_flag && *a.skip_flag != 0) return;   // uniform
  for (int m = threadIdx.x; m < Plan<N>::kTab; m += T) tw[m] = a.tab[m];
  const Tile t = tile_of<N, C, AXIS>(blockIdx.x);

  // ---- load
  if (MODE == S_DELTA) {
    tile_load<N, C, T>(s, t.isQ ? a.dk.Q : a.dk.M, t);
  } else {
#pragma unroll
    for (int q = 0; q < NC; ++q) tile_load<N, C, T>(s + q * N * C, t.isQ ? a.f[q0 + q].Q : a.f[q0 + q].M, t);
  }
  __syncthreads();

  if (MODE == S_ITER && RED) {
    const float kf = a.g.kf;
    for (int e = threadIdx.x; e < N * C; e += T) {
      const int i = e / C, c = e % C;
      const int ix = t.isQ ? t.c0 + c : t.a, kz = t.isQ ? H : t.c0 + c;
      const float kdx = (ix == H) ? 0.f : kf * (float)(ix < H ? ix : ix - N);
      const float kdz = (kz == H) ? 0.f : kf * (float)kz;
      const int p = Lay::phys(i, c);
      const float2 px = s[p], pz = s[2 * N * C + p];
      s[p] = make_float2(fmaf(kdx, px.x, kdz * pz.x), fmaf(kdx, px.y, kdz * pz.y));
    }
    __syncthreads();
  }

  // ---- S_ITER: fetch delta(k) and the previous source for this thread's elements now, so the
  // loads are in flight during the forward transforms instead of inside the element loop
  constexpr int PE = (N * C + T - 1) / T;
  float2 dkr[MODE == S_ITER ? PE : 1], spr[MODE == S_ITER ? PE : 1];
  if (MODE == S_ITER) {
    const float2* __restrict__ dkp = t.isQ ? a.dk.Q : a.dk.M;
    const float2* __restrict__ spp = t.isQ ? a.sbuf.Q : a.sbuf.M;
#pragma unroll
    for (int k = 0; k < PE; ++k) {
      const int e = threadIdx.x + k * T;
      if ((N * C) % T == 0 || e < N * C) {
        const int i = e / C, c = e % C;
        const size_t gi = t.base + (size_t)i * t.ls + (size_t)c * t.cs;
        dkr[k] = dkp[gi];
        spr[k] = spp[gi];
      }
    }
  }

  // ---- forward transform along the line
  if (MODE == S_FWD || MODE == S_ITER || MODE == S_FACTOR) {
#pragma unroll
    for (int q = 0; q < ((MODE == S_ITER && RED) ? 2 : NC); ++q) Plan<N>::template run<C, T, false, Lay>(s + q * N * C, tw);
  } else if (MODE == S_DELTA) {
    if (!a.d_is_k) Plan<N>::template run<C, T, false, Lay>(s, tw);
  }

  if (MODE == S_FACTOR) {
    const float* __restrict__ fac = a.fac + (t.isQ ? (size_t)N * N * H : 0);
    for (int e = threadIdx.x; e < N * C; e += T) {
      // consecutive threads on consecutive elements of the field, as the tile was loaded
      const int i = t.cs == 1 ? e / C : e % N, c = t.cs == 1 ? e % C : e / N;
      const int p = Lay::phys(i, c);
      s[p] = cscale(s[p], fac[t.base + (size_t)i * t.ls + (size_t)c * t.cs]);
    }
    __syncthreads();
  }

  float d2 = 0.f, s2 = 0.f;
  if (MODE == S_DELTA || MODE == S_ITER) {
    const Geometry& g = a.g;
#pragma unroll
    for (int k = 0; k < PE; ++k) {
      const int e = threadIdx.x + k * T;
      if ((N * C) % T != 0 && e >= N * C) break;
      const int i = e / C, c = e % C;
      // wavenumber indices of element (i, c): i runs along the pass axis
      int ix, ky, kz;
      if (AXIS == AX_X) {
        ix = i;
        if (!t.isQ) { ky = t.a; kz = t.c0 + c; } else { ky = t.c0 + c; kz = H; }
      } else {
        ky = i;
        if (!t.isQ) { ix = t.a; kz = t.c0 + c; } else { ix = t.c0 + c; kz = H; }
      }
      const int mx = (ix < H) ? ix : ix - N;
      const int my = (ky < H) ? ky : ky - N;
      const float kx = g.kf * mx, kyf = g.kf * my, kzf = g.kf * kz;
      const float k2 = kx * kx + kyf * kyf + kzf * kzf;
      const int p = Lay::phys(i, c);
      {
        const float kdx = (ix == H) ? 0.f : kx;
        const float kdy = (ky == H) ? 0.f : kyf;
        const float kdz = (kz == H) ? 0.f : kzf;
        const size_t gi = t.base + (size_t)i * t.ls + (size_t)c * t.cs;
        float2* Sp = t.isQ ? a.sbuf.Q : a.sbuf.M;
        float2 S;
        if (MODE == S_DELTA) {
          float2 dk = s[p];
          if (!a.d_is_k) {
            if (a.lognormal && ix == 0 && ky == 0 && kz == 0)
              dk.x -= (float)(a.red[RED_SUM_LOG]);   // subtract N^3 <ln(1+delta)> at k = 0
            (t.isQ ? a.dk.Q : a.dk.M)[gi] = dk;
          }
          S = cscale(dk, a.inv_b);
        } else {
          const float2 dk = dkr[MODE == S_ITER ? k : 0];
          // i k . P
          float dre, dim;
          if (RED) {   // slot 0 holds A = kdx P_x + kdz P_z
            const float2 pa = s[p], py = s[N * C + p];
            dre = fmaf(kdy, py.x, pa.x);
            dim = fmaf(kdy, py.y, pa.y);
          } else {
            const float2 px = s[p], py = s[N * C + p], pz = s[2 * N * C + p];
            dre = kdx * px.x + kdy * py.x + kdz * pz.x;
            dim = kdx * px.y + kdy * py.y + kdz * pz.y;
          }
          S = make_float2(fmaf(a.beta, -dim, dk.x * a.inv_b), fmaf(a.beta, dre, dk.y * a.inv_b));
        }
        if (k2 == 0.f) S = make_float2(0.f, 0.f);
        const float inv_k2 = (k2 > 0.f) ? 1.f / k2 : 0.f;
        if (MODE == S_ITER) {
          const float2 sp = spr[MODE == S_ITER ? k : 0];
          const float wgt = (kz == 0 || kz == H) ? 1.f : 2.f;
          const float fac = wgt * (kdx * kdx + kdy * kdy + kdz * kdz) * inv_k2 * inv_k2;
          const float ddx = S.x - sp.x, ddy = S.y - sp.y;
          d2 = fmaf(fac, ddx * ddx + ddy * ddy, d2);
          s2 = fmaf(fac, S.x * S.x + S.y * S.y, s2);
        }
        Sp[gi] = S;
        // Psi_j = i kd_j S / k^2, with the 1/N^3 of the inverse transform folded in
        const float2 iS = cscale(mul_i(S), inv_k2 * g.inv_n3);
        if (RED) {
          s[p] = iS;                           // G
          s[N * C + p] = cscale(iS, kdy);      // Psi_y
        } else {
          s[p] = cscale(iS, kdx);
          s[N * C + p] = cscale(iS, kdy);
          s[2 * N * C + p] = cscale(iS, kdz);
        }
      }
    }
    __syncthreads();
  }

  // ---- inverse transform along the line
  if (MODE == S_INV || MODE == S_DELTA || MODE == S_ITER || MODE == S_FACTOR) {
#pragma unroll
    for (int q = 0; q < (RED ? 2 : NS); ++q) Plan<N>::template run<C, T, true, Lay>(s + q * N * C, tw);
  }

  // ---- store
  if (RED) {
    tile_store_xz<N, C, T>(s, t.isQ ? a.f[0].Q : a.f[0].M, t.isQ ? a.f[2].Q : a.f[2].M, t, a.g.kf);
    tile_store<N, C, T>(s + N * C, t.isQ ? a.f[1].Q : a.f[1].M, t);
  } else {
#pragma unroll
    for (int q = 0; q < NS; ++q) tile_store<N, C, T>(s + q * N * C, t.isQ ? a.f[q0 + q].Q : a.f[q0 + q].M, t);
  }

  if (MODE == S_ITER) {
    double r0 = block_sum((double)d2, red_sh);
    double r1 = block_sum((double)s2, red_sh);
    if (threadIdx.x == 0) {
      a.partials[2 * blockIdx.x + 0] = r0;
      a.partials[2 * blockIdx.x + 1] = r1;
    }
  }
}

template <int N, int MODE, int NARROW = 0>
constexpr size_t spass_smem(int nslots) {
  return sizeof(float2) * ((size_t)((Plan<N>::kTab + 1) & ~1) + (size_t)nslots * N * SCols<N, MODE, NARROW>::v);
}

// ------------------------------------------------------------------------------------------------
// The k-space passes along y of the register-fused family, N = 8 x M x 8 (M = N/64): the butterfly j
// of the last forward stage produces X[j + (N/8) r] (r = 0..7), exactly the inputs of butterfly j of
// the first inverse stage.  So each thread loads its 8 points of a column straight from global memory
// into the first forward stage, keeps the last forward stage's outputs in registers for the source
// update, starts the inverse transform on them, and stores the last inverse stage straight to global
// memory: two shared-memory round trips per transform instead of three plus the staging of loads,
// stores and the update.
// A thread owns the edge butterfly j = tid / C of column tid % C; the middle stage's 64 butterflies of
// each line are dealt over the same threads (N = 384: 48 threads a column, 192 a CTA and three CTAs per
// SM, 8% faster than with 64 threads a column and two).
// ------------------------------------------------------------------------------------------------
template <int N, int C>
struct KFused {
  static constexpr int M = N / 64;             // radix of the middle stage (64 butterflies a line)
  static constexpr int NB = N / 8;             // edge butterflies a line
  static constexpr int TPC = NB;               // threads per column, one edge butterfly each
  static constexpr int T = TPC * C;
  static constexpr int kMinBlocks = T <= 192 ? 3 : (T <= 256 ? 2 : 1);
  static constexpr int OFF3 = (M - 1) * 8;     // the last stage's twiddles in the plan's table
  static constexpr int TAB = (Plan<N>::kTab + 1) & ~1;
  static constexpr size_t smem = sizeof(float2) * ((size_t)TAB + 2 * (size_t)N * C);   // one buffer per line
};

// Line and butterfly of a thread's p-th item of the middle stage (64 butterflies a line).
template <int TPC>
__device__ __forceinline__ int kline_item(int j, int p) {
  if (64 % TPC == 0) return p / (64 / TPC < 1 ? 1 : 64 / TPC);   // whole lines: known when compiled
  return (j + TPC * p) >> 6;
}
template <int TPC>
__device__ __forceinline__ int kline_mid(int j, int p) {
  if (64 % TPC == 0) return j + TPC * (p % (64 / TPC < 1 ? 1 : 64 / TPC));
  return (j + TPC * p) & 63;
}

// The transform as a cube (a, b, k) of 8 x M x 8 points: stage 1's butterfly j = a + 8 b turns the 8 points
// of a thread into k, stage 2's (a, k) turns b into c, stage 3's j = k + 8 c turns a into the output.  Every
// stage works in place, so a transform takes two barriers, and stage 3 leaves thread j reading exactly the
// places that the next transform's stage 1 may write when a and k swap places (ROLE 1): back-to-back
// transforms need no barrier between them.  Point (a, b, k) of a column: rows along z, x's low bits folded
// in so that neighbours along either fall in distinct banks.
template <int N, int C, int ROLE>
__device__ __forceinline__ int kcube(int a, int b, int k, int col) {
  const int x = ROLE ? k : a, z = ROLE ? a : k;
  return (8 * (b + KFused<N, C>::M * x) + (z ^ (x & ColLayout<C>::kMask))) * C + col;
}

struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};

// The N-point transforms of K lines of one column (the update: K = 2, A and P_y forward, G and Psi_y
// inverse; the vector x passes and delta: K = 1), stage by stage together (one buffer each, so a stage
// needs one barrier for all K): v[q][r] = x_q[j + (N/8) r] in, X_q[j + (N/8) r] out.  The places that stage 1
// writes must be free: a barrier since the last transform, or that one by the same lines in the other ROLE.
// Two barriers instead of the five of a transform that re-sorts between stages and frees its buffers: the
// streamed update 256 90 -> 88 us, 384 318 -> 282, 512 644 -> 611, 1024 8080 -> 6960.
template <bool INV, int N, int C, int K, int ROLE = 0, class Hook = NoHook>
__device__ __forceinline__ void kline_fft(float2 (&v)[K][8], float2* __restrict__ s, const float2* __restrict__ tw,
                                          int j, int col, Hook&& hook = Hook()) {
  using F = KFused<N, C>;
  constexpr int B = N * C, M = F::M, PM = (64 * K + F::TPC - 1) / F::TPC;
#pragma unroll
  for (int q = 0; q < K; ++q) {                            // stage 1 (NS = 1): no twiddles
    Dft<8, INV>::run(v[q]);
#pragma unroll
    for (int r = 0; r < 8; ++r) s[q * B + kcube<N, C, ROLE>(j & 7, j >> 3, r, col)] = v[q][r];
  }
  __syncthreads();
  hook();
#pragma unroll
  for (int p = 0; p < PM; ++p) {                           // stage 2 (NS = 8): items (line, butterfly)
    if ((64 * K) % F::TPC == 0 || j + F::TPC * p < 64 * K) {
      const int q = kline_item<F::TPC>(j, p), jm = kline_mid<F::TPC>(j, p), k = jm & 7;
      float2 u[M];
#pragma unroll
      for (int r = 0; r < M; ++r) u[r] = s[q * B + kcube<N, C, ROLE>(jm >> 3, r, k, col)];
#pragma unroll
      for (int r = 1; r < M; ++r) {
        float2 w = tw[(r - 1) * 8 + k];
        if (INV) w.y = -w.y;
        u[r] = cmul(u[r], w);
      }
      Dft<M, INV>::run(u);
#pragma unroll
      for (int r = 0; r < M; ++r) s[q * B + kcube<N, C, ROLE>(jm >> 3, r, k, col)] = u[r];
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < K; ++q) {                            // stage 3 (NS = N/8)
#pragma unroll
    for (int r = 0; r < 8; ++r) v[q][r] = s[q * B + kcube<N, C, ROLE>(r, j >> 3, j & 7, col)];
#pragma unroll
    for (int r = 1; r < 8; ++r) {
      float2 w = tw[F::OFF3 + (r - 1) * F::NB + j];
      if (INV) w.y = -w.y;
      v[q][r] = cmul(v[q][r], w);
    }
    Dft<8, INV>::run(v[q]);
  }
}

// Signed frequency of the point j + (N/8) r of a line, r known when compiled; exact, so kf times it is what
// kf times the integer is.
template <int N>
__device__ __forceinline__ float line_freq(float fj, int r) {
  return fj + (float)(r < 4 ? (N / 8) * r : (N / 8) * r - N);
}

// The start's k-space pass along y (S_DELTA): the y transform of delta (unless delta(k)
// is already stored), delta(k) and S_-1 = delta/b stored, Z[delta/b] with two inverse y transforms
// (G and Psi_y, as the update kernel leaves them), the first and last stages in registers.
template <int N, int C>
__global__ void __launch_bounds__(KFused<N, C>::T, KFused<N, C>::kMinBlocks) kdelta_fused_kernel(const SArgs a) {
  constexpr int T = KFused<N, C>::T, NB = KFused<N, C>::NB;
  constexpr int H = N / 2;
  extern __shared__ float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);
  float2* s = tw + KFused<N, C>::TAB;
  for (int m = threadIdx.x; m < Plan<N>::kTab; m += T) tw[m] = a.tab[m];
  const Tile t = tile_of<N, C, AX_Y>(blockIdx.x);
  const int col = threadIdx.x % C, j = threadIdx.x / C;
  float2* __restrict__ dkp = t.isQ ? a.dk.Q : a.dk.M;
  float2 d[1][8];
#pragma unroll
  for (int r = 0; r < 8; ++r)
    d[0][r] = dkp[t.base + (size_t)(j + NB * r) * t.ls + (size_t)col * t.cs];
  __syncthreads();   // twiddles
  if (!a.d_is_k) kline_fft<false, N, C, 1>(d, s, tw, j, col);

  const Geometry& g = a.g;
  float2* Sp = t.isQ ? a.sbuf.Q : a.sbuf.M;
  float2 v[2][8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int ky = j + NB * r;
    int ix, kz;
    if (!t.isQ) { ix = t.a; kz = t.c0 + col; } else { ix = t.c0 + col; kz = H; }
    const int mx = (ix < H) ? ix : ix - N;
    const float kx = g.kf * mx, kyf = g.kf * line_freq<N>((float)j, r), kzf = g.kf * kz;
    const float k2 = kx * kx + kyf * kyf + kzf * kzf;
    const float kdy = (r == 4 && j == 0) ? 0.f : kyf;
    const size_t gi = t.base + (size_t)ky * t.ls + (size_t)col * t.cs;
    float2 dk = d[0][r];
    if (!a.d_is_k) {
      if (a.lognormal && ix == 0 && ky == 0 && kz == 0) dk.x -= (float)(a.red[RED_SUM_LOG]);   // N^3 <ln(1+delta)>
      dkp[gi] = dk;
    }
    float2 S = cscale(dk, a.inv_b);
    if (k2 == 0.f) S = make_float2(0.f, 0.f);
    const float inv_k2 = (k2 > 0.f) ? 1.f / k2 : 0.f;
    Sp[gi] = S;
    const float2 iS = cscale(mul_i(S), inv_k2 * g.inv_n3);
    v[0][r] = iS;
    v[1][r] = cscale(iS, kdy);
  }
  kline_fft<true, N, C, 2, 1>(v, s, tw, j, col);
  // G (Psi_x = kdx G, Psi_z = kdz G) in the third field, Psi_y in the second, as the update
  // kernel leaves them
  float2* __restrict__ dy = t.isQ ? a.f[1].Q : a.f[1].M;
  float2* __restrict__ dg = t.isQ ? a.f[2].Q : a.f[2].M;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const size_t gi = t.base + (size_t)(j + NB * r) * t.ls + (size_t)col * t.cs;
    dy[gi] = v[1][r];
    dg[gi] = v[0][r];
  }
}

// The line transform along x of the family, N = E x G with G threads a column and E points a thread:
// a radix-E butterfly per thread straight from global memory (points jb + G r), one exchange through
// shared memory, and E / G radix-G butterflies per thread straight back (points jb + G h + E r; N = 384
// has 24 of them for 16 threads, so threads jb < 8 run a second one).  Tiles of C adjacent columns.
// The three-stage form (8 x M x 8) kept the L1's shared-memory pipe 60% busy and spilled; one exchange
// and two barriers a transform instead of two and four, inverse / forward us: 256 85 / 76 -> 68 / 70,
// 384 268 / 246 -> 227 / 230, 512 608 / 585 -> 585 / 573, 1024 5735 / 5660 -> 5580 / 5590.  What is left
// is load latency: two to four CTAs an SM overlap their load, transform and store phases only partly
// (reading lines at a 2 KB instead of a 1 MB stride changes nothing, 579 / 556 at 512).
template <int N, int C>
struct XLine {
  static constexpr int G = N == 1024 ? 32 : 16;
  static constexpr int E = N / G;              // 16, 24, 32, 32
  static constexpr int H = (E + G - 1) / G;    // second-stage butterflies a thread
  static constexpr int T = G * C;
  // CTAs per SM that the points a thread holds leave registers for (384 at 2, 3 CTAs: 274, 227 us inverse)
  static constexpr int kSM = E == 16 ? 4 : (E == 24 ? 3 : 2);
  static constexpr int kMinBlocks = T > 256 ? 1 : (T == 256 ? kSM : 2 * kSM);
  static constexpr int kTab = (G - 1) * E;     // second-stage twiddles [r - 1][j] = exp(-2 pi i r j / N)
  static constexpr int TAB = (kTab + 1) & ~1;
  static constexpr size_t smem = sizeof(float2) * ((size_t)TAB + (size_t)N * C);
  // row i of the tile, i = E q + r: with 8 columns a 128-byte wavefront holds two rows, whose low bits
  // must differ both for writes (consecutive q) and reads (consecutive r)
  __device__ __forceinline__ static int row(int q, int r, int col) {
    return (E * q + (C == 8 ? r ^ (q & 1) : r)) * C + col;
  }
};
template <int N>
constexpr int kXTab = kFusedMesh<N> ? (XLine<N, 16>::kTab + 1) & ~1 : 0;

// One N-point transform of the tile's columns: ld(x) supplies x[r] = X[jb + G r], st(h, y) takes
// y[r] = Y[jb + G h + E r].  Starts by writing s: a caller that ran it before syncs first.
template <bool INV, int N, int C, class Ld, class St>
__device__ __forceinline__ void xline_io(float2* __restrict__ s, const float2* __restrict__ tw, int jb, int col,
                                         Ld&& ld, St&& st) {
  using X = XLine<N, C>;
  constexpr int E = X::E, G = X::G;
  {
    float2 x[E];
    ld(x);
    DftFine<E, INV>::run(x);
#pragma unroll
    for (int r = 0; r < E; ++r) s[X::row(jb, r, col)] = x[r];
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < X::H; ++h) {
    const int j = jb + G * h;
    if (E % G == 0 || j < E) {
      float2 y[G];
#pragma unroll
      for (int r = 0; r < G; ++r) y[r] = s[X::row(r, j, col)];
#pragma unroll
      for (int r = 1; r < G; ++r) {
        float2 w = tw[(r - 1) * E + j];
        if (INV) w.y = -w.y;
        y[r] = cmul(y[r], w);
      }
      DftFine<G, INV>::run(y);
      st(h, y);
    }
  }
}

// PAIR = false: one component per CTA (blockIdx.y).  PAIR = true (1024): the vector passes between the
// register-fused k-space pass (y) and the fused z pass, which carry vectors in reduced forms: kx and
// kz (kdx, kdz: zero at the Nyquist index) are constant along a y line, so the y pass needs
// A = kdx P_x + kdz P_z and P_y and returns G (Psi_x = kdx G, Psi_z = kdz G) and Psi_y; and the
// observer offset dy (a fixed line of sight's y component) is constant along an x line, so the z
// pass hands over psi^ = r2c_z(psi) and Z^ = r2c_z(dz psi) with P_x = dx psi^, P_y = dy psi^.
// Two CTAs per tile, on adjacent block indices (role = blockIdx.x & 1), so that a field both read
// comes from HBM once and from the L2 the second time:
//   inverse: role 1 transforms Psi_y in the second field in place; role 0 transforms G (third field)
//            twice, Psi_x = IFFT_x(kdx G) into the first and Psi_z = kdz IFFT_x(G) into the third;
//   inverse in C form (a.cform, while the loop runs): the projection pass needs only
//            C = dx Psi_x + dy Psi_y and Psi_z, and dx varies along the x line (the output index)
//            while dy is the tile's constant, so role 0 leaves C = dx IFFT_x(kdx G) + dy IFFT_x(Psi_y)
//            in the first field and role 1 Psi_z = kdz IFFT_x(G) in the fourth (wf): two fields
//            written instead of three, and the projection pass reads two;
//   forward: role 1 leaves P_y = dy FFT_x(psi^) (first field) in the second; role 0 leaves
//            A = kdx FFT_x(dx psi^) + kdz FFT_x(Z^) in the third (its first product goes through the
//            L2 and is read back by the thread that wrote it).
__device__ __forceinline__ uint32_t opaque_u32(uint32_t x) {
  asm volatile("" : "+r"(x));
  return x;
}

template <bool INV, int N, int C, bool PAIR>
__global__ void __launch_bounds__(XLine<N, C>::T, XLine<N, C>::kMinBlocks) xline_kernel(const SArgs a) {
  using X = XLine<N, C>;
  constexpr int H = N / 2, T = X::T, E = X::E, G = X::G;
  extern __shared__ float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);
  float2* s = tw + X::TAB;
  if (!INV && a.skip_flag && *a.skip_flag != 0) return;   // uniform: device loop already converged
  for (int m = threadIdx.x; m < X::kTab; m += T) tw[m] = a.tabx[m];
  const int role = PAIR ? (int)(blockIdx.x & 1) : (int)blockIdx.y;
  // tiles of every y-plane, or (vector passes) of the planes [ybeg, ybeg + ycount): their M tiles
  // (ky, kz block) and the Nyquist tiles that hold their ky columns
  int ti = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  if (PAIR && a.ycount) {
    const int mt = a.ycount * (H / C);
    ti = ti < mt ? a.ybeg * (H / C) + ti : N * (H / C) + a.ybeg / C + (ti - mt);
  }
  const Tile t = tile_of<N, C, AX_X>(ti);
  const int col = threadIdx.x % C, jb = threadIdx.x / C;
  // element offsets fit 32 bits (at most N^3 / 2 complex points per field)
  const uint32_t o0 = (uint32_t)t.base + (uint32_t)(col * t.cs) + (uint32_t)jb * (uint32_t)t.ls;
  const uint32_t ls = (uint32_t)t.ls;
  // element offsets of a load's point r and of a store's point (h, r); stores re-derive the base
  // through an opaque copy, so no offset is kept live across a transform
  auto off_ld = [&](uint32_t base, int r) { return base + (uint32_t)(G * r) * ls; };
  auto off_st = [&](uint32_t base, int h, int r) { return base + (uint32_t)(G * h + E * r) * ls; };
  auto load = [&](const float2* __restrict__ P) {
    return [=, &off_ld](float2 (&x)[E]) {
#pragma unroll
      for (int r = 0; r < E; ++r) x[r] = P[off_ld(o0, r)];
    };
  };
  auto store = [&](float2* __restrict__ P, float scale) {
    return [=, &off_st](int h, const float2 (&y)[G]) {
      const uint32_t o = opaque_u32(o0);
#pragma unroll
      for (int r = 0; r < G; ++r) P[off_st(o, h, r)] = cscale(y[r], scale);
    };
  };
  const Geometry& g = a.g;
  const bool cf = PAIR && INV && a.cform && !(a.loop_flag && *a.loop_flag == 1);
  if (!PAIR || (INV && role == 1 && !cf)) {
    float2* __restrict__ P = t.isQ ? a.f[role].Q : a.f[role].M;
    xline_io<INV, N, C>(s, tw, jb, col, load(P), store(P, 1.f));
    return;
  }
  float2* __restrict__ P0 = t.isQ ? a.f[0].Q : a.f[0].M;
  float2* __restrict__ P1 = t.isQ ? a.f[1].Q : a.f[1].M;
  float2* __restrict__ P2 = t.isQ ? a.f[2].Q : a.f[2].M;
  const float dy = g.los_mode == 1 ? g.los.y : g.off[N + (t.isQ ? t.c0 + col : t.a)];
  if (!INV && role == 1) {   // P_y = dy FFT_x(psi^)
    xline_io<INV, N, C>(s, tw, jb, col, load(P0), store(P1, dy));
    return;
  }
  const float kf = g.kf;
  const float kdz = t.isQ ? 0.f : kf * (float)(t.c0 + col);   // M tiles: kz < N/2; Q tiles: kz = N/2
  // the line index i is kx in Fourier space and x in configuration space
  auto kdx = [&](int i) { return i == H ? 0.f : kf * (float)(i < H ? i : i - N); };
  auto dxv = [&](int i) { return g.los_mode == 1 ? g.los.x : g.off[i]; };
  // loads of G scaled by kdx (the inverse's x component)
  auto load_kdx_g = [&](float2 (&x)[E]) {
#pragma unroll
    for (int r = 0; r < E; ++r) x[r] = P2[off_ld(o0, r)];
#pragma unroll
    for (int r = 0; r < E; ++r) x[r] = cscale(x[r], kdx(jb + G * r));
  };
  if (cf) {
    // both roles start on G, so the pair reads it from HBM once
    if (role == 1) {   // Psi_z = kdz IFFT_x(G)
      float2* __restrict__ W = t.isQ ? a.wf.Q : a.wf.M;
      xline_io<INV, N, C>(s, tw, jb, col, load(P2), store(W, kdz));
      return;
    }
    // role 0: Psi_x = IFFT_x(kdx G) parked in the first field, then C = fmaf(dx, Psi_x, dy Psi_y),
    // rounded exactly as the projection pass forms it from the three components
    xline_io<INV, N, C>(s, tw, jb, col, load_kdx_g, store(P0, 1.f));
    __syncthreads();   // s is rewritten by the second transform
    xline_io<INV, N, C>(s, tw, jb, col, load(P1), [&](int h, const float2 (&y)[G]) {   // IFFT_x(Psi_y)
      const uint32_t o = opaque_u32(o0);
#pragma unroll
      for (int r = 0; r < G; ++r) {
        const float2 x = P0[off_st(o, h, r)];   // this thread's own Psi_x
        const float d = dxv(jb + G * h + E * r);
        P0[off_st(o, h, r)] = make_float2(fmaf(d, x.x, dy * y[r].x), fmaf(d, x.y, dy * y[r].y));
      }
    });
    return;
  }
  if (INV) {   // three components: Psi_x = IFFT_x(kdx G) into the first field, Psi_z = kdz IFFT_x(G)
    xline_io<INV, N, C>(s, tw, jb, col, load_kdx_g, store(P0, 1.f));
    __syncthreads();   // s is rewritten by the second transform
    xline_io<INV, N, C>(s, tw, jb, col, load(P2), store(P2, kdz));
    return;
  }
  // forward: kdz FFT_x(Z^) into the third field, then A = kdx FFT_x(dx psi^) + that
  xline_io<INV, N, C>(s, tw, jb, col, load(P2), store(P2, kdz));
  __syncthreads();   // s is rewritten by the second transform
  xline_io<INV, N, C>(s, tw, jb, col,
                      [&](float2 (&x)[E]) {
#pragma unroll
                        for (int r = 0; r < E; ++r) x[r] = P0[off_ld(o0, r)];
#pragma unroll
                        for (int r = 0; r < E; ++r) x[r] = cscale(x[r], dxv(jb + G * r));
                      },
                      [&](int h, const float2 (&y)[G]) {   // FFT_x(dx psi^)
                        const uint32_t o = opaque_u32(o0);
#pragma unroll
                        for (int r = 0; r < G; ++r) {
                          const float2 x = P2[off_st(o, h, r)];   // this thread's own kdz FFT_x(Z^)
                          const float k = kdx(jb + G * h + E * r);
                          P2[off_st(o, h, r)] = make_float2(fmaf(k, y[r].x, x.x), fmaf(k, y[r].y, x.y));
                        }
                      });
}

// One tile of the source update (Eq. iterative) from registers: v[0] = A and v[1] = P_y along the y
// line (Fourier x and z, configuration y), dk = delta(k) and sp = S_(n-1) at the thread's 8 points
// (already in Fourier y).  Forward y FFT, S_n = delta/b + beta i k . P_n, the Parseval norms
// (accumulated into d2, s2), Psi_n+1 = i kd S_n / k^2 as G (third field) and Psi_y (second field),
// inverse y FFT, stores.  kx and kz are constant along the y line, so the x and z terms of k . P
// arrive combined, A = kdx P_x + kdz P_z (the forward x pass forms it; FFT_y is linear), and
// Psi_x, Psi_z leave as one field G with Psi_x = kdx G, Psi_z = kdz G (the inverse x pass separates
// them).  s is written first: a caller that used it before syncs first.
template <int N, int C>
__device__ __forceinline__ void kiter_tile(const SArgs& a, const Tile& t, float2 (&v)[2][8], const float2 (&dk)[8],
                                           const float2 (&sp)[8], float2* __restrict__ s,
                                           const float2* __restrict__ tw, int j, int col, float& d2, float& s2) {
  constexpr int H = N / 2;
  const Geometry& g = a.g;
  int ix, kz;
  if (!t.isQ) { ix = t.a; kz = t.c0 + col; } else { ix = t.c0 + col; kz = H; }
  const int mx = (ix < H) ? ix : ix - N;
  const float kx = g.kf * mx, kzf = g.kf * kz;
  const float kdx = (ix == H) ? 0.f : kx;
  const float kdz = (kz == H) ? 0.f : kzf;
  constexpr int NB = KFused<N, C>::NB;
  kline_fft<false, N, C, 2>(v, s, tw, j, col);
  float2* Sp = t.isQ ? a.sbuf.Q : a.sbuf.M;
  const float kxz2 = kx * kx + kzf * kzf, kdxz2 = kdx * kdx + kdz * kdz;
  const float wgt = (kz == 0 || kz == H) ? 1.f : 2.f;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int ky = j + NB * r;
    const float kyf = g.kf * line_freq<N>((float)j, r);
    const float k2 = kxz2 + kyf * kyf;
    const float kdy = (r == 4 && j == 0) ? 0.f : kyf;
    const float2 pa = v[0][r], py = v[1][r];
    const float dre = fmaf(kdy, py.x, pa.x);
    const float dim = fmaf(kdy, py.y, pa.y);
    float2 S = make_float2(fmaf(a.beta, -dim, dk[r].x * a.inv_b), fmaf(a.beta, dre, dk[r].y * a.inv_b));
    if (k2 == 0.f) S = make_float2(0.f, 0.f);
    const float inv_k2 = (k2 > 0.f) ? 1.f / k2 : 0.f;
    const float fac = wgt * (kdxz2 + kdy * kdy) * inv_k2 * inv_k2;
    const float ddx = S.x - sp[r].x, ddy = S.y - sp[r].y;
    d2 = fmaf(fac, ddx * ddx + ddy * ddy, d2);
    s2 = fmaf(fac, S.x * S.x + S.y * S.y, s2);
    Sp[t.base + (size_t)ky * t.ls + (size_t)col * t.cs] = S;
    const float2 iS = cscale(mul_i(S), inv_k2 * g.inv_n3);
    v[0][r] = iS;
    v[1][r] = cscale(iS, kdy);
  }
  kline_fft<true, N, C, 2, 1>(v, s, tw, j, col);
  float2* __restrict__ dy = t.isQ ? a.f[1].Q : a.f[1].M;
  float2* __restrict__ dg = t.isQ ? a.f[2].Q : a.f[2].M;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const size_t gi = t.base + (size_t)(j + NB * r) * t.ls + (size_t)col * t.cs;
    dy[gi] = v[1][r];
    dg[gi] = v[0][r];
  }
}

// The tile's four inputs straight from global memory: A (third field), P_y (second), delta(k), S.
template <int N, int C>
__device__ __forceinline__ void kiter_load(const SArgs& a, const Tile& t, int j, int col, float2 (&v)[2][8],
                                           float2 (&dk)[8], float2 (&sp)[8]) {
  const float2* __restrict__ dkp = t.isQ ? a.dk.Q : a.dk.M;
  const float2* __restrict__ spp = t.isQ ? a.sbuf.Q : a.sbuf.M;
  constexpr int NB = KFused<N, C>::NB;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const size_t gi = t.base + (size_t)(j + NB * r) * t.ls + (size_t)col * t.cs;
    v[0][r] = (t.isQ ? a.f[2].Q : a.f[2].M)[gi];
    v[1][r] = (t.isQ ? a.f[1].Q : a.f[1].M)[gi];
    dk[r] = dkp[gi];
    sp[r] = spp[gi];
  }
}

template <int N, int C>
__global__ void __launch_bounds__(KFused<N, C>::T, KFused<N, C>::kMinBlocks) kiter_fused_kernel(const SArgs a) {
  constexpr int T = KFused<N, C>::T;
  extern __shared__ float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);
  float2* s = tw + KFused<N, C>::TAB;
  __shared__ double red_sh[T / 32];
  for (int m = threadIdx.x; m < Plan<N>::kTab; m += T) tw[m] = a.tab[m];
  const Tile t = tile_of<N, C, AX_Y>(blockIdx.x);
  const int col = threadIdx.x % C, j = threadIdx.x / C;
  // every global read of the tile up front
  float2 v[2][8], dk[8], sp[8];
  kiter_load<N, C>(a, t, j, col, v, dk, sp);
  __syncthreads();   // twiddles
  float d2 = 0.f, s2 = 0.f;
  kiter_tile<N, C>(a, t, v, dk, sp, s, tw, j, col, d2, s2);
  double r0 = block_sum((double)d2, red_sh);
  double r1 = block_sum((double)s2, red_sh);
  if (threadIdx.x == 0) {
    a.partials[2 * blockIdx.x + 0] = r0;
    a.partials[2 * blockIdx.x + 1] = r1;
  }
}

// ---- the source update with its inputs streamed by the tensor memory accelerator ---------------
// Persistent CTAs walk the Fourier-x/z tiles; a tile's four inputs (A, P_y, delta(k), S_(n-1): boxes
// of a 3-D map over the half grid M [kx][ky][kz < N/2], at most 256 ky by the tile's kz) land in one
// shared-memory stage by cp.async.bulk.tensor, completing on an mbarrier.  As soon as the threads have
// copied the tile into their registers the next tile's copies are issued into the same stage, so they
// stream in while this tile's transforms and stores run.  The Nyquist tiles (a different layout, 2/(N+2)
// of the data) follow with plain loads.  Each CTA's norms go to its partials.  Every wait is bounded: a wait that
// gives up sets the fault word (the host returns RECON_ERR_TIMEOUT), waits once more for the copies, and the CTA
// returns with NaN norms (the device loop then stops).
// The kernel with direct loads is bound by the L1's data pipe, most of its wavefronts the 32-byte
// segments of its 4-column tiles' rows, and wider tiles leave it one CTA per SM with nothing to overlap.
// Streaming takes the loads off that pipe and overlaps them within one CTA, so the tiles are 8 columns
// (64-byte rows; 16 at 256: 106 us, 4 at 512: 1405 us); a 1024 line leaves room for 4.  Direct against
// streamed, us per update kernel: 256 mesh 114 / 88, 384 457 / 282, 512 1026 / 611 (6.1 TB/s, 0.9 of the
// copy rate), 1024 10460 / 6960.
template <int N>
struct TCols {
  static constexpr int v = N < 1024 ? 8 : 4;
};

template <int N, int C>
struct KTma {
  static constexpr int T = KFused<N, C>::T;
  static constexpr int kBoxes = (N + 255) / 256;                      // boxes of a tile's field, at most 256 rows each
  static constexpr int kRows = N / kBoxes;
  static_assert(N % kBoxes == 0, "equal boxes");
  static constexpr size_t kS = sizeof(float2) * ((size_t)KFused<N, C>::TAB + 2 * (size_t)N * C);
  static constexpr size_t kBufOff = (kS + 127) & ~(size_t)127;
  static constexpr size_t kField = sizeof(float2) * (size_t)N * C;   // one field's tile
  static constexpr size_t kBarOff = kBufOff + 4 * kField;
  static constexpr size_t smem = kBarOff + 16;
  static constexpr uint32_t kTx = 4u * (uint32_t)kField;
  static constexpr int kMinBlocks = smem <= 110 * 1024 ? 2 : 1;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tma_load3(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

__device__ __forceinline__ bool bar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for a phase of the barrier, two seconds of the global timer at most; the last try comes after the limit,
// so a process that was not scheduled meanwhile does not give up on copies that have landed.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  if (bar_try_wait(bar, parity)) return true;
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t0));
  do {
    if (bar_try_wait(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t1));
  } while (t1 - t0 <= 2000000000ull);
  return bar_try_wait(bar, parity);
}

template <int N, int C>
__global__ void __launch_bounds__(KFused<N, C>::T, KTma<N, C>::kMinBlocks) kiter_tma_kernel(const SArgs a,
                                                                       const __grid_constant__ KIterMaps maps) {
  using K = KTma<N, C>;
  constexpr int T = K::T, H = N / 2, MT = N * (H / C), QT = N / C;
  extern __shared__ __align__(128) float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);
  float2* s = tw + KFused<N, C>::TAB;
  const float2* buf = reinterpret_cast<const float2*>(reinterpret_cast<char*>(ssm) + K::kBufOff);
  uint64_t* bar_p = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(ssm) + K::kBarOff);
  __shared__ double red_sh[T / 32];
  bool give_up = false;
  const uint32_t bar = smem_addr(bar_p), dst = smem_addr(buf);
  for (int m = threadIdx.x; m < Plan<N>::kTab; m += T) tw[m] = a.tab[m];
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  __syncthreads();
  const int col = threadIdx.x % C, j = threadIdx.x / C;
  auto issue = [&](int tt) {   // thread 0: the four fields' boxes of tile tt
    const int kx = tt / (H / C), c0 = (tt % (H / C)) * C;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(K::kTx) : "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int h = 0; h < K::kBoxes; ++h)
        if (!(a.drop == 2 && q == 1 && tt == 0))
          tma_load3(dst + (uint32_t)(q * K::kField + h * (K::kField / K::kBoxes)), &maps.m[q], c0, K::kRows * h, kx, bar);
  };
  double dsum = 0.0, ssum = 0.0;   // norms over the CTA's tiles
  float2 v[2][8], dk[8], sp[8];
  uint32_t parity = 0;
  if (threadIdx.x == 0 && (int)blockIdx.x < MT) issue(blockIdx.x);
  for (int tt = blockIdx.x; tt < MT; tt += gridDim.x) {
    const bool ok = bar_wait(bar, parity);
    if (!ok) {
      *a.fault = 1;
      bar_wait(bar, parity);
    }
    parity ^= 1u;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int e = (j + KFused<N, C>::NB * r) * C + col;
      v[0][r] = buf[e];
      v[1][r] = buf[N * C + e];
      dk[r] = buf[2 * N * C + e];
      sp[r] = buf[3 * N * C + e];
    }
    // the stage is free, and so is s
    if (__syncthreads_or(!ok)) {
      give_up = true;
      break;
    }
    if (threadIdx.x == 0 && tt + (int)gridDim.x < MT) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      issue(tt + gridDim.x);
    }
    float d2 = 0.f, s2 = 0.f;
    kiter_tile<N, C>(a, tile_of<N, C, AX_Y>(tt), v, dk, sp, s, tw, j, col, d2, s2);
    dsum += d2;
    ssum += s2;
  }
  if (!give_up) {
    for (int q = blockIdx.x; q < QT; q += gridDim.x) {   // Nyquist tiles: plain loads
      const Tile t = tile_of<N, C, AX_Y>(MT + q);
      kiter_load<N, C>(a, t, j, col, v, dk, sp);
      float d2 = 0.f, s2 = 0.f;
      kiter_tile<N, C>(a, t, v, dk, sp, s, tw, j, col, d2, s2);
      dsum += d2;
      ssum += s2;
    }
  }
  double r0 = block_sum(dsum, red_sh);
  double r1 = block_sum(ssum, red_sh);
  if (threadIdx.x == 0) {
    if (give_up) r0 = r1 = __longlong_as_double(0x7ff8000000000000ll);   // NaN: the loop stops
    a.partials[2 * blockIdx.x + 0] = r0;
    a.partials[2 * blockIdx.x + 1] = r1;
  }
}

// ---- the vector x passes, streamed (256, 384 and 512) ---------------------------------------------
// Three transforms of two fields a tile, in the representations that xline_kernel describes:
//   inverse: IFFT_x(kdx G), IFFT_x(G) and IFFT_x(Psi_y) of the third and second fields, left as C and Psi_z
//            in the first and fourth (C form) or as Psi_x, Psi_y and Psi_z in the first three;
//   forward: FFT_x(dx psi^), FFT_x(psi^) and FFT_x(Z^) of the first and third fields, left as P_y in the second
//            and A in the third.
// Streamed as the source update above is: persistent CTAs whose next tile's fields (boxes of [x][1 y][kz])
// arrive while this tile is transformed, the Nyquist tiles (and every tile where the maps could not be
// built) by plain loads.  The lines go through one exchange buffer one after the other and a thread holds
// 16 points at most, so one or two CTAs fill the SM's threads; each field's stage is refilled as soon as its
// last reader has passed a barrier.  A wait that gives up sets the fault word (the host returns
// RECON_ERR_TIMEOUT) and leaves NaN in its tile; its CTA issues no further copy, waits once more for those on
// their way, and returns.
// The pass is bound by the reads and writes at a stride of a whole plane, each 2 MB page giving a tile one or
// two rows: 16 columns (128-byte rows) against 8 (64 bytes), inverse / forward us, 512 450 / 444 against
// 563 / 537, 384 194 / 192 against 195 / 191, 256 61 / 59 against 62 / 61.  The kernel that one tile's two
// CTAs ran with loads to registers (xline_kernel's pairs) took 585 / 573, 227 / 230 and 68 / 70.  A 1024
// line leaves room for 8 columns (6790 / 6580 us; 4 of all three lines at once 12700 / 12300), so that mesh
// keeps the pairs at 16 (5570 / 5580).
template <int N>
constexpr bool kVLine = kFusedMesh<N> && N < 1024;
constexpr int kVCols = 16;

template <int N, int C>
struct VLine {
  static constexpr int T = KFused<N, C>::T;
  static constexpr int kBoxes = KTma<N, C>::kBoxes, kRows = KTma<N, C>::kRows;
  static constexpr size_t kField = sizeof(float2) * (size_t)N * C;
  static constexpr size_t kBufOff = (sizeof(float2) * (size_t)KFused<N, C>::TAB + kField + 127) & ~(size_t)127;
  static constexpr size_t kBarOff = kBufOff + 2 * kField;
  static constexpr size_t kDxOff = kBarOff + 16;
  static constexpr size_t smem = kDxOff + sizeof(float) * (size_t)N;
  static constexpr int kMinBlocks = T <= 512 ? 2 : 1;   // what shared memory holds
};

template <bool INV, int N, int C>
__global__ void __launch_bounds__(KFused<N, C>::T, VLine<N, C>::kMinBlocks) vline_kernel(const SArgs a,
                                                                                         const __grid_constant__ VLineMaps maps) {
  using K = VLine<N, C>;
  constexpr int T = K::T, H = N / 2, NB = KFused<N, C>::NB;
  extern __shared__ __align__(128) float4 ssm[];
  float2* tw = reinterpret_cast<float2*>(ssm);
  float2* s = tw + KFused<N, C>::TAB;
  const float2* buf = reinterpret_cast<const float2*>(reinterpret_cast<char*>(ssm) + K::kBufOff);
  float* dxs = reinterpret_cast<float*>(reinterpret_cast<char*>(ssm) + K::kDxOff);   // dx of the line's points
  __shared__ int give_up;
  if (!INV && a.skip_flag && *a.skip_flag != 0) return;   // uniform: device loop already converged
  const uint32_t bar = smem_addr(reinterpret_cast<char*>(ssm) + K::kBarOff), dst = smem_addr(buf);
  for (int m = threadIdx.x; m < Plan<N>::kTab; m += T) tw[m] = a.tab[m];
  for (int m = threadIdx.x; m < N; m += T) dxs[m] = a.g.los_mode == 1 ? a.g.los.x : a.g.off[m];
  if (threadIdx.x == 0) {
    give_up = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar + 8) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  __syncthreads();
  // tiles of every y-plane, or of the planes [ybeg, ybeg + ycount): their M tiles (ky, kz block), then
  // the Nyquist tiles that hold their ky columns
  const int ny = a.ycount ? a.ycount : N, mt = ny * (H / C), tiles = mt + ny / C, streamed = maps.on ? mt : 0;
  auto tile_id = [&](int tt) { return tt < mt ? a.ybeg * (H / C) + tt : N * (H / C) + a.ybeg / C + (tt - mt); };
  const int col = threadIdx.x % C, j = threadIdx.x / C;
  auto issue = [&](int q, int tt) {   // thread 0: field q's boxes of tile tt
    if (threadIdx.x != 0 || tt >= streamed) return;
    const int ti = tile_id(tt), ky = ti / (H / C), c0 = (ti % (H / C)) * C;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar + 8 * q), "r"((uint32_t)K::kField) : "memory");
#pragma unroll
    for (int h = 0; h < K::kBoxes; ++h)
      if (!(a.drop == 1 && q == 1 && tt == 0))
        tma_load3(dst + (uint32_t)(q * K::kField + h * (K::kField / K::kBoxes)), &maps.m[q], c0, ky, K::kRows * h, bar + 8 * q);
  };
  const Geometry& g = a.g;
  const bool cf = INV && a.cform && !(a.loop_flag && *a.loop_flag == 1);
  // the line index is kx in Fourier space and x in configuration space
  const float fj = (float)j;
  auto kdx = [&](int r) { return r == 4 && j == 0 ? 0.f : g.kf * line_freq<N>(fj, r); };
  auto dxv = [&](int r) { return dxs[j + NB * r]; };
  uint32_t parity = 0;
  issue(0, blockIdx.x);
  issue(1, blockIdx.x);
  for (int tt = blockIdx.x; tt < tiles; tt += gridDim.x) {
    const int next = tt + gridDim.x;
    const Tile t = tile_of<N, C, AX_X>(tile_id(tt));
    // element offsets fit 32 bits (at most N^3 / 2 complex points per field)
    const uint32_t o0 = (uint32_t)t.base + (uint32_t)(col * t.cs) + (uint32_t)j * (uint32_t)t.ls;
    const uint32_t step = (uint32_t)NB * (uint32_t)t.ls;
    auto at = [&](int f) { return t.isQ ? a.f[f].Q : a.f[f].M; };
    auto wait = [&](int q) {
      if (tt >= streamed || bar_wait(bar + 8 * q, parity)) return true;
      give_up = 1;
      *a.fault = 1;
      bar_wait(bar + 8 * q, parity);   // the copies must not land after the CTA is gone
      return false;
    };
    auto load = [&](int q, int f, bool ok, float2 (&x)[8]) {   // the stage's field q, which is field f
      if (tt < streamed) {
#pragma unroll
        for (int r = 0; r < 8; ++r) x[r] = buf[q * N * C + (j + NB * r) * C + col];
      } else {
        const float2* __restrict__ p = at(f);
#pragma unroll
        for (int r = 0; r < 8; ++r) x[r] = p[o0 + r * step];
      }
      if (!ok) x[0].x = __int_as_float(0x7fc00000);
    };
    const float dy = g.los_mode == 1 ? g.los.y : g.off[N + (t.isQ ? t.c0 + col : t.a)];
    const float kdz = t.isQ ? 0.f : g.kf * (float)(t.c0 + col);   // M tiles: kz < N/2; Q tiles: kz = N/2
    float2 v[1][8], w[8];
    // the first field twice (kdx G, G; dx psi^, psi^), the second once (Psi_y; Z^)
    constexpr int F0 = INV ? 2 : 0, F1 = INV ? 1 : 2;
    bool ok = wait(0);
    load(0, F0, ok, v[0]);
#pragma unroll
    for (int r = 0; r < 8; ++r) v[0][r] = cscale(v[0][r], INV ? kdx(r) : dxv(r));
    kline_fft<INV, N, C, 1, 0>(v, s, tw, j, col);
#pragma unroll
    for (int r = 0; r < 8; ++r) w[r] = v[0][r];
    load(0, F0, ok, v[0]);
    int stop0 = 0, stop = 0;   // give_up, each read between two barriers with no wait in between
    kline_fft<INV, N, C, 1, 1>(v, s, tw, j, col, [&] {
      stop0 = give_up;
      if (!stop0) issue(0, next);
    });
    {
      float2* __restrict__ P = !INV ? at(1) : (cf ? (t.isQ ? a.wf.Q : a.wf.M) : at(2));
      const float sc = INV ? kdz : dy;
#pragma unroll
      for (int r = 0; r < 8; ++r) P[o0 + r * step] = cscale(v[0][r], sc);
    }
    ok = wait(1);
    load(1, F1, ok, v[0]);
    kline_fft<INV, N, C, 1, 0>(v, s, tw, j, col, [&] {
      stop = give_up;
      if (!stop) issue(1, next);
    });
    float2* __restrict__ P0 = at(INV ? 0 : 2);
    if (cf) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float d = dxv(r);
        P0[o0 + r * step] = make_float2(fmaf(d, w[r].x, dy * v[0][r].x), fmaf(d, w[r].y, dy * v[0][r].y));
      }
    } else if (INV) {
      float2* __restrict__ P1 = at(1);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        P0[o0 + r * step] = w[r];
        P1[o0 + r * step] = v[0][r];
      }
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float k = kdx(r);
        const float2 x = cscale(v[0][r], kdz);
        P0[o0 + r * step] = make_float2(fmaf(k, w[r].x, x.x), fmaf(k, w[r].y, x.y));
      }
    }
    if (stop) {
      if (!stop0 && next < streamed) bar_wait(bar, parity ^ 1u);   // the next tile's first field is on its way
      break;
    }
    if (tt < streamed) parity ^= 1u;
    __syncthreads();   // s is free
  }
}

// Stage twiddle tables of the N-point (strided passes) and N/2-point (Z pass) plans, built once
// from the float32 table of exp(-2 pi i m / N) that the host computed in float64.
template <int N>
__global__ void build_tables_kernel(const float2* __restrict__ tw, float2* tabS, float2* tabZ) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
  Plan<N>::template fill<1>(tabS, tw, tid, nthr);
  Plan<N / 2>::template fill<2>(tabZ, tw, tid, nthr);
  if constexpr (kFusedMesh<N>) {   // the x lines' second-stage twiddles behind the N-point plan's
    using X = XLine<N, 16>;
    float2* tx = tabS + ((Plan<N>::kTab + 1) & ~1);
    for (int e = tid; e < X::kTab; e += nthr) tx[e] = tw[(1 + e / X::E) * (e % X::E)];
  }
}

// ------------------------------------------------------------------------------------------------
// Launch tables
// ------------------------------------------------------------------------------------------------
// CTAs of a persistent kernel: as many as the device holds at once.
static inline cudaError_t persistent_grid(const void* k, int threads, size_t smem, int* grid) {
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sm = 0, occ = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem)) != cudaSuccess) return e;
  if (occ < 1) return cudaErrorInvalidConfiguration;
  *grid = occ * sm;
  return cudaSuccess;
}

template <int N>
struct MeshImpl {
  static constexpr int kZBlocks = N * N / kZWarps;   // rows / warps per CTA: upper bound of the Z grid
  template <int M_, int NARROW = 0>
  static constexpr int sblocks() {
    return N * ((N / 2) / SCols<N, M_, NARROW>::v) + N / SCols<N, M_, NARROW>::v;
  }
  static constexpr int kSBlocks = sblocks<S_ITER>();   // grid of the k-space pass (its partials)

  // persistent Z launch: exactly as many CTAs as fit on the device at once (occupancy x SMs),
  // never more than one row per warp
  template <int M_, int NC_>
  static cudaError_t zlaunch(const ZArgs& a, cudaStream_t st, int* grid_out) {
    static int grid = 0;
    const size_t smem = zpass_smem<N, NC_>(M_);
    const void* k = (const void*)zpass_kernel<N, M_, NC_>;
    if (grid == 0) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      int dev = 0, sm = 0, occ = 0;
      if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
      if ((e = cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kZThreads, smem)) != cudaSuccess) return e;
      if (occ < 1) return cudaErrorInvalidConfiguration;
      grid = occ * sm < kZBlocks ? occ * sm : kZBlocks;
    }
    if (grid_out) *grid_out = grid;
    void* args[] = {const_cast<ZArgs*>(&a)};
    return cudaLaunchKernel(k, dim3(grid), dim3(kZThreads), args, smem, st);
  }

  template <int M_>
  static cudaError_t zfused(const ZArgs& a, cudaStream_t st, int* grid_out) {
    if constexpr (kFusedMesh<N>) {
      static int grid = 0;
      const void* k = (const void*)zfused_kernel<N, M_>;
      const size_t smem = ZRow<N>::smem;
      if (grid == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        int dev = 0, sm = 0, occ = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kZThreads, smem)) != cudaSuccess) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        grid = occ * sm < kZBlocks ? occ * sm : kZBlocks;
      }
      if (a.ycount && (a.ybeg < 0 || a.ycount < 0 || a.ybeg + a.ycount > N)) return cudaErrorInvalidValue;
      const int rows_blocks = a.ycount ? (N * a.ycount + kZWarps - 1) / kZWarps : kZBlocks;
      const int g = grid < rows_blocks ? grid : rows_blocks;
      if (grid_out) *grid_out = g;
      void* args[] = {const_cast<ZArgs*>(&a)};
      return cudaLaunchKernel(k, dim3(g), dim3(kZThreads), args, smem, st);
    }
    return cudaErrorInvalidValue;
  }

  static cudaError_t zdelta_fused(const ZArgs& a, cudaStream_t st, int* grid_out) {
    if constexpr (kFusedMesh<N>) {
      static int grid = 0;
      const void* k = (const void*)zdelta_kernel<N>;
      if (grid == 0) {
        int g = 0;
        const cudaError_t e = persistent_grid(k, kZThreads, ZDeltaRow<N>::smem, &g);
        if (e != cudaSuccess) return e;
        grid = g < kZBlocks ? g : kZBlocks;
      }
      if (grid_out) *grid_out = grid;
      void* args[] = {const_cast<ZArgs*>(&a)};
      return cudaLaunchKernel(k, dim3(grid), dim3(kZThreads), args, ZDeltaRow<N>::smem, st);
    }
    return cudaErrorInvalidValue;
  }

  static cudaError_t zpass(int mode, int nc, const ZArgs& a, cudaStream_t st, int* grid_out) {
    if constexpr (kFusedMesh<N>) {
      if (mode == Z_DELTA && nc == 2 && !a.generic && a.ntap <= ZDeltaRow<N>::KT) return zdelta_fused(a, st, grid_out);
      if (nc == 3 && !a.generic) {
        if (mode == Z_PROJ) return zfused<Z_PROJ>(a, st, grid_out);
        if (mode == Z_FINAL) return zfused<Z_FINAL>(a, st, grid_out);
        if (mode == Z_RADIAL) return zfused<Z_RADIAL>(a, st, grid_out);
        if (mode == Z_WARM && a.clevel >= 1) return zfused<Z_WARM>(a, st, grid_out);
        if (mode == Z_USTART) return zfused<Z_USTART>(a, st, grid_out);
      }
    }
#define RG_Z(M_, NC_) \
  if (mode == M_ && nc == NC_) return zlaunch<M_, NC_>(a, st, grid_out);
    RG_Z(Z_FWD, 1) RG_Z(Z_INV, 1) RG_Z(Z_DELTA, 2) RG_Z(Z_PROJ, 3) RG_Z(Z_FINAL, 3) RG_Z(Z_USTART, 3)
    RG_Z(Z_RADIAL, 3) RG_Z(Z_WARM, 3)
#undef RG_Z
    return cudaErrorInvalidValue;
  }

  template <int M_, int NC_, int AX_, int NARROW = 0>
  static cudaError_t slaunch(const SArgs& a, cudaStream_t st, int ncomp) {
    const size_t smem = spass_smem<N, M_, NARROW>((M_ == S_DELTA || M_ == S_ITER) ? 3 : NC_);
    const void* k = (const void*)spass_kernel<N, M_, NC_, AX_, NARROW>;
    static bool attr = false;
    if (!attr) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      attr = true;
    }
    void* args[] = {const_cast<SArgs*>(&a)};
    return cudaLaunchKernel(k, dim3(sblocks<M_, NARROW>(), ncomp), dim3(SThreads<N, M_, NARROW>::v), args, smem,
                            st);
  }

  static int vmap_cols() {
    if constexpr (kVLine<N>) return kVCols;
    return 0;
  }
  static int kmap_cols() {
    if constexpr (kFusedMesh<N>) return TCols<N>::v;
    return 0;
  }

  static cudaError_t klaunch(const SArgs& a, cudaStream_t st) {
    if constexpr (kFusedMesh<N>) {
      constexpr int C = SCols<N, S_ITER>::v;
      if (a.tmaps) {   // inputs streamed by TMA into persistent CTAs
        constexpr int CT = TCols<N>::v;
        using K = KTma<N, CT>;
        const void* k = (const void*)kiter_tma_kernel<N, CT>;
        static int grid = 0;
        if (grid == 0) {
          const cudaError_t e = persistent_grid(k, K::T, K::smem, &grid);
          if (e != cudaSuccess) return e;
        }
        if (a.npart) *a.npart = grid;
        void* args[] = {const_cast<SArgs*>(&a), const_cast<KIterMaps*>(a.tmaps)};
        return cudaLaunchKernel(k, dim3(grid), dim3(K::T), args, K::smem, st);
      }
      const void* k = (const void*)kiter_fused_kernel<N, C>;
      static bool attr = false;
      if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KFused<N, C>::smem);
        if (e != cudaSuccess) return e;
        attr = true;
      }
      void* args[] = {const_cast<SArgs*>(&a)};
      return cudaLaunchKernel(k, dim3(sblocks<S_ITER>()), dim3(KFused<N, C>::T), args, KFused<N, C>::smem, st);
    }
    return cudaErrorInvalidValue;
  }

  static cudaError_t dlaunch(const SArgs& a, cudaStream_t st) {
    if constexpr (kFusedMesh<N>) {
      constexpr int C = SCols<N, S_DELTA>::v;
      const void* k = (const void*)kdelta_fused_kernel<N, C>;
      static bool attr = false;
      if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KFused<N, C>::smem);
        if (e != cudaSuccess) return e;
        attr = true;
      }
      void* args[] = {const_cast<SArgs*>(&a)};
      return cudaLaunchKernel(k, dim3(sblocks<S_DELTA>()), dim3(KFused<N, C>::T), args, KFused<N, C>::smem, st);
    }
    return cudaErrorInvalidValue;
  }

  // x lines of the family: C = 16 (128-byte rows) or 8 columns (line tile option); pair: the vector
  // passes of the register-fused k-space path (two CTA kinds on adjacent block indices, see xline_kernel)
  template <int C, bool PAIR>
  static cudaError_t xlaunch_c(bool inv, const SArgs& a, cudaStream_t st, int ncomp) {
    using X = XLine<N, C>;
    const void* k = inv ? (const void*)xline_kernel<true, N, C, PAIR> : (const void*)xline_kernel<false, N, C, PAIR>;
    static bool attr[2] = {false, false};
    if (!attr[inv]) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X::smem);
      if (e != cudaSuccess) return e;
      attr[inv] = true;
    }
    const int ny = PAIR && a.ycount ? a.ycount : N;
    if (PAIR && a.ycount && (ny % C || a.ybeg % C || a.ybeg < 0 || a.ybeg + ny > N)) return cudaErrorInvalidValue;
    SArgs ax = a;
    ax.tabx = a.tab + ((Plan<N>::kTab + 1) & ~1);
    void* args[] = {&ax};
    const int tiles = ny * ((N / 2) / C) + ny / C;
    // pairs: the two CTAs of a tile on adjacent block indices; single fields: components along y
    const dim3 grid = PAIR ? dim3(2 * tiles) : dim3(tiles, ncomp);
    return cudaLaunchKernel(k, grid, dim3(X::T), args, X::smem, st);
  }
  static cudaError_t xlaunch(bool inv, const SArgs& a, cudaStream_t st, int ncomp, bool pair) {
    if constexpr (kFusedMesh<N>) {
      if constexpr (!kVLine<N>)
        if (pair) return a.narrow ? xlaunch_c<8, true>(inv, a, st, ncomp) : xlaunch_c<16, true>(inv, a, st, ncomp);
      return xlaunch_c<16, false>(inv, a, st, ncomp);
    }
    return cudaErrorInvalidValue;
  }

  // the vector x passes: persistent CTAs over the tiles of all y-planes or of a batch of them
  template <bool INV>
  static cudaError_t vlaunch(const SArgs& a, cudaStream_t st) {
    if constexpr (kVLine<N>) {
      constexpr int C = kVCols;
      using K = VLine<N, C>;
      if (a.ycount && (a.ycount % C || a.ybeg % C || a.ybeg < 0 || a.ybeg + a.ycount > N)) return cudaErrorInvalidValue;
      const void* k = (const void*)vline_kernel<INV, N, C>;
      static int grid = 0;
      if (grid == 0) {
        const cudaError_t e = persistent_grid(k, K::T, K::smem, &grid);
        if (e != cudaSuccess) return e;
      }
      VLineMaps none{};
      const int ny = a.ycount ? a.ycount : N, tiles = ny * ((N / 2) / C) + ny / C;
      void* args[] = {const_cast<SArgs*>(&a), a.vmaps ? const_cast<VLineMaps*>(&a.vmaps[INV]) : &none};
      return cudaLaunchKernel(k, dim3(tiles < grid ? tiles : grid), dim3(K::T), args, K::smem, st);
    }
    return cudaErrorInvalidValue;
  }

  static cudaError_t spass(int mode, int nc, int axis, const SArgs& a, cudaStream_t st) {
    if (a.npart) *a.npart = kSBlocks;   // S_ITER with one tile a CTA
    if (nc < 1 || nc > 3) return cudaErrorInvalidValue;
    // plain passes: one component per CTA, components along gridDim.y
    if (mode == S_FWD && axis == AX_Y) return slaunch<S_FWD, 1, AX_Y>(a, st, nc);
    if (mode == S_INV && axis == AX_Y) return slaunch<S_INV, 1, AX_Y>(a, st, nc);
    if (mode == S_FACTOR && axis == AX_Y && nc == 1) return slaunch<S_FACTOR, 1, AX_Y>(a, st, 1);
    if constexpr (kFusedMesh<N>) {
      // the vector x passes next to the register-fused k-space passes carry their representation
      if ((mode == S_FWD || mode == S_INV) && axis == AX_X && !a.generic && nc == 3) {
        if constexpr (kVLine<N>) return mode == S_INV ? vlaunch<true>(a, st) : vlaunch<false>(a, st);
        return xlaunch(mode == S_INV, a, st, nc, true);
      }
      if ((mode == S_FWD || mode == S_INV) && axis == AX_X && !a.narrow && !a.generic)
        return xlaunch(mode == S_INV, a, st, nc, false);
    }
    if (mode == S_FWD && axis == AX_X)
      return a.narrow ? slaunch<S_FWD, 1, AX_X, 1>(a, st, nc) : slaunch<S_FWD, 1, AX_X>(a, st, nc);
    if (mode == S_INV && axis == AX_X)
      return a.narrow ? slaunch<S_INV, 1, AX_X, 1>(a, st, nc) : slaunch<S_INV, 1, AX_X>(a, st, nc);
    if constexpr (kFusedMesh<N>) {
      if (mode == S_DELTA && axis == AX_Y && !a.generic) return dlaunch(a, st);
      if (mode == S_ITER && axis == AX_Y && nc == 3 && !a.generic) return klaunch(a, st);
    }
    if (mode == S_DELTA && axis == AX_Y) return slaunch<S_DELTA, 1, AX_Y>(a, st, 1);
    if (mode == S_ITER && axis == AX_Y && nc == 3) return slaunch<S_ITER, 3, AX_Y>(a, st, 1);
    return cudaErrorInvalidValue;
  }

  static cudaError_t build_tables(const float2* tw, float2* tabS, float2* tabZ, cudaStream_t st) {
    build_tables_kernel<N><<<4, 256, 0, st>>>(tw, tabS, tabZ);
    return cudaGetLastError();
  }

  static const MeshKernels* table() {
    static const MeshKernels t = {N, kZBlocks, kSBlocks, ((Plan<N>::kTab + 1) & ~1) + kXTab<N>, Plan<N / 2>::kTab, kFusedMesh<N> ? 1 : 0,
                                  kmap_cols(), vmap_cols(), &zpass, &spass, &build_tables};
    return &t;
  }
};

}  // namespace RG_KNS
}  // namespace rg
