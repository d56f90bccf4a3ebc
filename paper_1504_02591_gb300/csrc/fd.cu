// fd.cu: the finite-difference configuration-space method of Sec. 2.1 (Eq. mainpot), the paper's
// comparison method, as a matrix-free operator on the GPU.
//
// A phi = grad^2 phi + beta div((grad phi . r) r) with the stencils of Sec. 2.1: the 7-point
// Laplacian over the 6 face neighbours (set A) and, for the line-of-sight term,
//   -2 phi_0 / g^2 + sum_B (x_i^2 / (g^2 r^2) +- x_i / (g r^2)) phi_(+-i)
//                  + sum_C (-1)^p x_i x_j / (2 g^2 r^2) phi_(+-i,+-j)
// (x the node's offset from the observer, r = |x|; B the face and C the edge neighbours; p = 0 when
// the two offsets share their sign).  For a fixed line of sight u the term is
// sum_ij u_i u_j d_i d_j phi with the same second differences and no 1/r term.  phi = 0 outside the
// mesh.  The solver (recon.cu) inverts A with BiCGStab preconditioned by the FFT inverse of the
// periodic 7-point Laplacian; this file holds its kernels.
//
// Arithmetic: float64 runs at 1/64 of the float32 rate on this GPU, and the stencil in float64 took 385
// of 1600 us an iteration at 128^3 for 8 MB of data.  The kernels work in pairs of float32 (hi + lo, sums and
// products with their exact rounding errors carried along: Dekker 1971, Knuth's two-sum), about 45
// bits, and round once to float32 on output; the sums over the mesh keep such pairs per thread and
// continue in float64 per block.  Powers of two (exact) keep them inside float32's range: a node's offsets
// are taken over the largest of them, the operator's sums times about 1 / g^2, the right-hand side over
// about 1 / b.  BiCGStab's scalars live on the device: each reduction's last block forms the scalar the next
// kernel needs, so an iteration runs without the host.
#include "cic.h"
#include "fd.h"

namespace rg {

namespace {

// ---- pairs of float32 --------------------------------------------------------------------------
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ F2 add(F2 a, F2 b) {
  F2 s = two_sum(a.h, b.h);
  s.l = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  return s;
}
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
  F2 p = two_prod(a.h, b.h);
  p.l = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l));
  return p;
}
__device__ __forceinline__ F2 split(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ float round2(F2 a) { return __fadd_rn(a.h, a.l); }

// Running sums of a thread: acc += a b.
__device__ __forceinline__ void acc_prod(F2& acc, float a, float b) {
  const F2 p = two_prod(a, b);
  F2 s = two_sum(acc.h, p.h);
  s.l = __fadd_rn(s.l, __fadd_rn(acc.l, p.l));
  acc = s;
}

// ---- the operator ------------------------------------------------------------------------------
__device__ __forceinline__ float at(const float* __restrict__ p, int n, int x, int y, int z) {
  if ((unsigned)x >= (unsigned)n || (unsigned)y >= (unsigned)n || (unsigned)z >= (unsigned)n) return 0.f;
  return __ldg(p + ((size_t)x * n + y) * n + z);
}

// With D+_d, D-_d the second and first differences along d and E_de the mixed one,
//   A phi = [ sum_d (1 + beta n_d^2) D+_d + beta sum_d (g n_d / r) D-_d
//             + beta / 2 sum_(d<e) n_d n_e E_de - 2 beta (1 - |n|^2) phi_0 ] / g^2,    n = x / r
// (the last term is the rounding of a fixed direction's length; zero for a radial one, and at the
// observer's node, where n = 0, the whole line-of-sight term is zero).
struct Coef {
  F2 b, g, ig2, u[3], k0;   // beta sp, g, 1 / (sp g^2), fixed direction, -2 beta sp (1 - |u|^2)
};

__device__ __forceinline__ float fd_operator(const float* __restrict__ phi, int n, int x, int y, int z, const FDArgs& a,
                                             const Coef& k) {
  const float p0 = at(phi, n, x, y, z);
  F2 acc;
  F2 fp[3];   // sp beta times n_d / r (radial: x_d / r^2) or u_d (fixed)
  const bool rsd = a.beta != 0.0;
  float xs[3] = {0.f, 0.f, 0.f};
  F2 inv = {0.f, 0.f}, gs = k.g;
  if (rsd && a.los_mode != 1) {
    xs[0] = a.off[x];
    xs[1] = a.off[n + y];
    xs[2] = a.off[2 * n + z];
    // lengths over the power of two at or below the largest offset, so that r^2 is 1 to 12
    const int ex = (int)(__float_as_uint(fmaxf(fabsf(xs[0]), fmaxf(fabsf(xs[1]), fabsf(xs[2])))) >> 23);
    const float us = __uint_as_float((uint32_t)(254 - min(ex, 253)) << 23);
#pragma unroll
    for (int d = 0; d < 3; ++d) xs[d] *= us;
    const F2 r2 = add(add(two_prod(xs[0], xs[0]), two_prod(xs[1], xs[1])), two_prod(xs[2], xs[2]));
    if (r2.h > 0.f) {
      const float i0 = __frcp_rn(r2.h);
      const float e = __fmaf_rn(-r2.l, i0, __fmaf_rn(-r2.h, i0, 1.f));
      inv = {i0, __fmul_rn(e, i0)};
      gs = {k.g.h * us, k.g.l * us};
    }
  }
  acc = {0.f, 0.f};
  F2 dp[3], dm[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float f1 = at(phi, n, x + (d == 0), y + (d == 1), z + (d == 2));
    const float f0 = at(phi, n, x - (d == 0), y - (d == 1), z - (d == 2));
    const F2 s = two_sum(f1, f0);
    F2 q = two_sum(s.h, -2.f * p0);
    q.l = __fadd_rn(q.l, s.l);
    dp[d] = q;
    dm[d] = two_sum(f1, -f0);
    acc = add(acc, q);
  }
  acc.h *= a.sp;
  acc.l *= a.sp;
  if (rsd) {
    const bool fixed = a.los_mode == 1;
#pragma unroll
    for (int d = 0; d < 3; ++d) fp[d] = mul(k.b, fixed ? k.u[d] : mul(F2{xs[d], 0.f}, inv));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const F2 xd = fixed ? k.u[d] : F2{xs[d], 0.f};
      acc = add(acc, mul(mul(fp[d], xd), dp[d]));
      if (!fixed) acc = add(acc, mul(mul(fp[d], gs), dm[d]));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int e = d + 1; e < 3; ++e) {
        float f[2][2];
#pragma unroll
        for (int s0 = 0; s0 < 2; ++s0)
#pragma unroll
          for (int s1 = 0; s1 < 2; ++s1) {
            const int o0 = s0 ? -1 : 1, o1 = s1 ? -1 : 1;
            f[s0][s1] = at(phi, n, x + (d == 0 ? o0 : 0), y + (d == 1 ? o0 : (e == 1 ? o1 : 0)), z + (e == 2 ? o1 : 0));
          }
        const F2 pa = two_sum(f[0][0], f[1][1]), pb = two_sum(f[0][1], f[1][0]);
        F2 m = two_sum(pa.h, -pb.h);
        m.l = __fadd_rn(m.l, __fsub_rn(pa.l, pb.l));
        m.h *= 0.5f;
        m.l *= 0.5f;
        const F2 xe = fixed ? k.u[e] : F2{xs[e], 0.f};
        acc = add(acc, mul(mul(fp[d], xe), m));
      }
    if (fixed) acc = add(acc, mul(k.k0, F2{p0, 0.f}));
  }
  return round2(mul(acc, k.ig2));
}

__device__ __forceinline__ Coef coefficients(const FDArgs& a) {
  Coef k;
  k.b = split(a.beta * a.sp);
  k.g = split(a.g);
  k.ig2 = split(1.0 / (a.sp * a.g * a.g));
  k.u[0] = split(a.los.x);
  k.u[1] = split(a.los.y);
  k.u[2] = split(a.los.z);
  k.k0 = split(-2.0 * a.beta * a.sp * (1.0 - (a.los.x * a.los.x + a.los.y * a.los.y + a.los.z * a.los.z)));
  return k;
}

// Block sums of up to three pairs, in float64: partials[3 b + q]; the last block of the grid to finish adds
// them in block order and returns true in its thread 0 with the totals.
__device__ __forceinline__ double block_total(double v) {
  __shared__ double sh[8];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
  return r;
}

template <int Q>
__device__ __forceinline__ bool grid_totals(const F2 (&acc)[Q], double* __restrict__ partials,
                                            unsigned int* __restrict__ counter, double (&tot)[Q]) {
  __shared__ bool last;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const double s = block_total((double)acc[q].h + (double)acc[q].l);
    if (threadIdx.x == 0) partials[Q * blockIdx.x + q] = s;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  const volatile double* vp = partials;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    double s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) s += vp[Q * b + q];
    tot[q] = block_total(s);
  }
  if (threadIdx.x == 0) *counter = 0u;
  return threadIdx.x == 0;
}

constexpr int kGrid = 152 * 4;

// r = r^ = delta / b (delta plus the constant c), x = 0; |r|^2 starts the solver's scalars.
__global__ void __launch_bounds__(256) fd_init_kernel(const float* __restrict__ delta, float c, double inv_b,
                                                      float* __restrict__ x, float* __restrict__ r,
                                                      float* __restrict__ rh, size_t n, FDState* __restrict__ st,
                                                      double tol, double* __restrict__ partials) {
  F2 acc[1] = {{0.f, 0.f}};
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    const float v = (float)((double)(delta[i] + c) * inv_b);
    x[i] = 0.f;
    r[i] = v;
    rh[i] = v;
    acc_prod(acc[0], v, v);
  }
  double tot[1];
  if (grid_totals(acc, partials, &st->counter, tot)) {
    st->bnorm = sqrt(tot[0]);
    st->rho = tot[0];
    st->rho_old = st->alpha = st->omega = 1.0;
    st->res = tot[0] > 0.0 ? 1.0 : 0.0;
    st->tol = tol;
    st->it = 0;
    st->done = st->res > tol ? 0 : 1;
  }
}

// Start of an iteration: p = r + (rho / rho_old)(alpha / omega)(p - omega v) (p = r in the first), and
// its copy for the preconditioner.
__global__ void __launch_bounds__(256) fd_dir_kernel(const float* __restrict__ r, const float* __restrict__ v,
                                                     float* __restrict__ p, float* __restrict__ pre, float scale,
                                                     size_t n, const FDState* __restrict__ st) {
  if (st->done) return;
  const bool first = st->it == 0;
  const F2 bt = split((st->rho / st->rho_old) * (st->alpha / st->omega)), om = split(-st->omega);
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    float y = r[i];
    if (!first) y = round2(add(F2{y, 0.f}, mul(bt, add(F2{p[i], 0.f}, mul(om, F2{v[i], 0.f})))));
    p[i] = y;
    pre[i] = y * scale;
  }
}

// out = A phi and the inner products with w (and with itself); mode 0: alpha = rho / (w . out);
// mode 1: omega = (out . w) / (out . out); mode 2: out - b and its norm (the true residual), always run.
template <int MODE>
__global__ void __launch_bounds__(256) fd_apply_kernel(const float* __restrict__ phi, float* __restrict__ out,
                                                       const float* __restrict__ w, FDArgs a, FDState* __restrict__ st,
                                                       double* __restrict__ partials) {
  if (MODE != 2 && st->done) return;
  const int n = a.n;
  const Coef k = coefficients(a);
  const int total = n * n * n;   // at most 1024^3
  F2 acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int e = blockIdx.x * 256 + threadIdx.x; e < total; e += gridDim.x * 256) {
    const float o = fd_operator(phi, n, e / (n * n), (e / n) % n, e % n, a, k);
    const float ww = w[e];
    if (MODE == 2) {
      const float d = __fsub_rn(o, ww);
      acc_prod(acc[0], d, d);
    } else {
      out[e] = o;
      acc_prod(acc[0], o, ww);
      if (MODE == 1) acc_prod(acc[1], o, o);
    }
  }
  double tot[2];
  if (grid_totals(acc, partials, &st->counter, tot)) {
    if (MODE == 0) st->alpha = st->rho / tot[0];
    if (MODE == 1) st->omega = tot[1] > 0.0 ? tot[0] / tot[1] : 0.0;
    if (MODE == 2) st->true_res = st->bnorm > 0.0 ? sqrt(tot[0]) / st->bnorm : 0.0;
  }
}

// s = r - alpha v and its copy for the preconditioner; ends the solve (with x += alpha ph still to do)
// when |s| is small enough.
__global__ void __launch_bounds__(256) fd_s_kernel(const float* __restrict__ r, const float* __restrict__ v,
                                                   float* __restrict__ s, float* __restrict__ pre, float scale,
                                                   size_t n, FDState* __restrict__ st, double* __restrict__ partials) {
  if (st->done) return;
  const F2 al = split(-st->alpha);
  F2 acc[1] = {{0.f, 0.f}};
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    const float y = round2(add(F2{r[i], 0.f}, mul(al, F2{v[i], 0.f})));
    s[i] = y;
    pre[i] = y * scale;
    acc_prod(acc[0], y, y);
  }
  double tot[1];
  if (grid_totals(acc, partials, &st->counter, tot)) {
    const double res = sqrt(tot[0]) / st->bnorm;
    if (res <= st->tol) {
      st->res = res;
      st->it += 1;
      st->done = 2;   // fd_update adds alpha ph and makes it 1
    }
  }
}

// x += alpha ph + omega sh, r = s - omega t, the next rho = r^ . r and |r|: the iteration's end.
__global__ void __launch_bounds__(256) fd_update_kernel(float* __restrict__ x, const float* __restrict__ ph,
                                                        const float* __restrict__ sh, const float* __restrict__ s,
                                                        const float* __restrict__ t, const float* __restrict__ rh,
                                                        float* __restrict__ r, size_t n, FDState* __restrict__ st,
                                                        double* __restrict__ partials) {
  const int done = st->done;
  if (done == 1) return;
  const double omega = done == 2 ? 0.0 : st->omega;
  const F2 al = split(st->alpha), om = split(omega), mom = split(-omega);
  F2 acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    F2 y = add(F2{x[i], 0.f}, mul(al, F2{ph[i], 0.f}));
    if (done == 0) {
      y = add(y, mul(om, F2{sh[i], 0.f}));
      const float q = round2(add(F2{s[i], 0.f}, mul(mom, F2{t[i], 0.f})));
      r[i] = q;
      acc_prod(acc[0], q, q);
      acc_prod(acc[1], rh[i], q);
    }
    x[i] = round2(y);
  }
  double tot[2];
  if (grid_totals(acc, partials, &st->counter, tot)) {
    if (done == 2) {
      st->done = 1;
    } else {
      const double res = sqrt(tot[0]) / st->bnorm;
      st->it += 1;
      st->res = res;
      st->rho_old = st->rho;
      st->rho = tot[1];
      if (!(res > st->tol) || !isfinite(res) || omega == 0.0) st->done = 1;
    }
  }
}

__global__ void __launch_bounds__(256) fd_gradient_kernel(const float* __restrict__ phi, float* __restrict__ psi,
                                                          FDArgs a) {
  const int n = a.n;
  const size_t total = (size_t)n * n * n;
  const F2 h = split(-0.5 / a.g);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(e / ((size_t)n * n)), y = (int)((e / n) % n), z = (int)(e % n);
    psi[e] = a.un * round2(mul(two_sum(at(phi, n, x + 1, y, z), -at(phi, n, x - 1, y, z)), h));
    psi[total + e] = a.un * round2(mul(two_sum(at(phi, n, x, y + 1, z), -at(phi, n, x, y - 1, z)), h));
    psi[2 * total + e] = a.un * round2(mul(two_sum(at(phi, n, x, y, z + 1), -at(phi, n, x, y, z - 1)), h));
  }
}

// 1 / (N^3 lambda) of the periodic 7-point Laplacian on the half grid, formed once per solve in float64
// (per application it took 231 us at 128^3): [kx][ky][kz < N/2] then the Nyquist plane [kx][ky].
__global__ void __launch_bounds__(256) fd_factor_kernel(float* __restrict__ fac, int n, double L, double scale) {
  const int h = n / 2;
  const size_t nm = (size_t)n * n * h, nq = (size_t)n * n;
  const double g = L / n, n3 = (double)n * n * n * scale;
  const double k0 = -L * L / (3.0 * M_PI * M_PI) / n3;
  extern __shared__ double cs[];   // 2 cos(2 pi m / N) - 2
  for (int m = threadIdx.x; m < n; m += blockDim.x) cs[m] = 2.0 * cospi(2.0 * m / n) - 2.0;
  __syncthreads();
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < nm + nq; e += (size_t)gridDim.x * blockDim.x) {
    int kx, ky, kz;
    if (e < nm) {
      kx = (int)(e / ((size_t)n * h));
      ky = (int)((e / h) % n);
      kz = (int)(e % h);
    } else {
      kx = (int)((e - nm) / n);
      ky = (int)((e - nm) % n);
      kz = h;
    }
    // the sign of a wavenumber does not matter
    const double lam = (cs[kx] + cs[ky] + cs[kz]) / (g * g);
    fac[e] = (float)((kx | ky | kz) == 0 ? k0 : 1.0 / (lam * n3));
  }
}

}  // namespace

cudaError_t launch_fd_init(const float* delta, float c, double inv_b, float* x, float* r, float* rh, size_t n, FDState* st,
                           double tol, double* partials, cudaStream_t s) {
  fd_init_kernel<<<kGrid, 256, 0, s>>>(delta, c, inv_b, x, r, rh, n, st, tol, partials);
  return cudaGetLastError();
}

cudaError_t launch_fd_dir(const float* r, const float* v, float* p, float* pre, float scale, size_t n, const FDState* st,
                          cudaStream_t s) {
  fd_dir_kernel<<<kGrid, 256, 0, s>>>(r, v, p, pre, scale, n, st);
  return cudaGetLastError();
}

cudaError_t launch_fd_apply(int mode, const float* phi, float* out, const float* w, const FDArgs& a, FDState* st,
                            double* partials, cudaStream_t s) {
  if (mode == 0) fd_apply_kernel<0><<<kGrid, 256, 0, s>>>(phi, out, w, a, st, partials);
  else if (mode == 1) fd_apply_kernel<1><<<kGrid, 256, 0, s>>>(phi, out, w, a, st, partials);
  else fd_apply_kernel<2><<<kGrid, 256, 0, s>>>(phi, out, w, a, st, partials);
  return cudaGetLastError();
}

cudaError_t launch_fd_s(const float* r, const float* v, float* sv, float* pre, float scale, size_t n, FDState* st,
                        double* partials, cudaStream_t s) {
  fd_s_kernel<<<kGrid, 256, 0, s>>>(r, v, sv, pre, scale, n, st, partials);
  return cudaGetLastError();
}

cudaError_t launch_fd_update(float* x, const float* ph, const float* sh, const float* sv, const float* t, const float* rh,
                             float* r, size_t n, FDState* st, double* partials, cudaStream_t s) {
  fd_update_kernel<<<kGrid, 256, 0, s>>>(x, ph, sh, sv, t, rh, r, n, st, partials);
  return cudaGetLastError();
}

cudaError_t launch_fd_gradient(const float* phi, float* psi, const FDArgs& a, cudaStream_t st) {
  fd_gradient_kernel<<<152 * 8, 256, 0, st>>>(phi, psi, a);
  return cudaGetLastError();
}

cudaError_t launch_fd_factor(float* fac, int n, double L, double scale, cudaStream_t st) {
  fd_factor_kernel<<<kGrid, 256, n * sizeof(double), st>>>(fac, n, L, scale);
  return cudaGetLastError();
}

}  // namespace rg
