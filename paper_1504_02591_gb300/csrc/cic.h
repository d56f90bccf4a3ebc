// cic.h: launchers of the particle kernels and the reduction helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

namespace rg {

struct ShiftArgs {
  const float* psi[3];   // real Psi components, N^3 each
  const float4* psi4;    // or null; the same as (x, y, z, 0) per node
  int n;
  double scale;          // N / L
  double L;
  int is_galaxy;
  float f;               // growth rate of the galaxy RSD term
  int los_mode;          // 0 radial, 1 fixed
  float3 los;            // fixed LOS unit vector
  const float* off;      // 3 N node offsets from the observer, per axis (radial)
  float H;               // cell size: a particle's offset is off[node] + t H, its image in [0, L)
  int periodic;
  float* shift;          // (n, 3) out
  double* pos_out;       // (n, 3) out or null
};

// The rare branches below are calls: inlined, the compiler turns them into predicated float64 operations that
// every particle pays (3e7 float64 positions to the nearest nodes: 652 us so, 330 with calls).
[[maybe_unused]] static __device__ __noinline__ long long floor_far(double x, double s, double c) { return __double2ll_rd(fma(x, s, c)); }
[[maybe_unused]] static __device__ __noinline__ double widen_far(float x) { return (double)x; }

// x in float64 by integer operations (the conversion takes a float64 slot); subnormals, infinities and NaN by
// the conversion.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), e = (u >> 23) & 255u;
  if (e - 1u < 254u || u << 1 == 0)
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (u << 1 ? 0x38000000u : 0u))), (int)(u << 29));
  return widen_far(x);
}

// floor(x s + c) for x s + c as one exact product and sum: a fused multiply-add rounded down onto
// 1.5 x 2^52, whose low mantissa bits are then the integer.  One float64 operation where a product and a
// conversion take two (float64 runs at 1/64 of the float32 rate here, and positions are float64).  c is
// an integer; sums outside +-2^51 (positions hundreds of boxes away) and NaN take the conversion.
__device__ __forceinline__ long long floor_scaled(double x, double s, double c) {
  const double magic = 6755399441055744.0;   // 1.5 x 2^52
  const double v = __fma_rd(x, s, magic + c);
  const long long b = __double_as_longlong(v);
  if ((b >> 52) == 0x433) return b - 0x4338000000000000ll;
  return floor_far(x, s, c);
}

// y - floor(y / L) L, stepped back once more if that rounds to L: a shifted position wrapped into the box.
// Positions in [-L, 2L) take at most one addition (the same value: floor(y / L) is -1, 0 or 1 there, and
// non-negative doubles order as their bits); only others pay the float64 division, which on this GPU
// costs more than the rest of the shift.
__device__ __forceinline__ double wrap_box(double y, double L) {
  const long long b = __double_as_longlong(y);
  if ((unsigned long long)b < (unsigned long long)__double_as_longlong(L)) return y;
  if (b < 0 ? y >= -L : y < L + L) y = b < 0 ? y + L : y - L;
  else y = y - floor(y / L) * L;
  return y >= L ? y - L : y;
}

// Rows of three values of 32 consecutive particles (p0 + lane, those below np) stored through the warp's 96
// slots of shared memory: three full-line stores instead of three strided ones whose partial sectors the
// L2 would have to merge.  Every lane of the warp calls it.
template <typename T>
__device__ __forceinline__ void warp_store3(T* __restrict__ dst, long long p0, long long np, const T (&v)[3],
                                            T* __restrict__ slots) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 3; ++c) slots[3 * lane + c] = v[c];
  __syncwarp();
  const long long left = 3 * (np - p0);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (lane + 32 * c < left) dst[3 * p0 + lane + 32 * c] = slots[lane + 32 * c];
}

constexpr int kDepositBlocks = 152 * 8;

// CIC (or, with ngp, nearest-grid-point) deposit; the weight sum of each block into partials.
cudaError_t launch_deposit(const void* pos, int dtype, const float* w, long long np, int n, double L,
                           float* rho, double* partials, int blocks, cudaStream_t st, int ngp = 0);
// Counts of particles in nbins equal radial shells [rmin, rmax) about obs (counts zeroed by the caller).
cudaError_t launch_radial_hist(const void* pos, int dtype, long long np, double3 obs, double rmin, double rmax,
                               int nbins, unsigned long long* counts, cudaStream_t st);
// FKP weights: wtab (device, nbins + 1 floats) of each particle's shell, wtab[nbins] outside the shells.
cudaError_t launch_fkp(const void* pos, int dtype, long long np, double3 obs, double rmin, double rmax, int nbins,
                       const float* wtab, float* w, cudaStream_t st);
// psi4[i] = (x[i], y[i], z[i], 0), n a multiple of 4.
cudaError_t launch_pack_psi(const float* const psi[3], float4* psi4, size_t n, cudaStream_t st);
cudaError_t launch_shift(const void* pos, int dtype, long long np, const ShiftArgs& a, cudaStream_t st);
// red[dst + q] (=|+=) the sum over b < nblocks of partials[b nq + q], q < nq <= 4, in a fixed order.
// bsum (kFinalizeBlocks x 4 doubles) and counter (zeroed; left zeroed) let several blocks share the
// sum; with nulls one block does it.
constexpr int kFinalizeBlocks = 64;
cudaError_t launch_finalize(const double* partials, int nblocks, int nq, double* red, int dst, int accumulate,
                            cudaStream_t st, double* bsum = nullptr, unsigned int* counter = nullptr);
cudaError_t launch_add_scalar(float* x, size_t n, float v, cudaStream_t st);

// Ratio statistics of the paper's diagnostics (Eq. ratio; Tables 1-3): per block, the number of
// ratios num/den inside [lo, hi] (a zero denominator is outside), their sum and sum of squares in
// float64, and the number of points: partials[4 b + 0..3].
struct RatioArgs {
  const float* num[3];   // radial form: the two vector fields (Psi_real, Psi_est), N^3 each
  const float* den[3];
  int n;
  double scale;          // N / L
  int los_mode;
  float3 los;
  const float* off;      // 3 N node offsets from the observer
  float H;
  double lo, hi;
  double* partials;
};
// (Psi_num . r)/(Psi_den . r) at each particle, both fields CIC-interpolated, r the particle's line
// of sight (its image in [0, L), as in the shift).
cudaError_t launch_radial_ratio(const void* pos, int dtype, long long np, const RatioArgs& a, int blocks,
                                cudaStream_t st);
// num[i] / den[i] over n values.
cudaError_t launch_ratio(const float* num, const float* den, size_t n, double lo, double hi, double* partials,
                         int blocks, cudaStream_t st);

}  // namespace rg
