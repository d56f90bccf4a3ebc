// fd.h: kernels of the finite-difference configuration-space method (Sec. 2.1, Eq. mainpot).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "types.h"

namespace rg {

struct FDArgs {
  int n;
  double g;              // mesh spacing L / N
  double beta;           // coefficient of the line-of-sight term (f / b)
  int los_mode;          // 0 radial, 1 fixed
  double3 los;           // fixed line of sight (unit)
  const float* off;      // 3 N node offsets from the observer (radial)
  // powers of two that keep the pairs of float32 inside their range whatever the units
  float sp;              // about 1 / g^2: the operator's sums are formed times sp
  float pre;             // about g: the preconditioner's input times pre, its factor over pre
  float un;              // phi holds the potential over un
};

// Scalars of the BiCGStab solve, on the device: written by the last block of the reduction that forms
// them, read by the kernels behind it.
struct FDState {
  double bnorm, rho, rho_old, alpha, omega, res, tol, true_res;
  int it;                // iterations done
  int done;              // 0 running, 2 |s| small enough (x += alpha ph pending), 1 ended
  unsigned int counter;  // blocks done in the running reduction (zero between kernels)
};

// The kernels of one iteration, in order; each returns at once when the solve has ended (st->done).
// Reductions use partials (2 x 608 doubles).  pre: the vector the preconditioner transforms in place, times scale.
cudaError_t launch_fd_init(const float* delta, float c, double inv_b, float* x, float* r, float* rh, size_t n, FDState* st,
                           double tol, double* partials, cudaStream_t s);
cudaError_t launch_fd_dir(const float* r, const float* v, float* p, float* pre, float scale, size_t n, const FDState* st,
                          cudaStream_t s);
// out = A phi (the 7-point Laplacian plus beta times the line-of-sight stencil of Sec. 2.1, phi = 0
// outside the mesh) and its inner products: mode 0 alpha = rho / (w . out), mode 1 omega = (out . w) /
// (out . out), mode 2 only |A phi - w| / bnorm (out unused).
cudaError_t launch_fd_apply(int mode, const float* phi, float* out, const float* w, const FDArgs& a, FDState* st,
                            double* partials, cudaStream_t s);
cudaError_t launch_fd_s(const float* r, const float* v, float* sv, float* pre, float scale, size_t n, FDState* st,
                        double* partials, cudaStream_t s);
cudaError_t launch_fd_update(float* x, const float* ph, const float* sh, const float* sv, const float* t, const float* rh,
                             float* r, size_t n, FDState* st, double* partials, cudaStream_t s);
// Psi_j = -un (phi(+j) - phi(-j)) / (2 g), phi = 0 outside the mesh; psi holds 3 N^3 values.
cudaError_t launch_fd_gradient(const float* phi, float* psi, const FDArgs& a, cudaStream_t st);
// The preconditioner's Fourier-space factor on the library's half grid (M: [kx][ky][kz < N/2], then
// Q: kz = N/2): 1 / (N^3 lambda(k)), lambda the periodic 7-point Laplacian's eigenvalue
// sum_i (2 cos(k_i g) - 2) / g^2, and -L^2 / (3 pi^2 N^3) at k = 0, over scale; N^2 (N/2 + 1) floats.
cudaError_t launch_fd_factor(float* fac, int n, double L, double scale, cudaStream_t st);

}  // namespace rg
