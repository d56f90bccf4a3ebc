// bricks.cu: brick-sorted particle pipeline for the CIC deposit and the reconstruction shift.
//
// Particles are packed into 16-byte records (per axis: node index << 21 | 21-bit fraction of a cell,
// rounded down; then the weight) and counting-sorted by their 8^3-cell brick.  The deposit
// then gives each brick to one warp, which accumulates the CIC weights (Sec. 3 mass assignment,
// here cloud-in-cell) of its particles into a 9^3 node tile in shared memory and flushes the tile
// with one global atomic per non-zero node.  The shift (Sec. 1, reversing Eq. Lagrange) stages the
// brick's 9^3 nodes of the three Psi components in shared memory and interpolates every particle of
// the brick from there; the results are written in sorted order and gathered back into the catalogue's
// own order by a pass of their own (brick_unsort).
#include "bricks.h"

#include "cic.h"

namespace rg {

namespace {

constexpr int kWarps = 8;                 // warps per CTA in the brick kernels
constexpr int kTile = (kBrickNodes + 3) & ~3;   // a staged component, a multiple of 16 bytes
constexpr uint32_t kFracOne = 1u << kFracBits;
constexpr uint32_t kFracMask = kFracOne - 1;

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// Node index and 21-bit fraction of a grid coordinate u = x scale: T = floor(u 2^21) (scale21 is scale
// 2^21); node = T >> 21 = floor(u) (arithmetic shift, also for negative u), fraction = T mod 2^21.
// Rounding down keeps a point just below the periodic boundary on its own side (its image stays below L,
// where its line of sight points).
__device__ __forceinline__ uint32_t pack_axis(double x, double scale21, int n) {
  const long long T = floor_scaled(x, scale21, 0.0);
  int c = (int)(T >> kFracBits);
  if (c < 0 || c >= n) c = ((c % n) + n) % n;   // outside [0, L): periodic image
  return ((uint32_t)c << kFracBits) | (uint32_t)(T & (long long)kFracMask);
}

template <typename PT>
__device__ __forceinline__ void pack(const PT* __restrict__ pos, long long p, double scale21, int n,
                                     uint32_t (&q)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) q[a] = pack_axis(widen(pos[3 * p + a]), scale21, n);
}

__device__ __forceinline__ uint32_t brick_key(const uint32_t (&q)[3], int nb) {
  const uint32_t bx = (q[0] >> kFracBits) / kBrick, by = (q[1] >> kFracBits) / kBrick,
                 bz = (q[2] >> kFracBits) / kBrick;
  return (bx * (uint32_t)nb + by) * (uint32_t)nb + bz;
}

// Count particles per brick; each particle keeps its brick and its arrival rank in the brick.  The
// positions (and weights) are read here only, once: each particle's packed record is kept in input
// order for the scatter.
template <typename PT>
__global__ void __launch_bounds__(256) count_kernel(const PT* __restrict__ pos, const float* __restrict__ w,
                                                    long long np, double scale, int n, int nb,
                                                    uint32_t* __restrict__ hist, uint32_t* __restrict__ key,
                                                    uint32_t* __restrict__ rank, uint4* __restrict__ pre) {
  const double scale21 = scale * (double)kFracOne;   // exact: a power of two
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    uint32_t q[3];
    pack(pos, p, scale21, n, q);
    const uint32_t k = brick_key(q, nb);
    key[p] = k;
    rank[p] = atomicAdd(hist + k, 1u);
    pre[p] = make_uint4(q[0], q[1], q[2], __float_as_uint(w ? w[p] : 1.f));
  }
}

// Place every particle's record at offs[brick] + rank, its slot, which replaces its key.
__global__ void __launch_bounds__(256) scatter_kernel(const uint4* __restrict__ pre, long long np,
                                                      const uint32_t* __restrict__ offs, uint32_t* __restrict__ key_slot,
                                                      const uint32_t* __restrict__ rank, uint4* __restrict__ rec) {
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += (long long)gridDim.x * blockDim.x) {
    const uint32_t slot = offs[key_slot[p]] + rank[p];
    rec[slot] = pre[p];
    key_slot[p] = slot;
  }
}

// Exclusive scan of m counts: blocks of 1024 (256 threads x 4), then the block sums, then the add.
__global__ void __launch_bounds__(256) scan_blocks_kernel(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                                                          uint32_t* __restrict__ bsum, int m) {
  __shared__ uint32_t wsum[8];
  const int base = blockIdx.x * 1024 + threadIdx.x * 4;
  uint32_t v[4], s = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[j] = (base + j < m) ? in[base + j] : 0u;
    s += v[j];
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  uint32_t woff = 0, tot = 0;
  for (int i = 0; i < 8; ++i) {
    if (i < warp) woff += wsum[i];
    tot += wsum[i];
  }
  uint32_t run = woff + x - s;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (base + j < m) out[base + j] = run;
    run += v[j];
  }
  if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) scan_sums_kernel(uint32_t* __restrict__ bsum, int nblk, uint32_t* __restrict__ total) {
  __shared__ uint32_t wsum[32];
  const int base = threadIdx.x * 4;
  uint32_t v[4], s = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[j] = (base + j < nblk) ? bsum[base + j] : 0u;
    s += v[j];
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  uint32_t woff = 0, tot = 0;
  for (int i = 0; i < 32; ++i) {
    if (i < warp) woff += wsum[i];
    tot += wsum[i];
  }
  uint32_t run = woff + x - s;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (base + j < nblk) bsum[base + j] = run;
    run += v[j];
  }
  if (threadIdx.x == 0) *total = tot;
}

__global__ void __launch_bounds__(256) scan_add_kernel(uint32_t* __restrict__ out, const uint32_t* __restrict__ bsum,
                                                       int m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) out[i] += bsum[i / 1024];
}

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__global__ void __launch_bounds__(kWarps * 32) deposit_kernel(const uint32_t* __restrict__ offs,
                                                              const uint4* __restrict__ rec, int n, int nb,
                                                              float* __restrict__ rho, double* __restrict__ partials) {
  __shared__ float tiles[kWarps][kBrickNodes];
  __shared__ double wsh[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* tile = tiles[warp];
  const int nb3 = nb * nb * nb;
  const float inv = 1.f / (float)kFracOne;
  double wsum = 0.0;
  for (int b = blockIdx.x * kWarps + warp; b < nb3; b += gridDim.x * kWarps) {
    const uint32_t s0 = offs[b], s1 = offs[b + 1];
    if (s0 == s1) continue;
    for (int j = lane; j < kBrickNodes; j += 32) tile[j] = 0.f;
    __syncwarp();
    const int ox = (b / (nb * nb)) * kBrick, oy = ((b / nb) % nb) * kBrick, oz = (b % nb) * kBrick;
    float bw = 0.f;   // this lane's weight in the brick (float64 once per brick, not per particle)
    for (uint32_t i = s0 + lane; i < s1; i += 32) {
      const uint4 r = rec[i];
      const float wv = __uint_as_float(r.w);
      bw += wv;
      const int lx = (int)(r.x >> kFracBits) - ox, ly = (int)(r.y >> kFracBits) - oy, lz = (int)(r.z >> kFracBits) - oz;
      const float tx = (float)(r.x & kFracMask) * inv, ty = (float)(r.y & kFracMask) * inv,
                  tz = (float)(r.z & kFracMask) * inv;
      const float wx0 = wv * (1.f - tx), wx1 = wv * tx, wy0 = 1.f - ty, wy1 = ty, wz0 = 1.f - tz, wz1 = tz;
      const int c = (lx * kBrickHalo + ly) * kBrickHalo + lz;
      constexpr int DY = kBrickHalo, DX = kBrickHalo * kBrickHalo;
      atomicAdd(tile + c, wx0 * wy0 * wz0);
      atomicAdd(tile + c + 1, wx0 * wy0 * wz1);
      atomicAdd(tile + c + DY, wx0 * wy1 * wz0);
      atomicAdd(tile + c + DY + 1, wx0 * wy1 * wz1);
      atomicAdd(tile + c + DX, wx1 * wy0 * wz0);
      atomicAdd(tile + c + DX + 1, wx1 * wy0 * wz1);
      atomicAdd(tile + c + DX + DY, wx1 * wy1 * wz0);
      atomicAdd(tile + c + DX + DY + 1, wx1 * wy1 * wz1);
    }
    wsum += bw;
    __syncwarp();
    for (int j = lane; j < kBrickNodes; j += 32) {
      const float v = tile[j];
      if (v != 0.f) {
        int gx = ox + j / (kBrickHalo * kBrickHalo), gy = oy + (j / kBrickHalo) % kBrickHalo, gz = oz + j % kBrickHalo;
        if (gx >= n) gx -= n;
        if (gy >= n) gy -= n;
        if (gz >= n) gz -= n;
        atomicAdd(rho + ((size_t)gx * n + gy) * n + gz, v);
      }
    }
    __syncwarp();
  }
  wsum = warp_sum_d(wsum);
  if (lane == 0) wsh[warp] = wsum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < kWarps; ++i) s += wsh[i];
    partials[blockIdx.x] = s;
  }
}

// The shifts of particles [p0, p0 + m) from their sorted slots, in catalogue order, and (pos_out) the
// shifted positions; shift, pos_out and pos are those of particle p0.  A particle's result is one 16-byte
// random read; written back scattered, as 12- or 24-byte pieces of sectors, it cost twice (512 mesh, 3e7
// survey tracers: sort and shift 3.42 ms before, 7.4 with positions).
template <typename PT>
__global__ void __launch_bounds__(256) unsort_kernel(const float4* __restrict__ res, const uint32_t* __restrict__ slot,
                                                     long long m, const PT* __restrict__ pos, int periodic, double L,
                                                     float* __restrict__ shift, double* __restrict__ pos_out) {
  __shared__ double slots_sm[8][96];
  double* slots = slots_sm[threadIdx.x >> 5];
  for (long long p0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); p0 < m;
       p0 += (long long)gridDim.x * blockDim.x) {
    const long long pl = p0 + (threadIdx.x & 31), p = pl < m ? pl : m - 1;
    const float4 r = __ldg(res + slot[p]);
    const float d[3] = {r.x, r.y, r.z};
    warp_store3(shift, p0, m, d, reinterpret_cast<float*>(slots));
    if (pos_out) {
      double y[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        y[c] = widen(pos[3 * p + c]) + d[c];
        if (periodic) y[c] = wrap_box(y[c], L);
      }
      warp_store3(pos_out, p0, m, y, slots);
    }
  }
}

// One warp a brick.  The staging is what the pass costs (729 nodes for 16 tracers at 1024 mesh cells a side and
// 3.3e7 tracers): rows go in as two 16-byte pieces and a ninth node, 24 requests a brick instead of 69 of
// 4-byte loads, without registers in between, while the first records and the next brick's bounds are on
// their way.  Shift kernel, us: 1024 mesh, 3.3e7 clustered tracers 13340 / 11650; 512, 3e7 525 / 511.
template <int BYTES>
__device__ __forceinline__ void copy_async(uint32_t dst, const float* src) {
  if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}

__global__ void __launch_bounds__(kWarps * 32) shift_kernel(const uint32_t* __restrict__ offs,
                                                            const uint4* __restrict__ rec, int n, int nb,
                                                            const BrickShiftArgs a, float4* __restrict__ out) {
  extern __shared__ float ssm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* tile = ssm + warp * 3 * kTile;
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile);
  const int nb3 = nb * nb * nb;
  const float inv = 1.f / (float)kFracOne;
  const float Hf = (float)a.H;
  const int step = gridDim.x * kWarps;
  uint32_t n0 = 0, n1 = 0;   // the next brick's records
  int b = blockIdx.x * kWarps + warp;
  if (b < nb3) n0 = offs[b], n1 = offs[b + 1];
  for (; b < nb3; b += step) {
    const uint32_t s0 = n0, s1 = n1;
    if (b + step < nb3) n0 = offs[b + step], n1 = offs[b + step + 1];
    if (s0 == s1) continue;
    uint4 r = rec[s0 + lane < s1 ? s0 + lane : s0];   // on its way while the tile is staged
    const int ox = (b / (nb * nb)) * kBrick, oy = ((b / nb) % nb) * kBrick, oz = (b % nb) * kBrick;
    // a tile's (x, y) rows: 8 nodes as two 16-byte pieces each, then every row's ninth
    constexpr int R = kBrickHalo * kBrickHalo;
    auto row = [&](int r) {
      int gx = ox + r / kBrickHalo, gy = oy + r % kBrickHalo;
      if (gx >= n) gx -= n;
      if (gy >= n) gy -= n;
      return ((size_t)gx * n + gy) * n;
    };
    const int gz8 = oz + kBrick == n ? 0 : oz + kBrick;
#pragma unroll 4
    for (int e = lane; e < 3 * 2 * R; e += 32) {
      const int q = e / (2 * R), k = e % (2 * R);
      copy_async<16>(dst + 4u * (uint32_t)(q * kTile + 4 * k), a.psi[q] + row(k >> 1) + oz + 4 * (k & 1));
    }
#pragma unroll 4
    for (int e = lane; e < 3 * R; e += 32) {
      const int q = e / R, r = e % R;
      copy_async<4>(dst + 4u * (uint32_t)(q * kTile + 8 * R + r), a.psi[q] + row(r) + gz8);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncwarp();
    for (uint32_t i = s0 + lane; i < s1; i += 32) {
      if (i != s0 + lane) r = rec[i];
      const int cx = (int)(r.x >> kFracBits), cy = (int)(r.y >> kFracBits), cz = (int)(r.z >> kFracBits);
      const float tx = (float)(r.x & kFracMask) * inv, ty = (float)(r.y & kFracMask) * inv,
                  tz = (float)(r.z & kFracMask) * inv;
      const int rw = (cx - ox) * kBrickHalo + (cy - oy), lz = cz - oz;
      // node (row, z): 8 row + z, a row's ninth at 8 R + row
      const int c0 = 8 * rw + lz, c1 = lz == kBrick - 1 ? 8 * R + rw : c0 + 1, s1z = lz == kBrick - 1 ? 1 : 8;
      const float cw[8] = {(1.f - tx) * (1.f - ty) * (1.f - tz), (1.f - tx) * (1.f - ty) * tz,
                           (1.f - tx) * ty * (1.f - tz),         (1.f - tx) * ty * tz,
                           tx * (1.f - ty) * (1.f - tz),         tx * (1.f - ty) * tz,
                           tx * ty * (1.f - tz),                 tx * ty * tz};
      const int co[8] = {c0, c1, c0 + 8, c1 + s1z, c0 + 8 * kBrickHalo, c1 + s1z * kBrickHalo, c0 + 8 * (kBrickHalo + 1),
                         c1 + s1z * (kBrickHalo + 1)};
      float ps[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc = fmaf(cw[k], tile[q * kTile + co[k]], acc);
        ps[q] = acc;
      }
      float d[3];
      if (a.is_galaxy) {
        float rx, ry, rz;
        if (a.los_mode == 1) {
          rx = a.los.x; ry = a.los.y; rz = a.los.z;
        } else {
          const float dx = fmaf(tx, Hf, a.off[cx]), dy = fmaf(ty, Hf, a.off[n + cy]), dz = fmaf(tz, Hf, a.off[2 * n + cz]);
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
      out[i] = make_float4(d[0], d[1], d[2], 0.f);
    }
    __syncwarp();
  }
}

constexpr int kGrid = 152 * 8;

}  // namespace

size_t brick_scratch_bytes(int n) {
  const size_t nb3 = (size_t)(n / kBrick) * (n / kBrick) * (n / kBrick);
  const size_t ch = (size_t)sort_chunk(n);
  return a256(nb3 * 4) + a256((nb3 + 1) * 4) + a256(4096 * 4) + 2 * a256(ch * 16) + 2 * a256(ch * 4);
}

BrickBuffers brick_buffers(char* base, int n, double L) {
  BrickBuffers b{};
  b.n = n;
  b.nb = n / kBrick;
  b.scale = (double)n / L;
  b.chunk = sort_chunk(n);
  const size_t nb3 = (size_t)b.nb * b.nb * b.nb;
  const size_t ch = (size_t)b.chunk;
  b.hist = reinterpret_cast<uint32_t*>(base);
  base += a256(nb3 * 4);
  b.offs = reinterpret_cast<uint32_t*>(base);
  base += a256((nb3 + 1) * 4);
  b.bsum = reinterpret_cast<uint32_t*>(base);
  base += a256(4096 * 4);
  b.rec = reinterpret_cast<uint4*>(base);
  base += a256(ch * 16);
  b.key = reinterpret_cast<uint32_t*>(base);
  base += a256(ch * 4);
  b.rank = reinterpret_cast<uint32_t*>(base);
  base += a256(ch * 4);
  b.pre = reinterpret_cast<uint4*>(base);
  return b;
}

int brick_grid() { return kGrid; }

cudaError_t brick_sort(const BrickBuffers& b, const void* pos, int dtype, const float* w, long long np, cudaStream_t st) {
  if (np <= 0 || np > b.chunk) return np == 0 ? cudaSuccess : cudaErrorInvalidValue;
  const int m = b.nb * b.nb * b.nb;
  const int nblk = (m + 1023) / 1024;
  if (nblk > 4096) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(b.hist, 0, (size_t)m * 4, st);
  if (e != cudaSuccess) return e;
  long long want = (np + 255) / 256;
  const int blocks = (int)(want < kGrid * 2 ? want : kGrid * 2);
  if (dtype == 0)
    count_kernel<double><<<blocks, 256, 0, st>>>((const double*)pos, w, np, b.scale, b.n, b.nb, b.hist, b.key, b.rank,
                                                  b.pre);
  else
    count_kernel<float><<<blocks, 256, 0, st>>>((const float*)pos, w, np, b.scale, b.n, b.nb, b.hist, b.key, b.rank,
                                                 b.pre);
  scan_blocks_kernel<<<nblk, 256, 0, st>>>(b.hist, b.offs, b.bsum, m);
  scan_sums_kernel<<<1, 1024, 0, st>>>(b.bsum, nblk, b.offs + m);
  scan_add_kernel<<<(m + 255) / 256 < kGrid ? (m + 255) / 256 : kGrid, 256, 0, st>>>(b.offs, b.bsum, m);
  scatter_kernel<<<blocks, 256, 0, st>>>(b.pre, np, b.offs, b.key, b.rank, b.rec);
  return cudaGetLastError();
}

cudaError_t brick_deposit(const BrickBuffers& b, float* rho, double* partials, cudaStream_t st) {
  deposit_kernel<<<kGrid, kWarps * 32, 0, st>>>(b.offs, b.rec, b.n, b.nb, rho, partials);
  return cudaGetLastError();
}

cudaError_t brick_shift(const BrickBuffers& b, const BrickShiftArgs& a, cudaStream_t st) {
  const size_t smem = sizeof(float) * kWarps * 3 * kTile;
  cudaError_t e = cudaFuncSetAttribute((const void*)shift_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  shift_kernel<<<kGrid, kWarps * 32, smem, st>>>(b.offs, b.rec, b.n, b.nb, a, reinterpret_cast<float4*>(b.pre));
  return cudaGetLastError();
}

cudaError_t brick_unsort(const BrickBuffers& b, const BrickShiftArgs& a, long long p0, long long m, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  const long long want = (m + 255) / 256;
  const int blocks = (int)(want < 152 * 16 ? want : 152 * 16);
  const float4* res = reinterpret_cast<const float4*>(b.pre);
  if (a.dtype == 0)
    unsort_kernel<double><<<blocks, 256, 0, st>>>(res, b.key + p0, m, (const double*)a.pos, a.periodic, a.L, a.shift, a.pos_out);
  else
    unsort_kernel<float><<<blocks, 256, 0, st>>>(res, b.key + p0, m, (const float*)a.pos, a.periodic, a.L, a.shift, a.pos_out);
  return cudaGetLastError();
}

}  // namespace rg
