// Setup and bookkeeping kernels: phase-map voxelisation (integer), the BFCS
// body-force field, input validation, FP64 reductions of the residual and the
// translated-averaging accumulation (Eqs. 3.5-3.6).
#include "kernels.h"
#include "resid.cuh"

#include <atomic>
#include <cstddef>

namespace bfcs {

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)((blockDim.x + 31) / 32); ++w) t += red[w];
  return t;   // valid in thread 0
}

static std::atomic<long long> g_launches{0};
void count_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

bool supported_len(int n) {
  switch (n) {
    case 4: case 6: case 8: case 12: case 16: case 24: case 32: case 48: case 64:
    case 96: case 128: case 192: case 256: return true;
    default: return false;
  }
}

constexpr int kRedThreads = 256;

// ---------------------------------------------------------------- a1: phase map
// A voxel with doubled centre 2i+1 (cell coordinates) is inside sphere
// (X, Y, Z, T, phase) when the squared periodic minimum-image distance on the
// doubled grid is <= T; the last containing sphere wins; else phase 0.
__device__ __forceinline__ int min_image2(int v, int n2) {   // v in doubled units, period n2 = 2n
  int d = v % n2;
  if (d < 0) d += n2;
  if (d >= n2 / 2) d -= n2;
  return d;
}

__global__ void k_voxelize(int8_t* out, int nx, int ny, int nz, int cx, int cy, int cz,
                           const int* __restrict__ sph, int nsph) {
  // one thread per voxel of the unit cell; its phase is written to every
  // periodic replica of that voxel in the grid
  extern __shared__ int ssph[];
  const long long ncell = (long long)cx * cy * cz;
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int x = (int)(v % cx), y = (int)((v / cx) % cy), z = (int)(v / ((long long)cx * cy));
  const int ix = 2 * x + 1, iy = 2 * y + 1, iz = 2 * z + 1;
  int ph = 0;
  for (int base = 0; base < nsph; base += 1024) {
    const int cnt = min(1024, nsph - base);
    __syncthreads();
    for (int k = threadIdx.x; k < cnt * 5; k += blockDim.x) ssph[k] = sph[base * 5 + k];
    __syncthreads();
    if (v < ncell) {
      for (int k = 0; k < cnt; ++k) {
        const int* S = ssph + 5 * k;
        const int dx = min_image2(ix - S[0], 2 * cx);
        const int dy = min_image2(iy - S[1], 2 * cy);
        const int dz = min_image2(iz - S[2], 2 * cz);
        if (dx * dx + dy * dy + dz * dz <= S[3]) ph = S[4];
      }
    }
  }
  if (v >= ncell) return;
  const int rx = nx / cx, ry = ny / cy, rz = nz / cz;
  for (int kz = 0; kz < rz; ++kz)
    for (int ky = 0; ky < ry; ++ky)
      for (int kx = 0; kx < rx; ++kx)
        out[((long long)(kz * cz + z) * ny + (ky * cy + y)) * nx + (kx * cx + x)] = (int8_t)ph;
}

cudaError_t launch_voxelize(int8_t* out, int nx, int ny, int nz, int cx, int cy, int cz,
                            const int* sph_dev, int nsph, cudaStream_t s) {
  const long long ncell = (long long)cx * cy * cz;
  const unsigned grid = (unsigned)((ncell + 255) / 256);
  k_voxelize<<<grid, 256, 1024 * 5 * sizeof(int), s>>>(out, nx, ny, nz, cx, cy, cz, sph_dev, nsph);
  count_launches(1);
  return cudaGetLastError();
}

// voxel (x, y, z) of linear index v = x + nx (y + ny z): 32-bit unsigned
// arithmetic when the grid has fewer than 2^32 voxels (`small`), else 64-bit
__device__ __forceinline__ void lin_xyz(long long v, int nx, int ny, bool small, int& x, int& y, int& z) {
  if (small) {
    const unsigned u = (unsigned)v, t = u / (unsigned)nx;
    x = (int)(u - t * (unsigned)nx);
    y = (int)(t % (unsigned)ny);
    z = (int)(t / (unsigned)ny);
  } else {
    x = (int)(v % nx);
    y = (int)((v / nx) % ny);
    z = (int)(v / ((long long)nx * ny));
  }
}

// ---------------------------------------------------------------- a2: body force
// b1 = d phi/d x1, phi = (1 - r^2/a^2)^3 for r < a (Eq. 2.5 form), at voxel
// centres i + 0.5, periodic minimum image about the centre; FP64, mean removed.
// rn = (1/nx, 1/ny, 1/nz) in FP32 for the screen: a product and a quotient can
// round differently only at offsets of exactly half a period, where both images
// are equally far, so the screen's decision is the same.
__device__ __forceinline__ double bf_value(int x, int y, int z, int nx, int ny, int nz, float3 rn, double cx,
                                           double cy, double cz, double a) {
  {
    // cheap FP32 screen: voxels clearly outside the support (beyond a + 1 voxel) are 0
    float fx = (float)x + 0.5f - (float)cx, fy = (float)y + 0.5f - (float)cy, fz = (float)z + 0.5f - (float)cz;
    fx -= (float)nx * rintf(fx * rn.x);
    fy -= (float)ny * rintf(fy * rn.y);
    fz -= (float)nz * rintf(fz * rn.z);
    const float lim = (float)a + 1.0f;
    if (fabsf(fx) > lim || fabsf(fy) > lim || fabsf(fz) > lim) return 0.0;
  }
  double dx = x + 0.5 - cx, dy = y + 0.5 - cy, dz = z + 0.5 - cz;
  dx -= nx * rint(dx / nx);
  dy -= ny * rint(dy / ny);
  dz -= nz * rint(dz / nz);
  const double r2 = dx * dx + dy * dy + dz * dz, a2 = a * a;
  if (!(r2 < a2)) return 0.0;
  const double s = 1.0 - r2 / a2;
  return -6.0 * dx * s * s / a2;
}

constexpr int kBfBlocks = 1024;

__global__ void k_bf_partial(double* part, long long n, int nx, int ny, int nz, double cx, double cy,
                             double cz, double a) {
  __shared__ double red[32];
  double acc = 0.0;
  const bool small = n <= 0xFFFFFFFFLL;
  const float3 rn = make_float3(1.0f / (float)nx, 1.0f / (float)ny, 1.0f / (float)nz);
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    lin_xyz(v, nx, ny, small, x, y, z);
    acc += bf_value(x, y, z, nx, ny, nz, rn, cx, cy, cz, a);
  }
  const double t = block_sum(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void k_sum_parts(double* part, int nparts, double* out, double scale) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[i];
  const double t = block_sum(acc, red);
  if (threadIdx.x == 0) *out = t * scale;
}

template <typename R>
__global__ void k_bf_write(R* b, long long n, int nx, int ny, int nz, double cx, double cy, double cz,
                           double a, const double* mean) {
  const double m = *mean;
  const bool small = n <= 0xFFFFFFFFLL;
  const float3 rn = make_float3(1.0f / (float)nx, 1.0f / (float)ny, 1.0f / (float)nz);
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    lin_xyz(v, nx, ny, small, x, y, z);
    b[v] = (R)(bf_value(x, y, z, nx, ny, nz, rn, cx, cy, cz, a) - m);
    b[n + v] = R(0);
    b[2 * n + v] = R(0);
  }
}

int body_force_scratch(long long) { return kBfBlocks + 1; }

template <typename R>
cudaError_t launch_body_force(R* b, int nx, int ny, int nz, double cx, double cy, double cz, double a,
                              double* scratch, cudaStream_t s) {
  const long long n = (long long)nx * ny * nz;
  k_bf_partial<<<kBfBlocks, kRedThreads, 0, s>>>(scratch, n, nx, ny, nz, cx, cy, cz, a);
  k_sum_parts<<<1, kRedThreads, 0, s>>>(scratch, kBfBlocks, scratch + kBfBlocks, 1.0 / (double)n);
  k_bf_write<R><<<kBfBlocks, kRedThreads, 0, s>>>(b, n, nx, ny, nz, cx, cy, cz, a, scratch + kBfBlocks);
  count_launches(3);
  return cudaGetLastError();
}

// Same three kernels with a caller-chosen block count; the scratch holds
// `blocks` FP64 partial sums and the mean at scratch[blocks].
template <typename R>
cudaError_t launch_body_force_blocks(R* b, int nx, int ny, int nz, double cx, double cy, double cz,
                                     double a, int blocks, double* scratch, cudaStream_t s) {
  const long long n = (long long)nx * ny * nz;
  k_bf_partial<<<blocks, kRedThreads, 0, s>>>(scratch, n, nx, ny, nz, cx, cy, cz, a);
  k_sum_parts<<<1, kRedThreads, 0, s>>>(scratch, blocks, scratch + blocks, 1.0 / (double)n);
  k_bf_write<R><<<blocks, kRedThreads, 0, s>>>(b, n, nx, ny, nz, cx, cy, cz, a, scratch + blocks);
  count_launches(3);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- polarization (Eq. 5.7)
template <typename R>
__global__ void k_polarize(R* tau, const R* eps, const int8_t* phase, PhaseTab<R> tab, long long n) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int ph = phase[v];
    ph = (ph >= 0 && ph < kMaxPhases) ? ph : 0;
    const R l1 = tab.lam1[ph], m2 = R(2) * tab.mu1[ph];
    R e[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) e[c] = eps[c * n + v];
    const R lt = l1 * (e[0] + e[1] + e[2]);
#pragma unroll
    for (int c = 0; c < 6; ++c) tau[c * n + v] = m2 * e[c] + (c < 3 ? lt : R(0));
  }
}

template <typename R>
cudaError_t launch_polarize(R* tau, const R* eps, const int8_t* phase, const PhaseTab<R>& tab, long long n,
                            cudaStream_t s) {
  const long long want = (n + kRedThreads - 1) / kRedThreads;
  const int blocks = (int)std::min<long long>(want, 8LL * 152);
  k_polarize<R><<<std::max(blocks, 1), kRedThreads, 0, s>>>(tau, eps, phase, tab, n);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- validation
constexpr int kValBlocks = 512;

// partials of member blockIdx.y: [8][gridDim.x]: per component sum b_c, sum |b_c|, then
// the phase ids' minimum and maximum
template <typename R>
__global__ void k_validate(const __grid_constant__ ValArgs<R> va, long long n, double* part) {
  __shared__ double red[32];
  __shared__ int smin, smax;
  const int8_t* phase = va.phase[blockIdx.y];
  const R* b = va.b[blockIdx.y];
  part += (long long)blockIdx.y * 8 * gridDim.x;
  if (threadIdx.x == 0) { smin = 127; smax = -128; }
  __syncthreads();
  int lmin = 127, lmax = -128;
  double s[3] = {0, 0, 0}, sa[3] = {0, 0, 0};
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const int ph = phase[v];
    lmin = min(lmin, ph); lmax = max(lmax, ph);
    if (b != nullptr) {
#pragma unroll
      for (int c = 0; c < 3; ++c) { const double x = (double)b[c * n + v]; s[c] += x; sa[c] += fabs(x); }
    }
  }
  atomicMin(&smin, lmin);
  atomicMax(&smax, lmax);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double t = block_sum(s[c], red);
    if (threadIdx.x == 0) part[(2 * c) * gridDim.x + blockIdx.x] = t;
    const double ta = block_sum(sa[c], red);
    if (threadIdx.x == 0) part[(2 * c + 1) * gridDim.x + blockIdx.x] = ta;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    part[6 * gridDim.x + blockIdx.x] = (double)smin;
    part[7 * gridDim.x + blockIdx.x] = (double)smax;
  }
}

// one warp per quantity of member blockIdx.x
__global__ void k_validate_final(const double* part, int nparts, int* iout, double* dout) {
  const int m = blockIdx.x, j = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* p = part + ((long long)m * 8 + j) * nparts;
  if (j < 6) {
    double acc = 0.0;
    for (int i = lane; i < nparts; i += 32) acc += p[i];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0) dout[6 * m + (j & 1) * 3 + j / 2] = acc;
  } else {
    int v = j == 6 ? 127 : -128;
    for (int i = lane; i < nparts; i += 32) v = j == 6 ? min(v, (int)p[i]) : max(v, (int)p[i]);
    for (int off = 16; off > 0; off >>= 1) {
      const int w = __shfl_down_sync(0xffffffffu, v, off);
      v = j == 6 ? min(v, w) : max(v, w);
    }
    if (lane == 0) iout[2 * m + j - 6] = v;
  }
}

int validate_scratch() { return 8 * kValBlocks; }

// All members in two launches (three a member, each a few blocks' latency, took 3% of a
// batch of 64^3 solves); at least four voxels a thread.
template <typename R>
cudaError_t launch_validate(const ValArgs<R>& va, int batch, long long n, int* iout, double* dout, double* scratch,
                            cudaStream_t s) {
  const int blocks = (int)std::max<long long>(1, std::min<long long>(kValBlocks, n / (4 * kRedThreads)));
  k_validate<R><<<dim3(blocks, batch), kRedThreads, 0, s>>>(va, n, scratch);
  k_validate_final<<<batch, 256, 0, s>>>(scratch, blocks, iout, dout);
  count_launches(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- residual denominators
// sum over modes with xi != 0 of w |b_hat|^2 (w = 2 for 0 < kx < nx/2: the
// mirrored half of the spectrum), giving the full-spectrum norm of b_hat.
template <typename R>
__global__ void k_bden(const C2<R>* bhat, Geo g, ResidSlot* part, long long b_ms) {
  __shared__ double red[32];
  const int m = blockIdx.y;
  bhat += m * b_ms;
  part += m * gridDim.x;
  const long long modes = (long long)g.nz * g.ny * g.mx;
  double acc = 0.0;
  // 32-bit index arithmetic: a member's spectrum has at most 256 * 256 * 129 modes
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (int)modes; i += gridDim.x * blockDim.x) {
    const int kx = i % g.mx;
    const int r = i / g.mx;
    const int ky = r % g.ny, kz = r / g.ny;
    const int sx = signed_k(kx, g.nx), sy = signed_k(ky, g.ny), sz = signed_k(kz, g.nz);
    if (sx == 0 && sy == 0 && sz == 0) continue;
    const double w = (kx == 0 || 2 * kx == g.nx) ? 1.0 : 2.0;
    const long long gi = (long long)r * g.p + kx;
    if constexpr (sizeof(R) == 4) {
      // |b_hat|^2 of the mode in FP32 (relative 1e-7 is ample for a normaliser), summed in
      // FP64: one FP64 operation per mode instead of twelve on GB300's slow FP64 pipe
      float t = 0.0f;
      for (int c = 0; c < 3; ++c) {
        const C2<R> v = bhat[c * g.cs + gi];
        t += v.x * v.x + v.y * v.y;
      }
      acc += w * (double)t;
    } else {
      for (int c = 0; c < 3; ++c) {
        const C2<R> v = bhat[c * g.cs + gi];
        acc += w * ((double)v.x * v.x + (double)v.y * v.y);
      }
    }
  }
  const double t = block_sum(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x].num = t;
}

__global__ void k_bden_final(const ResidSlot* part, int nparts, IterState* st) {
  __shared__ double red[32];
  const int m = blockIdx.x;
  part += m * nparts;
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[i].num;
  const double t = block_sum(acc, red);
  if (threadIdx.x == 0) st[m].bden = sqrt(t);
}

template <typename R>
cudaError_t launch_bden(const C2<R>* bhat, const Geo& g, ResidSlot* part, IterState* st, cudaStream_t s,
                        int batch, long long b_ms) {
  const int blocks = 512;
  k_bden<R><<<dim3(blocks, batch), kRedThreads, 0, s>>>(bhat, g, part, b_ms);
  k_bden_final<<<batch, kRedThreads, 0, s>>>(part, blocks, st);
  count_launches(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- residual reduction (Eq. 5.11)
__global__ void k_init_states(IterState* st, const Member* mem, double tol) {
  IterState* s = st + blockIdx.x;
  int* w = reinterpret_cast<int*>(s);
  for (int i = threadIdx.x; i < (int)(offsetof(IterState, resid_last) / sizeof(int)); i += blockDim.x) w[i] = 0;
  if (threadIdx.x == 0) {
    const double t = mem[blockIdx.x].tol;
    s->tol = t >= 0.0 ? t : tol;
    s->maxit = 0;
  }
}
cudaError_t launch_init_states(IterState* st, const Member* mem, int batch, double tol, cudaStream_t s) {
  k_init_states<<<batch, 32, 0, s>>>(st, mem, tol);
  count_launches(1);
  return cudaGetLastError();
}
__global__ void k_set_maxit(IterState* st, int batch, int maxit) {
  for (int m = threadIdx.x; m < batch; m += blockDim.x) st[m].maxit = maxit;
}
cudaError_t launch_set_maxit(IterState* st, int batch, int maxit, cudaStream_t s) {
  k_set_maxit<<<1, 64, 0, s>>>(st, batch, maxit);
  count_launches(1);
  return cudaGetLastError();
}

__global__ void k_resid_final(const __grid_constant__ ResidArgs a) { resid_step(a, blockIdx.x); }

cudaError_t launch_resid_final(const ResidArgs& a, int batch, cudaStream_t s) {
  k_resid_final<<<batch, 1024, 0, s>>>(a);
  count_launches(1);
  return cudaGetLastError();
}

struct SlotIdx { int idx[kMaxBatch]; };

__global__ void k_defect_final(const ResidSlot* part, int nparts, IterState* sts, SlotIdx si, int maxdim) {
  __shared__ double red[32];
  const int j = blockIdx.x;
  part += j * nparts;
  double acc = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) acc += part[i].num;
  const double t = block_sum(acc, red);
  if (threadIdx.x != 0) return;
  IterState* st = sts + si.idx[j];
  const double* s0 = st->tau0;
  const double s0n = sqrt(s0[0] * s0[0] + s0[1] * s0[1] + s0[2] * s0[2] +
                          2.0 * (s0[3] * s0[3] + s0[4] * s0[4] + s0[5] * s0[5]));
  const double den = st->bden + 6.283185307179586 / (double)maxdim * s0n;
  st->resid_final = den > 0.0 ? sqrt(t) / den : sqrt(t);
}

cudaError_t launch_defect_final(const ResidSlot* part, int nparts, IterState* st, const int* idx_host, int batch,
                                int maxdim, cudaStream_t s) {
  SlotIdx si{};
  for (int j = 0; j < batch; ++j) si.idx[j] = idx_host[j];
  k_defect_final<<<batch, kRedThreads, 0, s>>>(part, nparts, st, si, maxdim);
  count_launches(1);
  return cudaGetLastError();
}

bool col_variant_valid(int v, int n) {
  if (v == 0) return true;
  if (v < 0 || v >= kColVariants || n < 32 || !supported_len(n)) return false;
  if (col_variant_tma(v)) return n <= 256;   // one box of n rows (a box edge is at most 256)
  if (!col_variant_swap(v)) return true;
  return n != 64 && n != 256;   // 64 = 8 x 8 and 256 = 16 x 16 have one order only
}

// ---------------------------------------------------------------- a10: translated averaging
// acc layout (30 x N, FP64): <u> 3, <u>^(1) 3, <eps> 6, <eps>^(1) 6, <sigma> 6, <sigma>^(1) 6.
// Members are added in order, each voxel by one thread: the sums stay in registers over
// the members of a launch (a launch per member read and wrote all 30 sums each time): 16 of
// 64^3 943 -> 273 us.  A launch of one member (max_batch = 1) reads and writes the 15 sums
// over inclusions at every voxel too, 1.10 GB instead of 0.87 at 128^3 with a quarter
// inclusions, and takes 196 us where one pass over all 15 fields took 455.
template <typename R>
__global__ void k_accumulate(double* acc, int* hits, const __grid_constant__ AccArgs<R> a, int batch, int nx, int ny,
                             int nz) {
  const long long n = (long long)nx * ny * nz;
  const bool small = n <= 0xFFFFFFFFLL;
  // blockIdx.y: 0 the displacement (3 + 3 sums and the hits), 1 and 2 the strain, 3 and 4
  // the stress, three components each (6 + 6 sums of registers)
  const int part = blockIdx.y;
  const int field0 = part == 0 ? 12 : part <= 2 ? (part - 1) * 3 : 6 + (part - 3) * 3;   // in eps | sig | u
  const int out0 = part == 0 ? 0 : part <= 2 ? 6 + (part - 1) * 3 : 18 + (part - 3) * 3;
  const int in_off = part == 0 ? 3 : 6;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    lin_xyz(v, nx, ny, small, x, y, z);
    double s[3], si[3];
    int h = part == 0 ? hits[v] : 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s[c] = acc[(out0 + c) * n + v];
      si[c] = acc[(out0 + in_off + c) * n + v];
    }
    for (int m = 0; m < batch; ++m) {
      int xs = x - a.sx[m]; if (xs < 0) xs += nx;
      int ys = y - a.sy[m]; if (ys < 0) ys += ny;
      int zs = z - a.sz[m]; if (zs < 0) zs += nz;
      const bool in = a.phase[m][((long long)zs * ny + ys) * nx + xs] != 0;
      const R* f = a.fields[m] + (long long)field0 * n + v;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double val = (double)f[c * n];
        s[c] += val;
        if (in) si[c] += val;
      }
      if (in) ++h;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc[(out0 + c) * n + v] = s[c];
      acc[(out0 + in_off + c) * n + v] = si[c];
    }
    if (part == 0) hits[v] = h;
  }
}

template <typename R>
cudaError_t launch_accumulate(double* acc, int* hits, AccArgs<R> a, int batch, int nx, int ny, int nz,
                              cudaStream_t s) {
  // shifts reduced to [0, n) once: the per-voxel translation is then one compare
  for (int m = 0; m < batch; ++m) {
    a.sx[m] = ((a.sx[m] % nx) + nx) % nx;
    a.sy[m] = ((a.sy[m] % ny) + ny) % ny;
    a.sz[m] = ((a.sz[m] % nz) + nz) % nz;
  }
  k_accumulate<R><<<dim3(2 * 152, 5), 256, 0, s>>>(acc, hits, a, batch, nx, ny, nz);
  count_launches(1);
  return cudaGetLastError();
}

__global__ void k_scale(double* acc, long long count, double f) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    acc[i] *= f;
}

cudaError_t launch_scale(double* acc, long long count, double f, cudaStream_t s) {
  k_scale<<<4 * 152, 256, 0, s>>>(acc, count, f);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- small device -> pinned-host reads
// A kernel writes the words straight into the pinned host buffer (its address is
// valid on the device under unified addressing): the read takes no copy engine, so
// it never waits behind large transfers that other streams keep on the engines.
__global__ void k_copy_words(unsigned* dst, const unsigned* src, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
  __threadfence_system();
}
cudaError_t launch_copy_words(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  k_copy_words<<<1, 256, 0, s>>>((unsigned*)dst, (const unsigned*)src, (int)(bytes / sizeof(unsigned)));
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- RVE diagnostic (Def. 2.2)
// Shell maxima of the pointwise norm about a centre on the half-voxel lattice
// (doubled coordinates c2): voxel v lies in shell k = floor(d) where (2d)^2 =
// D2 is an integer, so the shell is decided exactly (k = isqrt(D2) >> 1).  Per
// block the maxima are kept in shared memory as the bit patterns of
// non-negative doubles (their unsigned order is the numeric order), then merged
// into bits[] with one atomicMax per shell: the result does not depend on order.
template <typename R>
__global__ void __launch_bounds__(256) k_radial_max(const R* f, int ncomp, int nx, int ny, int nz, int c2x, int c2y,
                                                  int c2z, int nbins, unsigned long long* bits,
                                                  unsigned long long* counts) {
  extern __shared__ unsigned long long rsh[];      // [nbins] maxima, [nbins] counts
  for (int i = threadIdx.x; i < 2 * nbins; i += blockDim.x) rsh[i] = 0ull;
  __syncthreads();
  const int n = nx * ny * nz;                      // at most 256^3
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const int x = v % nx, y = (v / nx) % ny, z = v / (nx * ny);
    int dx = (2 * x + 1 - c2x) % (2 * nx), dy = (2 * y + 1 - c2y) % (2 * ny), dz = (2 * z + 1 - c2z) % (2 * nz);
    if (dx < 0) dx += 2 * nx;
    if (dy < 0) dy += 2 * ny;
    if (dz < 0) dz += 2 * nz;
    if (dx > nx) dx -= 2 * nx;
    if (dy > ny) dy -= 2 * ny;
    if (dz > nz) dz -= 2 * nz;
    const int D2 = dx * dx + dy * dy + dz * dz;
    int r = (int)sqrtf((float)D2);
    while (r * r > D2) --r;
    while ((r + 1) * (r + 1) <= D2) ++r;
    const int k = r >> 1;
    if (k >= nbins) continue;
    double q = 0.0;
    for (int c = 0; c < ncomp; ++c) {
      const double fc = (double)f[(long long)c * n + v];
      q += (c < 3 ? 1.0 : 2.0) * fc * fc;
    }
    atomicMax(&rsh[k], (unsigned long long)__double_as_longlong(sqrt(q)));
    atomicAdd(&rsh[nbins + k], 1ull);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbins; i += blockDim.x)
    if (rsh[nbins + i] != 0ull) {
      atomicMax(&bits[i], rsh[i]);
      atomicAdd(&counts[i], rsh[nbins + i]);
    }
}

template <typename R>
cudaError_t launch_radial_max(const R* f, int ncomp, int nx, int ny, int nz, const int c2[3], int nbins,
                              unsigned long long* bits, unsigned long long* counts, cudaStream_t s) {
  k_radial_max<R><<<2 * 152, 256, 2 * (size_t)nbins * sizeof(unsigned long long), s>>>(
      f, ncomp, nx, ny, nz, c2[0], c2[1], c2[2], nbins, bits, counts);
  count_launches(1);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- effective moduli (Eqs. 6.1-6.3, 3.2)
// Per member m (blockIdx.y): the 13 FP64 sums  sum sigma_c (6), sum over the
// inclusion voxels (phase != 0) of eps_c (6) and their count, as one partial per
// block in part[(m * gridDim.x + block) * 13 + j]; k_moduli_final adds them in
// block order, so the result does not depend on the launch.
template <typename R>
__global__ void __launch_bounds__(256) k_moduli_partial(ModArgs<R> a, double* part) {
  const int m = blockIdx.y;
  const R* eps = a.eps[m];
  const R* sig = a.sig[m];
  const long long n = a.n;
  double acc[kModSums];
#pragma unroll
  for (int j = 0; j < kModSums; ++j) acc[j] = 0.0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    const bool in = a.phase[v] != 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      acc[c] += (double)sig[c * n + v];
      if (in) acc[6 + c] += (double)eps[c * n + v];
    }
    if (in) acc[12] += 1.0;
  }
  __shared__ double red[kModSums][8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < kModSums; ++j) {
    double t = acc[j];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(0xffffffffu, t, off);
    if (lane == 0) red[j][w] = t;
  }
  __syncthreads();
  if (threadIdx.x < kModSums) {
    double t = 0.0;
    for (int k = 0; k < (int)blockDim.x / 32; ++k) t += red[threadIdx.x][k];
    part[((long long)m * gridDim.x + blockIdx.x) * kModSums + threadIdx.x] = t;
  }
}

__global__ void k_moduli_final(const double* part, int nparts, double* out) {
  const int m = blockIdx.x, j = threadIdx.x;
  if (j >= kModSums) return;
  double t = 0.0;
  for (int k = 0; k < nparts; ++k) t += part[((long long)m * nparts + k) * kModSums + j];
  out[m * kModSums + j] = t;
}

template <typename R>
cudaError_t launch_moduli(const ModArgs<R>& a, int batch, double* part, double* out, cudaStream_t s) {
  k_moduli_partial<R><<<dim3(kModParts, batch), 256, 0, s>>>(a, part);
  k_moduli_final<<<batch, 32, 0, s>>>(part, kModParts, out);
  count_launches(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- precision-ladder helpers
__global__ void k_cast_d2f(float* dst, const double* src, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}
template <bool ADD>
__global__ void k_f2d(const __grid_constant__ F2dArgs a, long long count) {
  double* dst = a.dst[blockIdx.y];
  const float* src = a.src[blockIdx.y];
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = ADD ? dst[i] + (double)src[i] : (double)src[i];
}
cudaError_t launch_cast_d2f(float* dst, const double* src, long long count, cudaStream_t s) {
  k_cast_d2f<<<8 * 152, 256, 0, s>>>(dst, src, count);
  count_launches(1);
  return cudaGetLastError();
}
cudaError_t launch_f2d(const F2dArgs& a, int batch, long long count, bool add, cudaStream_t s) {
  const int blocks = (int)std::max<long long>(1, std::min<long long>(8 * 152, (count + 1023) / 1024));
  if (add) k_f2d<true><<<dim3(blocks, batch), 256, 0, s>>>(a, count);
  else k_f2d<false><<<dim3(blocks, batch), 256, 0, s>>>(a, count);
  count_launches(1);
  return cudaGetLastError();
}

__global__ void k_cast_spec(C2<float>* dst, const C2<double>* src, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const C2<double> v = src[i];
    dst[i] = mk<float>((float)v.x, (float)v.y);
  }
}
cudaError_t launch_cast_spec(C2<float>* dst, const C2<double>* src, const Geo& g, int ncomp, cudaStream_t s) {
  k_cast_spec<<<8 * 152, 256, 0, s>>>(dst, src, (long long)ncomp * g.cs);
  count_launches(1);
  return cudaGetLastError();
}

// float-float spectrum -> complex64 (the FP32 phases' copy of the load)
__global__ void k_cast_spec_ff(C2<float>* dst, const C2<ff>* src, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const C2<ff> v = src[i];
    dst[i] = mk<float>((float)v.x, (float)v.y);
  }
}
cudaError_t launch_cast_spec_ff(C2<float>* dst, const C2<ff>* src, const Geo& g, int ncomp, cudaStream_t s) {
  k_cast_spec_ff<<<8 * 152, 256, 0, s>>>(dst, src, (long long)ncomp * g.cs);
  count_launches(1);
  return cudaGetLastError();
}

__global__ void k_stress(const __grid_constant__ StressArgs a, const __grid_constant__ PhaseTab<double> tab, int nx,
                         int ny, int nz) {
  const int m = blockIdx.y;
  double* const sig = a.sig[m];
  if (sig == nullptr) return;                    // a member without this output
  const double* const eps = a.eps[m];
  const int8_t* const phase = a.phase[m];
  const int sx = a.sx[m], sy = a.sy[m], sz = a.sz[m];
  const long long n = (long long)nx * ny * nz;
  const bool small = n <= 0xFFFFFFFFLL;
  // shifts reduced to [0, n) once: the per-voxel translation is then one compare
  const int sxr = ((sx % nx) + nx) % nx, syr = ((sy % ny) + ny) % ny, szr = ((sz % nz) + nz) % nz;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    lin_xyz(v, nx, ny, small, x, y, z);
    int xs = x - sxr; if (xs < 0) xs += nx;
    int ys = y - syr; if (ys < 0) ys += ny;
    int zs = z - szr; if (zs < 0) zs += nz;
    const int ph = phase[((long long)zs * ny + ys) * nx + xs];
    const double e0 = eps[v], e1 = eps[n + v], e2 = eps[2 * n + v];
    const double lt = tab.lam[ph] * (e0 + e1 + e2), m2 = 2.0 * tab.mu[ph];
    sig[v] = lt + m2 * e0;
    sig[n + v] = lt + m2 * e1;
    sig[2 * n + v] = lt + m2 * e2;
    for (int c = 3; c < 6; ++c) sig[c * n + v] = m2 * eps[c * n + v];
  }
}
cudaError_t launch_stress(const StressArgs& a, int batch, const PhaseTab<double>& tab, int nx, int ny, int nz,
                          cudaStream_t s) {
  const long long n = (long long)nx * ny * nz;
  const int blocks = (int)std::max<long long>(1, std::min<long long>(8 * 152, (n + 255) / 256));
  k_stress<<<dim3(blocks, batch), 256, 0, s>>>(a, tab, nx, ny, nz);
  count_launches(1);
  return cudaGetLastError();
}

#define BFCS_INST(R)                                                                              \
  template cudaError_t launch_body_force<R>(R*, int, int, int, double, double, double, double,     \
                                            double*, cudaStream_t);                               \
  template cudaError_t launch_polarize<R>(R*, const R*, const int8_t*, const PhaseTab<R>&, long long,  \
                                          cudaStream_t);                                          \
  template cudaError_t launch_body_force_blocks<R>(R*, int, int, int, double, double, double,      \
                                                   double, int, double*, cudaStream_t);           \
  template cudaError_t launch_validate<R>(const ValArgs<R>&, int, long long, int*, double*, double*, cudaStream_t);                                 \
  template cudaError_t launch_bden<R>(const C2<R>*, const Geo&, ResidSlot*, IterState*,            \
                                      cudaStream_t, int, long long);                              \
  template cudaError_t launch_accumulate<R>(double*, int*, AccArgs<R>, int, int, int, int, cudaStream_t);                                        \
  template cudaError_t launch_moduli<R>(const ModArgs<R>&, int, double*, double*, cudaStream_t);   \
  template cudaError_t launch_radial_max<R>(const R*, int, int, int, int, const int*, int,           \
                                            unsigned long long*, unsigned long long*, cudaStream_t);
BFCS_INST(float)
BFCS_INST(double)
#undef BFCS_INST

}  // namespace bfcs
