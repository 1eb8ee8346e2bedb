// Learned warm start / surrogate: a 3D U-net on periodic volumes, trained and
// run by the kernels in this file (BF16 activations and weights, FP32
// accumulation, FP32 master weights, gradients and Adam moments).  The paper
// motivates learned surrogates of the averaged response (Sec. 6, Eqs.
// 6.9-6.10, Fig. 5); the architecture is the project's:
//   widths 32, 32, 32, 48; two circular 3^3 convolutions per level with leaky
//   ReLU (slope 0.1); 2^3 average pooling; 2^3 stride-2 transposed
//   convolutions up (run as a 1^3 convolution to 8 C channels plus a pixel
//   shuffle); skip concatenation [upsampled, skip]; 1^3 head to the 6 strain
//   components.
//
// Activations are channels-last [b][z][y][x][c] BF16.  Convolutions are
// implicit GEMMs on the tensor cores: rows = voxels, columns = output channels,
// K = taps x input channels (3^3 layers: tcgen05, unet_conv.cu; pointwise
// layers: unet_gemm.cu).  A weight gradient is a second GEMM (rows = output channels,
// columns = input channels, K = voxels): tcgen05 for the 3^3 layers with 32 output
// channels, mma.sync for the pointwise ones (unet_wgrad.cu) and for the two 48-channel
// layers (k_wgrad below).  Each block sums a run of voxels, and the blocks' partial sums are
// added in a fixed order (deterministic).
#include "bfcs.h"
#include "unet_kernels.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

namespace bfcs {
namespace net {

__device__ __forceinline__ unsigned ld32(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }

// fine voxel offset of sub-voxel o = 4 oz + 2 oy + ox on a grid of pitch (FX, FY)
__device__ __forceinline__ long long sub_off(int o, int FX, int FY) {
  return ((long long)(o >> 2) * FY + ((o >> 1) & 1)) * FX + (o & 1);
}

// ------------------------------------------------------------------ convolution (forward / data gradient)
// 3^3 circular convolution on the warp-level tensor cores (BFCS_NET_TCGEN05=0),
// operands straight from global memory
constexpr int kConvWarps = 4;
constexpr int kConvNT = 8;   // n8 tiles per block (64 columns)

__global__ void __launch_bounds__(kConvWarps * 32) k_conv(ConvArgs a) {
  chain_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const long long nvox = (long long)a.v.nx * a.v.ny * a.v.nz;
  const int b = blockIdx.z;
  const long long row0 = (long long)blockIdx.x * (kConvWarps * 32) + warp * 32;   // 2 m16 tiles per warp
  const int col0 = blockIdx.y * (kConvNT * 8);
  const int ntiles = min(kConvNT, (a.cout_p - col0) / 8);
  float acc[2][kConvNT][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < kConvNT; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
  // fragment rows g and g + 8 of both m16 tiles (clamped; stores are guarded)
  int cx[4], cy[4], cz[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long r = min(row0 + (q >> 1) * 16 + (q & 1) * 8 + g, nvox - 1);
    cx[q] = (int)(r % a.v.nx);
    cy[q] = (int)((r / a.v.nx) % a.v.ny);
    cz[q] = (int)(r / ((long long)a.v.nx * a.v.ny));
  }
  const bf16* inb = a.in + (long long)b * nvox * a.ldi + a.offi;
  for (int tap = 0; tap < 27; ++tap) {
    const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    const bf16* rp[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      rp[q] = inb + (((long long)wrap(cz[q] + dz, a.v.nz) * a.v.ny + wrap(cy[q] + dy, a.v.ny)) * a.v.nx +
                     wrap(cx[q] + dx, a.v.nx)) * a.ldi;
    const bf16* wt = a.w + (long long)tap * a.cout_p * a.cin;
    for (int kc = 0; kc < a.cin; kc += 16) {
      unsigned af[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        af[i][0] = ld32(rp[2 * i] + kc + 2 * t);
        af[i][1] = ld32(rp[2 * i + 1] + kc + 2 * t);
        af[i][2] = ld32(rp[2 * i] + kc + 2 * t + 8);
        af[i][3] = ld32(rp[2 * i + 1] + kc + 2 * t + 8);
      }
#pragma unroll
      for (int j = 0; j < kConvNT; ++j) {
        if (j < ntiles) {
          const bf16* wr = wt + (long long)(col0 + j * 8 + g) * a.cin + kc + 2 * t;
          const unsigned b0 = ld32(wr), b1 = ld32(wr + 8);
          mma16816(acc[0][j], af[0], b0, b1);
          mma16816(acc[1][j], af[1], b0, b1);
        }
      }
    }
  }
  // epilogue: bias, activation or gate, store
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = q >> 1, h = q & 1;
    const long long r = row0 + i * 16 + h * 8 + g;
    if (r >= nvox) continue;
#pragma unroll
    for (int j = 0; j < kConvNT; ++j) {
      if (j >= ntiles) continue;
      const int col = col0 + j * 8 + 2 * t;
      float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
      if (a.bias != nullptr) {
        v0 += a.bias[col % a.bias_mod];
        v1 += a.bias[(col + 1) % a.bias_mod];
      }
      if (a.act) {
        v0 = v0 > 0.f ? v0 : kSlope * v0;
        v1 = v1 > 0.f ? v1 : kSlope * v1;
      }
      __nv_bfloat162 o = __floats2bfloat162_rn(v0, v1);
      if (a.gate != nullptr) {
        const bf16* y = a.gate + ((long long)b * nvox + r) * a.ldg + a.offg + col;
        if (!(__bfloat162float(y[0]) > 0.f)) o.x = __float2bfloat16(__bfloat162float(o.x) * kSlope);
        if (!(__bfloat162float(y[1]) > 0.f)) o.y = __float2bfloat16(__bfloat162float(o.y) * kSlope);
      }
      bf16* dst = (bf16*)a.out + ((long long)b * nvox + r) * a.ldo + a.offo + col;
      *reinterpret_cast<__nv_bfloat162*>(dst) = o;
    }
  }
}

// ------------------------------------------------------------------ weight gradient
// dW[tap][co][ci] = sum over (b, v) of dY[b][v][co] X[b][v + d_tap][ci] of a 3^3 layer on the
// warp-level tensor cores: the 48-channel layers (0.2% of a gradient's products), and every
// 3^3 layer with BFCS_NET_TCGEN05=0.  Block (chunk, tap): voxels [chunk * rows_per, ...);
// partial[chunk][tap][cout_p][cin] in FP32.
constexpr int kWgRows = 64;

__global__ void __launch_bounds__(128) k_wgrad(WgArgs a) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tap = blockIdx.y;
  const int CP = a.cout_p + 8, XP = a.cin + 8;      // row pitches: 16-byte multiples, conflict-free ldmatrix
  bf16* sD = reinterpret_cast<bf16*>(smraw);        // [64][CP]
  bf16* sX = sD + kWgRows * CP;                     // [64][XP]
  const unsigned sDa = (unsigned)__cvta_generic_to_shared(sD), sXa = (unsigned)__cvta_generic_to_shared(sX);
  const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
  const long long nvox = (long long)a.v.nx * a.v.ny * a.v.nz;
  const long long total = nvox * a.batch;
  const long long start = (long long)blockIdx.x * a.chunk;
  const long long stop = min(start + a.chunk, total);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = a.cout_p / 16;
  float sum[4][4][4] = {};                          // [m16 tile][n8 tile of this warp][4]
  const int dvec = a.cout_p / 8, xvec = a.cin / 8;
  for (long long r0 = start; r0 < stop; r0 += kWgRows) {
    __syncthreads();
    for (int idx = threadIdx.x; idx < kWgRows * (dvec + xvec); idx += blockDim.x) {
      const int row = idx / (dvec + xvec), cv = idx - row * (dvec + xvec);
      const long long gr = r0 + row;
      uint4 val = make_uint4(0u, 0u, 0u, 0u);
      if (gr < stop) {
        if (cv < dvec) {
          val = *reinterpret_cast<const uint4*>(a.dy + gr * a.ldd + a.offd + cv * 8);
        } else {
          const long long b = gr / nvox;
          const long long vv = gr - b * nvox;
          const int x = (int)(vv % a.v.nx), y = (int)((vv / a.v.nx) % a.v.ny),
                    z = (int)(vv / ((long long)a.v.nx * a.v.ny));
          const long long nb = ((long long)wrap(z + dz, a.v.nz) * a.v.ny + wrap(y + dy, a.v.ny)) * a.v.nx +
                               wrap(x + dx, a.v.nx);
          val = *reinterpret_cast<const uint4*>(a.x + (b * nvox + nb) * a.ldx + a.offx + (cv - dvec) * 8);
        }
      }
      bf16* dst = cv < dvec ? sD + row * CP + cv * 8 : sX + row * XP + (cv - dvec) * 8;
      *reinterpret_cast<uint4*>(dst) = val;
    }
    __syncthreads();
    // the stage's 64 rows in accumulators of their own, added to the running sums with
    // rounding: the tensor core truncates each accumulation, and over the thousand
    // steps of a chunk that bias grows to 1e-5 of the sum
    float acc[4][4][4] = {};
#pragma unroll
    for (int ks = 0; ks < kWgRows; ks += 16) {
      const int mi = lane >> 3, rr = lane & 7;
      unsigned bq[2][4];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int n0 = (warp + 4 * p) * 16;
        if (n0 < a.cin) ldsm_x4_trans(bq[p], sXa + 2u * ((ks + (mi & 1) * 8 + rr) * XP + n0 + (mi >> 1) * 8));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i >= mt) continue;
        unsigned af[4];
        ldsm_x4_trans(af, sDa + 2u * ((ks + (mi >> 1) * 8 + rr) * CP + i * 16 + (mi & 1) * 8));
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const int n0 = (warp + 4 * p) * 16;
          if (n0 < a.cin) {
            mma16816(acc[i][2 * p], af, bq[p][0], bq[p][1]);
            mma16816(acc[i][2 * p + 1], af, bq[p][2], bq[p][3]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) sum[i][j][q] += acc[i][j][q];
  }
  const int g = lane >> 2, t = lane & 3;
  float* out = a.part + ((long long)blockIdx.x * 27 + tap) * a.cout_p * a.cin;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (i >= mt) continue;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int n0 = (warp + 4 * p) * 16 + h * 8;
        if (n0 >= a.cin) continue;
        const float* c = sum[i][2 * p + h];
        const int co = i * 16 + g, ci = n0 + 2 * t;
        out[(long long)co * a.cin + ci] = c[0];
        out[(long long)co * a.cin + ci + 1] = c[1];
        out[(long long)(co + 8) * a.cin + ci] = c[2];
        out[(long long)(co + 8) * a.cin + ci + 1] = c[3];
      }
    }
  }
}

// ------------------------------------------------------------------ elementwise
// network input (B, 4, N) FP32 -> channels-last BF16 [B][N][16] (channels 4..15 zero)
__global__ void k_features_in(const float* x, bf16* out, long long n, int batch) {
  chain_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n * batch;
       i += (long long)gridDim.x * blockDim.x) {
    const long long b = i / n, v = i - b * n;
    __align__(16) bf16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16(c < 4 ? x[(b * 4 + c) * n + v] : 0.f);
    reinterpret_cast<uint4*>(out + i * 16)[0] = reinterpret_cast<const uint4*>(o)[0];
    reinterpret_cast<uint4*>(out + i * 16)[1] = reinterpret_cast<const uint4*>(o)[1];
  }
}
// 2^3 average pooling, fine -> coarse (channels-last views), 8 channels (16 bytes) per thread
__global__ void k_pool(const bf16* in, int ldi, int offi, bf16* out, int ldo, int offo, int C, Vol coarse,
                       int batch) {
  chain_wait();
  const long long nc = (long long)coarse.nx * coarse.ny * coarse.nz;
  const int FX = 2 * coarse.nx, FY = 2 * coarse.ny, cv = C / 8;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nc * batch * cv;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / cv;
    const int c = (int)(i - r * cv) * 8;
    const unsigned rr = (unsigned)r, yz = rr / coarse.nx, x = rr - yz * coarse.nx;   // rows < 2^31 / 8
    const unsigned zb = yz / coarse.ny, y = yz - zb * coarse.ny;                      // zb = b nz + z
    const long long f0 = ((long long)(2 * zb) * FY + 2 * y) * FX + 2 * x;
    uint4 v[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) v[o] = *reinterpret_cast<const uint4*>(in + (f0 + sub_off(o, FX, FY)) * ldi + offi + c);
    __align__(16) bf16 s8[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float s = 0.f;
#pragma unroll
      for (int o = 0; o < 8; ++o) s += __bfloat162float(reinterpret_cast<const bf16*>(&v[o])[k]);
      s8[k] = __float2bfloat16(0.125f * s);
    }
    *reinterpret_cast<uint4*>(out + r * ldo + offo + c) = *reinterpret_cast<const uint4*>(s8);
  }
}
// pooling gradient added into the fine gradient, dfine[2u + o][c] += dcoarse[u][c] / 8,
// then the activation's derivative there from the sign of the saved output y (gate8);
// 8 channels (16 bytes) of one fine voxel per thread
__global__ void k_unpool_gate(const bf16* dco, int ldc, int offc, bf16* dfine, int ldf, int offf, const bf16* y,
                              int ldy, int offy, int C, Vol fine, int batch) {
  chain_wait();
  const long long nf = (long long)fine.nx * fine.ny * fine.nz;
  const int cv = C / 8;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nf * batch * cv;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / cv;
    const int c = (int)(i - r * cv) * 8;
    const unsigned rr = (unsigned)r, yz = rr / fine.nx, x = rr - yz * fine.nx;
    const unsigned zb = yz / fine.ny, yy = yz - zb * fine.ny;
    const long long u = ((long long)(zb / 2) * (fine.ny / 2) + yy / 2) * (fine.nx / 2) + x / 2;
    uint4* dp = reinterpret_cast<uint4*>(dfine + r * ldf + offf + c);
    const uint4 cg = *reinterpret_cast<const uint4*>(dco + u * ldc + offc + c);
    const uint4 yv = *reinterpret_cast<const uint4*>(y + r * ldy + offy + c);
    uint4 d = *dp;
    bf16* d8 = reinterpret_cast<bf16*>(&d);
    const bf16* c8 = reinterpret_cast<const bf16*>(&cg);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      d8[k] = __float2bfloat16(__bfloat162float(d8[k]) + 0.125f * __bfloat162float(c8[k]));
    gate8(reinterpret_cast<__nv_bfloat162*>(&d), yv);
    *dp = d;
  }
}
// bias gradient partials: part[block][c] = sum over this block's rows of dY[r][c];
// 8 channels (16 bytes) of a row per thread, thread sums added in thread order
constexpr int kBiasThreads = 256, kBiasBlocks = 304;
__global__ void __launch_bounds__(kBiasThreads) k_bias_grad(const bf16* dy, int ldd, int offd, int C, long long rows,
                                                            long long per, float* part) {
  chain_wait();
  __shared__ float red[kBiasThreads * 8];
  const int cv = C / 8, nr = kBiasThreads / cv;
  const int c = threadIdx.x % cv, j = threadIdx.x / cv;
  const long long r0 = blockIdx.x * per, r1 = min(rows, r0 + per);
  float s[8] = {};
  if (j < nr) {
#pragma unroll 4
    for (long long r = r0 + j; r < r1; r += nr) {
      const uint4 v = *reinterpret_cast<const uint4*>(dy + r * ldd + offd + c * 8);
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] += __bfloat162float(reinterpret_cast<const bf16*>(&v)[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) red[k * kBiasThreads + threadIdx.x] = s[k];
  __syncthreads();
  // 8 lanes per channel add the threads of its group in order, then one adds the lanes
  const int ch = threadIdx.x / 8, l = threadIdx.x % 8;
  for (int c0 = ch; c0 < C; c0 += kBiasThreads / 8) {
    const float* col = red + (c0 % 8) * kBiasThreads + c0 / 8;
    float t = 0.f;
    for (int q = l; q < nr; q += 8) t += col[q * cv];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o, 8);
    if (l == 0) part[(long long)blockIdx.x * C + c0] = t;
  }
}

// p - t of two floats without rounding (TwoSum): hi + lo
__device__ __forceinline__ ff exact_diff(float p, float t) {
  const float s = __fsub_rn(p, t), v = __fsub_rn(s, p);
  return ff_pair(s, __fsub_rn(__fsub_rn(p, __fsub_rn(s, v)), __fadd_rn(t, v)));
}
// the square of x and its rounding errors stay inside the FP32 range (x finite)
__device__ __forceinline__ bool ff_square_safe(float x) {
  const float m = fabsf(x);
  return (m > 1e-11f && m < 1e15f) || m == 0.f;
}
// The FP64 forms of the loss terms, out of line: inlined they are computed for every
// value and selected, and the FP64 pipe binds the pass again.
__device__ __noinline__ void loss_terms_f64(const float* p, const float* t, double& sn, double& sd) {
  for (int c = 0; c < 6; ++c) {
    const double x = t[c], d = (double)p[c] - x;
    sn += d * d;
    sd += x * x;
  }
}
__device__ __noinline__ float scaled_diff_f64(float p, float t, double f) { return (float)(((double)p - (double)t) * f); }
// Sum of squares as three floats, each at most an ulp of the one before it: TwoSum carries
// the rounding errors of the leading sum into the second and of that into the third, whose
// own rounding is 2^-24 of 2^-47 of the sum.  A voxel's squares (products without rounding
// from fused multiply-adds) come out to about 2^-68, so that their one rounding to FP64 is
// all that differs from an exact sum; 6 FP64 operations for 12 squares.
struct SqSum {
  float a = 0.f, b = 0.f, c = 0.f;
  static __device__ __forceinline__ float two_sum(float& s, float x) {
    const float t = __fadd_rn(s, x), v = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v));
    s = t;
    return e;
  }
  __device__ __forceinline__ void low(float x) { c = __fadd_rn(c, two_sum(b, x)); }
  __device__ __forceinline__ void add(float x) {                       // x^2
    const float q = __fmul_rn(x, x);
    low(two_sum(a, q));
    low(__fmaf_rn(x, x, -q));
  }
  __device__ __forceinline__ void add(ff x) {                          // (hi + lo)^2
    add(x.hi);
    const float h2 = __fadd_rn(x.hi, x.hi), q = __fmul_rn(h2, x.lo);
    low(q);
    c = __fadd_rn(c, __fmaf_rn(x.lo, x.lo, __fmaf_rn(h2, x.lo, -q)));
  }
  __device__ __forceinline__ double sum() const { return f2d_bits(a) + (f2d_bits(b) + f2d_bits(c)); }
};
// relative squared L2 loss: per (block, sample) sums of (p - t)^2 and t^2; one voxel
// per thread, planar fields (6 x n a sample).  The squares of a voxel are added in FP32
// pieces without loss (SqSum), voxels in FP64: with every term on the FP64 pipe the pass
// took 143 us for 8 samples of 64^3, now 63 us alone under the profiler; its 100 MB take
// 15.  Voxels with values outside the range of that form (tiny, huge, not finite) are
// formed in FP64.
constexpr int kLossBlocks = 64;
__global__ void k_loss(const float* pred, const float* target, long long n, double* num, double* den) {
  chain_wait();
  __shared__ double rn[32], rd[32];
  const int b = blockIdx.y;
  const float* pb = pred + (long long)b * 6 * n;
  const float* tb = target + (long long)b * 6 * n;
  double sn = 0.0, sd = 0.0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    SqSum vn, vd;
    float p6[6], t6[6];
    bool fast = true;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      p6[c] = pb[c * n + v];
      t6[c] = tb[c * n + v];
      const ff d = exact_diff(p6[c], t6[c]);
      vn.add(d);
      vd.add(t6[c]);
      fast = fast && ff_square_safe(d.hi) && ff_square_safe(t6[c]);
    }
    if (fast) {
      sn += vn.sum();
      sd += vd.sum();
    } else {
      double a0 = 0.0, a1 = 0.0;
      loss_terms_f64(p6, t6, a0, a1);
      sn += a0;
      sd += a1;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    sn += __shfl_down_sync(0xffffffffu, sn, off);
    sd += __shfl_down_sync(0xffffffffu, sd, off);
  }
  if ((threadIdx.x & 31) == 0) { rn[threadIdx.x >> 5] = sn; rd[threadIdx.x >> 5] = sd; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0, s1 = 0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) { s0 += rn[w]; s1 += rd[w]; }
    num[b * gridDim.x + blockIdx.x] = s0;
    den[b * gridDim.x + blockIdx.x] = s1;
  }
}
// The factor 2 / (den_b B) of the gradient, and loss = mean over b of num_b / den_b
// (written if loss != null): one warp per sample in turn, then thread 0 over the samples
__global__ void k_loss_final(const double* num, const double* den, int nblk, int batch, double* fac_b, double* rel_b,
                             double* loss) {
  chain_wait();
  const int lane = threadIdx.x & 31;
  for (int b = threadIdx.x >> 5; b < batch; b += blockDim.x >> 5) {
    double s0 = 0, s1 = 0;
    for (int k = lane; k < nblk; k += 32) { s0 += num[b * nblk + k]; s1 += den[b * nblk + k]; }
    for (int off = 16; off > 0; off >>= 1) {
      s0 += __shfl_down_sync(0xffffffffu, s0, off);
      s1 += __shfl_down_sync(0xffffffffu, s1, off);
    }
    if (lane == 0) { fac_b[b] = 2.0 / (s1 * batch); rel_b[b] = s0 / s1; }
  }
  __syncthreads();
  if (threadIdx.x == 0 && loss != nullptr) {
    double l = 0.0;
    for (int b = 0; b < batch; ++b) l += rel_b[b];
    *loss = l / batch;
  }
}
// dL/dpred = 2 (p - t) / (den_b B), written as the head's output gradient
// [B][N][16] BF16 (channels 6..15 zero); one voxel per thread.  The product is rounded to
// FP32 once; it comes from float-float arithmetic where that rounds as FP64 does (155 us of
// FP64 pipe for 8 samples of 64^3 otherwise) and from FP64 where not, or outside its range
__global__ void k_loss_grad(const float* pred, const float* target, const double* fac_b, long long n, bf16* dy) {
  chain_wait();
  const int b = blockIdx.y;
  const double fd = fac_b[b];
  const ff f = d2ff_bits(fd);       // (FP64 divisions and conversions by every thread took 65 us)
  const bool fast = f.hi > 1e-18f && f.hi < 1e18f;
  const float* pb = pred + (long long)b * 6 * n;
  const float* tb = target + (long long)b * 6 * n;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    __align__(16) bf16 o[16];
#pragma unroll
    for (int c = 6; c < 16; ++c) o[c] = __float2bfloat16(0.f);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const float p = pb[c * n + v], t = tb[c * n + v];
      const ff d = exact_diff(p, t), r = d * f;
      o[c] = __float2bfloat16(fast && ff_square_safe(d.hi) && ff_rounds_as_fp64(r) ? r.hi : scaled_diff_f64(p, t, fd));
    }
    uint4* d = reinterpret_cast<uint4*>(dy + ((long long)b * n + v) * 16);
    d[0] = reinterpret_cast<const uint4*>(o)[0];
    d[1] = reinterpret_cast<const uint4*>(o)[1];
  }
}
// Adam (Kingma and Ba 2014), bias-corrected, FP32 state
__global__ void k_adam(float* w, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  chain_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ------------------------------------------------------------------ weight layouts
// kind 0 conv3, 1 conv1, 2 up.  Forward layout [tap][cols][cin_p] with
// cols = cout_p (conv) or 8 cout (up, column o cout + co); data-gradient
// layout: conv [26 - tap][cin_p][cout_p] (flipped taps, transposed), up
// [cin_p][8 cout].  The flat vector holds PyTorch's shapes: conv
// W[co][ci][kz][ky][kx] (tap = 9 kz + 3 ky + kx), up W[ci][co][oz][oy][ox].
struct LayerDef { int kind, cin, cout, cin_p, cout_p; long long woff, boff; };
constexpr int kNumLayers = 18;
struct PackArgs {
  LayerDef def[kNumLayers];
  bf16 *fw[kNumLayers], *bw[kNumLayers];
};

// every layer in one launch (blockIdx.y = layer)
__global__ void k_pack(const float* flat, const __grid_constant__ PackArgs pa) {
  chain_wait();
  const LayerDef& L = pa.def[blockIdx.y];
  bf16* const fw = pa.fw[blockIdx.y];
  bf16* const bw = pa.bw[blockIdx.y];
  const int taps = L.kind == 0 ? 27 : 1;
  const int ocols = L.kind == 2 ? 8 * L.cout : L.cout_p;
  const int nf = taps * ocols * L.cin_p;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nf; i += gridDim.x * blockDim.x) {
    const int ci = i % L.cin_p;
    const int r = i / L.cin_p;
    const int col = r % ocols, tap = r / ocols;
    float w = 0.f;
    if (ci < L.cin) {
      if (L.kind == 2) {
        const int o = col / L.cout, co = col - o * L.cout;
        w = flat[L.woff + ((long long)ci * L.cout + co) * 8 + o];
      } else if (col < L.cout) {
        w = flat[L.woff + ((long long)col * L.cin + ci) * taps + tap];
      }
    }
    const bf16 wb = __float2bfloat16(w);
    fw[i] = wb;
    if (L.kind == 2) bw[(long long)ci * ocols + col] = wb;
    else bw[((long long)(taps == 27 ? 26 - tap : 0) * L.cin_p + ci) * L.cout_p + col] = wb;
  }
}

// A layer's gradients from their partials into the flat vector: weights [chunk][tap]
// [cols][cin_p] (layout of the forward weights), biases [block][bcols].  Blocks of 32
// outputs x 8 lanes: lane j adds partials j, j + 8, ... in order, the lanes are added
// pairwise (a fixed order).  One thread per output over all partials left the pass to
// the latency of up to 1024 dependent loads (18-120 us a layer).
constexpr int kRedOut = 32, kRedLanes = 8;
__global__ void __launch_bounds__(kRedOut * kRedLanes) k_reduce_grad(const float* wpart, int nchunks, const float* bpart,
                                                                    int nblk, int bcols, LayerDef L, float* gflat) {
  chain_wait();
  __shared__ float red[kRedLanes][kRedOut];
  const int o = threadIdx.x % kRedOut, j = threadIdx.x / kRedOut;
  const int taps = L.kind == 0 ? 27 : 1;
  const int ocols = L.kind == 2 ? 8 * L.cout : L.cout_p;
  const int per = taps * ocols * L.cin_p;
  const int wblocks = (per + kRedOut - 1) / kRedOut;
  const bool bias = (int)blockIdx.x >= wblocks;
  const int i = (bias ? (int)blockIdx.x - wblocks : (int)blockIdx.x) * kRedOut + o;
  const int count = bias ? bcols : per, parts = bias ? nblk : nchunks;
  const float* p = bias ? bpart : wpart;
  float s = 0.f;
  if (i < count) {
#pragma unroll 8
    for (int c = j; c < parts; c += kRedLanes) s += p[(long long)c * count + i];
  }
  red[j][o] = s;
  __syncthreads();
  if (j != 0 || i >= count) return;
#pragma unroll
  for (int h = 0; h < kRedLanes; h += 2) red[h][o] += red[h + 1][o];
  const float t = (red[0][o] + red[2][o]) + (red[4][o] + red[6][o]);
  if (bias) {
    if (i < L.cout) gflat[L.boff + i] = t;
    return;
  }
  const int ci = i % L.cin_p, r = i / L.cin_p, col = r % ocols, tap = r / ocols;
  if (ci >= L.cin) return;
  if (L.kind == 2) gflat[L.woff + ((long long)ci * L.cout + col % L.cout) * 8 + col / L.cout] = t;
  else if (col < L.cout) gflat[L.woff + ((long long)col * L.cin + ci) * taps + tap] = t;
}

// ------------------------------------------------------------------ features / outputs
// per sample: max |b| over 3 N values as the bits of a non-negative float
// (order-independent); sample = blockIdx.y, one atomic per block
template <typename R> struct SampleArgs {
  const R* b[kSampleArgs];
  const int8_t* phase[kSampleArgs];
};
template <typename R>
__global__ void k_absmax(const __grid_constant__ SampleArgs<R> sa, long long n3, unsigned* out) {
  chain_wait();
  __shared__ float red[32];
  const R* b = sa.b[blockIdx.y];
  float m = 0.f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf((float)b[i]));
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)blockDim.x / 32; ++w) m = fmaxf(m, red[w]);
    atomicMax(out + blockIdx.y, __float_as_uint(m));
  }
}
struct MuTab { float mu[BFCS_MAX_PHASES]; float mu_max; };
// x (4, N): b / s and mu / mu_max - 1/2; target (6, N) = eps mu_max / s (if eps)
template <typename R>
__global__ void k_prepare(const R* b, const int8_t* phase, MuTab mt, const unsigned* sbits, const R* eps, float* x,
                          float* target, long long n) {
  chain_wait();
  const float s = __uint_as_float(*sbits);
  const float inv = s > 0.f ? 1.f / s : 0.f;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < 3; ++c) x[c * n + v] = (float)b[c * n + v] * inv;
    x[3 * n + v] = mt.mu[phase[v]] / mt.mu_max - 0.5f;
    if (eps != nullptr) {
#pragma unroll
      for (int c = 0; c < 6; ++c) target[c * n + v] = (float)((double)eps[c * n + v] * mt.mu_max * inv);
    }
  }
}
// channels-last BF16 network inputs straight from b and phase (sample = blockIdx.y)
template <typename R>
__global__ void k_prepare_x0(const __grid_constant__ SampleArgs<R> sa, MuTab mt, const unsigned* sbits, bf16* x0,
                             long long n) {
  chain_wait();
  const R* b = sa.b[blockIdx.y];
  const int8_t* phase = sa.phase[blockIdx.y];
  x0 += (long long)blockIdx.y * n * 16;
  const float s = __uint_as_float(sbits[blockIdx.y]);
  const float inv = s > 0.f ? 1.f / s : 0.f;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    __align__(16) bf16 o[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) o[c] = __float2bfloat16(0.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c] = __float2bfloat16((float)b[c * n + v] * inv);
    o[3] = __float2bfloat16(mt.mu[phase[v]] / mt.mu_max - 0.5f);
    reinterpret_cast<uint4*>(x0 + v * 16)[0] = reinterpret_cast<const uint4*>(o)[0];
    reinterpret_cast<uint4*>(x0 + v * 16)[1] = reinterpret_cast<const uint4*>(o)[1];
  }
}

}  // namespace net
}  // namespace bfcs

// ====================================================================== host side
using bfcs::launch_chain;
using namespace bfcs::net;
using bfcs::count_launches;

namespace {

// (kind, cin, cout) in the order of the flat parameter vector
struct LayerSpec { int kind, cin, cout; };
constexpr LayerSpec kSpec[kNumLayers] = {
    {0, 4, 32},  {0, 32, 32},                 // e0a e0b
    {0, 32, 32}, {0, 32, 32},                 // e1a e1b
    {0, 32, 32}, {0, 32, 32},                 // e2a e2b
    {0, 32, 48}, {0, 48, 48},                 // e3a e3b
    {2, 48, 32}, {0, 64, 32}, {0, 32, 32},    // u2 d2a d2b
    {2, 32, 32}, {0, 64, 32}, {0, 32, 32},    // u1 d1a d1b
    {2, 32, 32}, {0, 64, 32}, {0, 32, 32},    // u0 d0a d0b
    {1, 32, 6},                               // head
};
enum { E0A, E0B, E1A, E1B, E2A, E2B, E3A, E3B, U2, D2A, D2B, U1, D1A, D1B, U0, D0A, D0B, HEAD };

long long param_count() {
  long long n = 0;
  for (const LayerSpec& s : kSpec) {
    const long long k = s.kind == 0 ? 27 : s.kind == 1 ? 1 : 8;
    n += k * s.cin * s.cout + s.cout;
  }
  return n;
}

int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }
int grid_for(long long n, int threads = 256) { return std::max(1, std::min(ceil_div(n, threads), 152 * 16)); }

struct View { bf16* p; int ld, off; };

}  // namespace

struct bfcs_net_s {
  int nx, ny, nz, maxb, flags;
  cudaStream_t st;
  Vol vol[4];
  long long n[4];
  LayerDef def[kNumLayers];
  bf16* fw[kNumLayers];
  bf16* bw[kNumLayers];
  char* base = nullptr;
  // activations
  bf16 *X0, *A0, *C0, *D0a, *D0b, *P0, *A1, *C1, *D1a, *D1b, *P1, *A2, *C2, *D2a, *D2b, *P2, *A3, *H3;
  float* OUT;                // head output (B, 6, n), training
  // gradients (training only)
  bf16 *dOUT = nullptr, *dA0, *dC0, *dD0a, *dD0b, *dP0, *dA1, *dC1, *dD1a, *dD1b, *dP1, *dA2, *dC2, *dD2a, *dD2b,
       *dP2, *dA3, *dH3;
  float* part = nullptr;     // weight / bias gradient partials
  long long part_cap = 0;
  double* lnum;              // loss partials
  double* lden;
  double* fac_b;
  double* rel_b;
  unsigned* sbits;           // per-sample max |b|
  int* err;                  // set by a kernel whose bounded wait expired
};

namespace {

cudaError_t pack_all(bfcs_net_s* N, const float* params) {
  PackArgs pa;
  for (int l = 0; l < kNumLayers; ++l) { pa.def[l] = N->def[l]; pa.fw[l] = N->fw[l]; pa.bw[l] = N->bw[l]; }
  launch_chain(true, k_pack, dim3(108, kNumLayers), 256, 0, N->st, params, pa);
  count_launches(1);
  return cudaGetLastError();
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess || n < 1)
      n = 1;
  }
  return n;
}

// BFCS_NET_TCGEN05=0 keeps the convolutions on the mma.sync kernels
bool tcgen05_enabled() {
  const char* e = std::getenv("BFCS_NET_TCGEN05");
  return !(e != nullptr && std::atoi(e) == 0);
}

cudaError_t launch_conv(const ConvArgs& a, long long nvox, int* err, cudaStream_t st) {
  if (rows_ok(a)) return launch_rows(a, sm_count(), st);
  if (!conv3_ok(a)) return cudaErrorInvalidValue;
  if (tcgen05_enabled()) return launch_conv3(a, sm_count(), err, st);
  launch_chain(true, k_conv, dim3(ceil_div(nvox, kConvWarps * 32), ceil_div(a.cout_p, kConvNT * 8), a.batch),
               kConvWarps * 32, 0, st, a);
  count_launches(1);
  return cudaGetLastError();
}

// forward GEMM of layer l: in -> out on the grid of level lv (coarse level for an up layer)
cudaError_t conv_fwd(bfcs_net_s* N, int l, const float* params, int B, View in, int lv, int out_mode, void* out,
                     int ldo, int offo) {
  const LayerDef& L = N->def[l];
  ConvArgs a{};
  a.in = in.p; a.ldi = in.ld; a.offi = in.off;
  a.cin = L.cin_p;
  a.w = N->fw[l];
  a.bias = params + L.boff;
  a.bias_mod = L.cout;
  a.cout_p = L.kind == 2 ? 8 * L.cout : L.cout_p;
  a.ksize = L.kind == 0 ? 3 : 1;
  a.v = N->vol[lv];
  a.batch = B;
  a.act = L.kind == 0 ? 1 : 0;
  a.in_mode = IN_CONV;
  a.out_mode = out_mode;
  a.out = out; a.ldo = ldo; a.offo = offo;
  a.up_c = L.cout;
  return launch_conv(a, N->n[lv], N->err, N->st);
}

cudaError_t pool(bfcs_net_s* N, View in, View out, int C, int coarse_lv, int B) {
  const long long tot = N->n[coarse_lv] * B * C / 8;
  launch_chain(true, k_pool, grid_for(tot), 256, 0, N->st, in.p, in.ld, in.off, out.p, out.ld, out.off, C,
               N->vol[coarse_lv], B);
  count_launches(1);
  return cudaGetLastError();
}

#define NET_TRY(x) \
  if ((e = (x)) != cudaSuccess) return e

cudaError_t forward(bfcs_net_s* N, const float* params, int B) {
  cudaError_t e;
  const int F = OUT_BF16;
  NET_TRY(conv_fwd(N, E0A, params, B, {N->X0, 16, 0}, 0, F, N->A0, 32, 0));
  NET_TRY(conv_fwd(N, E0B, params, B, {N->A0, 32, 0}, 0, F, N->C0, 64, 32));
  NET_TRY(pool(N, {N->C0, 64, 32}, {N->P0, 32, 0}, 32, 1, B));
  NET_TRY(conv_fwd(N, E1A, params, B, {N->P0, 32, 0}, 1, F, N->A1, 32, 0));
  NET_TRY(conv_fwd(N, E1B, params, B, {N->A1, 32, 0}, 1, F, N->C1, 64, 32));
  NET_TRY(pool(N, {N->C1, 64, 32}, {N->P1, 32, 0}, 32, 2, B));
  NET_TRY(conv_fwd(N, E2A, params, B, {N->P1, 32, 0}, 2, F, N->A2, 32, 0));
  NET_TRY(conv_fwd(N, E2B, params, B, {N->A2, 32, 0}, 2, F, N->C2, 64, 32));
  NET_TRY(pool(N, {N->C2, 64, 32}, {N->P2, 32, 0}, 32, 3, B));
  NET_TRY(conv_fwd(N, E3A, params, B, {N->P2, 32, 0}, 3, F, N->A3, 48, 0));
  NET_TRY(conv_fwd(N, E3B, params, B, {N->A3, 48, 0}, 3, F, N->H3, 48, 0));
  NET_TRY(conv_fwd(N, U2, params, B, {N->H3, 48, 0}, 3, OUT_SHUFFLE_UP, N->C2, 64, 0));
  NET_TRY(conv_fwd(N, D2A, params, B, {N->C2, 64, 0}, 2, F, N->D2a, 32, 0));
  NET_TRY(conv_fwd(N, D2B, params, B, {N->D2a, 32, 0}, 2, F, N->D2b, 32, 0));
  NET_TRY(conv_fwd(N, U1, params, B, {N->D2b, 32, 0}, 2, OUT_SHUFFLE_UP, N->C1, 64, 0));
  NET_TRY(conv_fwd(N, D1A, params, B, {N->C1, 64, 0}, 1, F, N->D1a, 32, 0));
  NET_TRY(conv_fwd(N, D1B, params, B, {N->D1a, 32, 0}, 1, F, N->D1b, 32, 0));
  NET_TRY(conv_fwd(N, U0, params, B, {N->D1b, 32, 0}, 1, OUT_SHUFFLE_UP, N->C0, 64, 0));
  NET_TRY(conv_fwd(N, D0A, params, B, {N->C0, 64, 0}, 0, F, N->D0a, 32, 0));
  NET_TRY(conv_fwd(N, D0B, params, B, {N->D0a, 32, 0}, 0, F, N->D0b, 32, 0));
  return cudaSuccess;
}

// the head over samples 0..B-1 of D0b: sample i to out[i] (6 x n), as the network's
// output or (predict) as the strain prediction
template <typename R>
cudaError_t head(bfcs_net_s* N, const float* params, int B, R* const* out, bool predict, float mu_max) {
  for (int i0 = 0; i0 < B; i0 += kSampleArgs) {
    const int k = std::min(kSampleArgs, B - i0);
    HeadArgs<R> a{};
    a.in = N->D0b + (long long)i0 * N->n[0] * 32;
    a.w = N->fw[HEAD];
    a.bias = params + N->def[HEAD].boff;
    a.n = N->n[0];
    a.sbits = N->sbits + i0;
    a.mu_max = mu_max;
    for (int i = 0; i < k; ++i) a.out[i] = out[i0 + i];
    const cudaError_t e = launch_head<R>(a, k, predict, sm_count(), N->st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t head_planar(bfcs_net_s* N, const float* params, int B, float* y) {
  std::vector<float*> out(B);
  for (int i = 0; i < B; ++i) out[i] = y + (long long)i * 6 * N->n[0];
  return head<float>(N, params, B, out.data(), false, 1.f);
}

// Backward of layer l.  dout: gradient w.r.t. the layer's pre-activation (gated where
// it was written); in: saved input; din: where the input gradient goes (p == null: not
// needed); gate: the saved output whose activation's derivative din takes (p == null:
// none: an up-convolution's or pooling's output, or a gradient still to be added to).
// lv: level of the GEMM rows (coarse level for an up layer).  Gradients go to grad.
cudaError_t layer_bwd(bfcs_net_s* N, float* grad, int l, int B, View dout, View in, View din, View gate, int lv) {
  const LayerDef& L = N->def[l];
  const bool up = L.kind == 2;
  const int taps = L.kind == 0 ? 27 : 1;
  const long long rows = N->n[lv] * B;                  // GEMM K rows of the weight gradient
  // weight gradient
  WgArgs w{};
  w.dy = dout.p; w.ldd = dout.ld; w.offd = dout.off;
  w.x = in.p; w.ldx = in.ld; w.offx = in.off;
  w.cin = L.cin_p;
  w.cout_p = up ? 8 * L.cout : L.cout_p;
  w.ksize = L.kind == 0 ? 3 : 1;
  w.v = N->vol[lv];
  w.batch = B;
  w.up_c = up ? L.cout : 0;
  const long long per = (long long)taps * w.cout_p * w.cin;
  const int bc = up ? L.cout : L.cout_p;                // channels of the output gradient view
  const bool tc = wgrad3_ok(w) && tcgen05_enabled(), pw = wgrad1_ok(w);
  int nchunks, nblk;                                    // partials of the weights and of the bias
  if (tc) {
    nblk = nchunks = wgrad3_chunks(w, sm_count());
  } else if (pw) {
    nchunks = wgrad1_chunks(w, sm_count());
    nblk = up ? nchunks / 2 : nchunks;
  } else {
    if (w.ksize != 3 || w.cout_p > 64) return cudaErrorInvalidValue;
    nchunks = std::min(ceil_div(152 * 8, taps), ceil_div(rows, kWgRows));
    w.chunk = (long long)ceil_div(ceil_div(rows, nchunks), kWgRows) * kWgRows;
    nchunks = ceil_div(rows, w.chunk);
    nblk = std::min(kBiasBlocks, ceil_div(rows, 64));
  }
  if ((long long)nchunks * per + (long long)nblk * bc > N->part_cap) return cudaErrorInvalidValue;
  w.part = N->part;
  w.bpart = N->part + (long long)nchunks * per;
  if (tc || pw) {   // with the bias gradient
    const cudaError_t e = tc ? launch_wgrad3(w, nchunks, N->err, N->st) : launch_wgrad1(w, sm_count(), N->st);
    if (e != cudaSuccess) return e;
  } else {
    const size_t smem = (size_t)kWgRows * (w.cout_p + 8 + w.cin + 8) * sizeof(bf16);
    launch_chain(true, k_wgrad, dim3(nchunks, taps), 128, smem, N->st, w);
    launch_chain(true, k_bias_grad, nblk, kBiasThreads, 0, N->st, dout.p, dout.ld, dout.off, bc, rows,
                 (rows + nblk - 1) / nblk, w.bpart);
    count_launches(2);
  }
  launch_chain(true, k_reduce_grad, ceil_div(per, kRedOut) + ceil_div(bc, kRedOut), kRedOut * kRedLanes, 0, N->st,
               N->part, nchunks, w.bpart, nblk, bc, L, grad);
  count_launches(1);
  // input gradient: a convolution with the data-gradient weights
  if (din.p != nullptr) {
    ConvArgs a{};
    a.in = dout.p; a.ldi = dout.ld; a.offi = dout.off;
    a.cin = up ? 8 * L.cout : L.cout_p;
    a.w = N->bw[l];
    a.bias = nullptr; a.bias_mod = 1;
    a.cout_p = L.cin_p;
    a.ksize = L.kind == 0 ? 3 : 1;
    a.v = N->vol[lv];
    a.batch = B;
    a.act = 0;
    a.in_mode = up ? IN_GATHER_UP : IN_CONV;
    a.out_mode = OUT_BF16;
    a.out = din.p; a.ldo = din.ld; a.offo = din.off;
    a.up_c = L.cout;
    a.gate = gate.p; a.ldg = gate.ld; a.offg = gate.off;
    const cudaError_t e = launch_conv(a, N->n[lv], N->err, N->st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

// pooling gradient into the skip half of a concatenation's gradient, and its gate
cudaError_t unpool_gate(bfcs_net_s* N, View dco, View dfine, View y, int C, int fine_lv, int B) {
  const long long tot = N->n[fine_lv] * B * C / 8;
  launch_chain(true, k_unpool_gate, grid_for(tot), 256, 0, N->st, dco.p, dco.ld, dco.off, dfine.p, dfine.ld,
               dfine.off, y.p, y.ld, y.off, C, N->vol[fine_lv], B);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t backward(bfcs_net_s* N, float* g, int B) {
  cudaError_t e;
  const View none{nullptr, 0, 0};
  NET_TRY(layer_bwd(N, g, HEAD, B, {N->dOUT, 16, 0}, {N->D0b, 32, 0}, {N->dD0b, 32, 0}, {N->D0b, 32, 0}, 0));
  NET_TRY(layer_bwd(N, g, D0B, B, {N->dD0b, 32, 0}, {N->D0a, 32, 0}, {N->dD0a, 32, 0}, {N->D0a, 32, 0}, 0));
  NET_TRY(layer_bwd(N, g, D0A, B, {N->dD0a, 32, 0}, {N->C0, 64, 0}, {N->dC0, 64, 0}, none, 0));
  NET_TRY(layer_bwd(N, g, U0, B, {N->dC0, 64, 0}, {N->D1b, 32, 0}, {N->dD1b, 32, 0}, {N->D1b, 32, 0}, 1));
  NET_TRY(layer_bwd(N, g, D1B, B, {N->dD1b, 32, 0}, {N->D1a, 32, 0}, {N->dD1a, 32, 0}, {N->D1a, 32, 0}, 1));
  NET_TRY(layer_bwd(N, g, D1A, B, {N->dD1a, 32, 0}, {N->C1, 64, 0}, {N->dC1, 64, 0}, none, 1));
  NET_TRY(layer_bwd(N, g, U1, B, {N->dC1, 64, 0}, {N->D2b, 32, 0}, {N->dD2b, 32, 0}, {N->D2b, 32, 0}, 2));
  NET_TRY(layer_bwd(N, g, D2B, B, {N->dD2b, 32, 0}, {N->D2a, 32, 0}, {N->dD2a, 32, 0}, {N->D2a, 32, 0}, 2));
  NET_TRY(layer_bwd(N, g, D2A, B, {N->dD2a, 32, 0}, {N->C2, 64, 0}, {N->dC2, 64, 0}, none, 2));
  NET_TRY(layer_bwd(N, g, U2, B, {N->dC2, 64, 0}, {N->H3, 48, 0}, {N->dH3, 48, 0}, {N->H3, 48, 0}, 3));
  NET_TRY(layer_bwd(N, g, E3B, B, {N->dH3, 48, 0}, {N->A3, 48, 0}, {N->dA3, 48, 0}, {N->A3, 48, 0}, 3));
  NET_TRY(layer_bwd(N, g, E3A, B, {N->dA3, 48, 0}, {N->P2, 32, 0}, {N->dP2, 32, 0}, none, 3));
  NET_TRY(unpool_gate(N, {N->dP2, 32, 0}, {N->dC2, 64, 32}, {N->C2, 64, 32}, 32, 2, B));
  NET_TRY(layer_bwd(N, g, E2B, B, {N->dC2, 64, 32}, {N->A2, 32, 0}, {N->dA2, 32, 0}, {N->A2, 32, 0}, 2));
  NET_TRY(layer_bwd(N, g, E2A, B, {N->dA2, 32, 0}, {N->P1, 32, 0}, {N->dP1, 32, 0}, none, 2));
  NET_TRY(unpool_gate(N, {N->dP1, 32, 0}, {N->dC1, 64, 32}, {N->C1, 64, 32}, 32, 1, B));
  NET_TRY(layer_bwd(N, g, E1B, B, {N->dC1, 64, 32}, {N->A1, 32, 0}, {N->dA1, 32, 0}, {N->A1, 32, 0}, 1));
  NET_TRY(layer_bwd(N, g, E1A, B, {N->dA1, 32, 0}, {N->P0, 32, 0}, {N->dP0, 32, 0}, none, 1));
  NET_TRY(unpool_gate(N, {N->dP0, 32, 0}, {N->dC0, 64, 32}, {N->C0, 64, 32}, 32, 0, B));
  NET_TRY(layer_bwd(N, g, E0B, B, {N->dC0, 64, 32}, {N->A0, 32, 0}, {N->dA0, 32, 0}, {N->A0, 32, 0}, 0));
  NET_TRY(layer_bwd(N, g, E0A, B, {N->dA0, 32, 0}, {N->X0, 16, 0}, none, none, 0));
  return cudaSuccess;
}

cudaError_t loss_and_grad(bfcs_net_s* N, int B, const float* target, double* loss_dev) {
  launch_chain(true, k_loss, dim3(kLossBlocks, B), 256, 0, N->st, N->OUT, target, N->n[0], N->lnum, N->lden);
  launch_chain(true, k_loss_final, 1, 256, 0, N->st, N->lnum, N->lden, kLossBlocks, B, N->fac_b, N->rel_b, loss_dev);
  const int bx = std::max(1, std::min(ceil_div(N->n[0], 256), ceil_div(152 * 16, B)));
  launch_chain(true, k_loss_grad, dim3(bx, B), 256, 0, N->st, N->OUT, target, N->fac_b, N->n[0], N->dOUT);
  count_launches(3);
  return cudaGetLastError();
}

int status_of(cudaError_t e) { return e == cudaSuccess ? BFCS_OK : BFCS_ERR_CUDA; }

void free_net(bfcs_net_s* N) {
  if (N->base) cudaFree(N->base);
  delete N;
}

float mu_table(int nphases, const bfcs_lame* phases, MuTab* mt) {
  float mx = 0.f;
  for (int p = 0; p < BFCS_MAX_PHASES; ++p) mt->mu[p] = 0.f;
  for (int p = 0; p < nphases; ++p) {
    mt->mu[p] = (float)phases[p].mu;
    mx = std::max(mx, mt->mu[p]);
  }
  mt->mu_max = mx;
  return mx;
}

bool valid_phases(int nphases, const bfcs_lame* phases) {
  if (nphases < 1 || nphases > BFCS_MAX_PHASES || phases == nullptr) return false;
  for (int p = 0; p < nphases; ++p)
    if (!(phases[p].mu > 0.0) || !std::isfinite(phases[p].mu)) return false;
  return true;
}

// strain predictions of `batch` samples, maxb at a time
template <typename R>
int predict(bfcs_net_s* N, const float* params, int batch, const R* const* b, const int8_t* const* phase, int nphases,
            const bfcs_lame* phases, R* const* eps_out) {
  MuTab mt;
  const float mu_max = mu_table(nphases, phases, &mt);
  const long long n = N->n[0];
  cudaError_t e = pack_all(N, params);
  for (int i0 = 0; i0 < batch && e == cudaSuccess; i0 += N->maxb) {
    const int B = std::min(N->maxb, batch - i0);
    cudaMemsetAsync(N->sbits, 0, B * sizeof(unsigned), N->st);
    for (int j0 = 0; j0 < B; j0 += kSampleArgs) {
      const int k = std::min(kSampleArgs, B - j0);
      SampleArgs<R> sa{};
      for (int j = 0; j < k; ++j) { sa.b[j] = b[i0 + j0 + j]; sa.phase[j] = phase[i0 + j0 + j]; }
      const int bx = std::max(1, std::min(ceil_div(n, 256), ceil_div(152 * 8, k)));
      launch_chain(true, k_absmax<R>, dim3(bx, k), 256, 0, N->st, sa, 3 * n, N->sbits + j0);
      launch_chain(true, k_prepare_x0<R>, dim3(bx, k), 256, 0, N->st, sa, mt, N->sbits + j0,
                   N->X0 + (long long)j0 * n * 16, n);
      count_launches(2);
    }
    e = forward(N, params, B);
    if (e == cudaSuccess) e = head<R>(N, params, B, eps_out + i0, true, mu_max);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  return status_of(e);
}

}  // namespace

extern "C" {

long long bfcs_net_param_count(void) { return param_count(); }

int bfcs_net_create(bfcs_net* out, int nx, int ny, int nz, int max_batch, int flags, void* stream) {
  if (out == nullptr) return BFCS_ERR_INVALID_ARG;
  *out = nullptr;
  if (nx < 8 || ny < 8 || nz < 8 || nx % 8 || ny % 8 || nz % 8 || max_batch < 1 || max_batch > 1024 ||
      (flags & ~BFCS_NET_TRAIN) != 0)
    return BFCS_ERR_INVALID_ARG;
  if ((long long)nx * ny * nz * max_batch > (1LL << 31)) return BFCS_ERR_INVALID_ARG;
  bfcs_net_s* N = new (std::nothrow) bfcs_net_s();
  if (N == nullptr) return BFCS_ERR_OOM;
  N->nx = nx; N->ny = ny; N->nz = nz; N->maxb = max_batch; N->flags = flags;
  N->st = (cudaStream_t)stream;
  for (int l = 0; l < 4; ++l) {
    N->vol[l] = {nx >> l, ny >> l, nz >> l};
    N->n[l] = (long long)(nx >> l) * (ny >> l) * (nz >> l);
  }
  long long off = 0;
  for (int l = 0; l < kNumLayers; ++l) {
    const LayerSpec& s = kSpec[l];
    LayerDef& L = N->def[l];
    L.kind = s.kind; L.cin = s.cin; L.cout = s.cout;
    L.cin_p = (s.cin + 15) / 16 * 16;
    L.cout_p = s.kind == 1 ? (s.cout + 15) / 16 * 16 : s.cout;
    L.woff = off;
    off += (long long)(s.kind == 0 ? 27 : s.kind == 1 ? 1 : 8) * s.cin * s.cout;
    L.boff = off;
    off += s.cout;
  }
  // one allocation, carved in 256-byte aligned pieces
  const long long B = max_batch;
  const bool train = (flags & BFCS_NET_TRAIN) != 0;
  std::vector<std::pair<void**, size_t>> req;
  auto add = [&](void* p, size_t bytes) { req.push_back({(void**)p, bytes}); };
  const long long* n = N->n;
  auto act = [&](bf16** p, int lv, int C) { add(p, (size_t)(B * n[lv] * C) * sizeof(bf16)); };
  act(&N->X0, 0, 16); act(&N->A0, 0, 32); act(&N->C0, 0, 64); act(&N->D0a, 0, 32); act(&N->D0b, 0, 32);
  act(&N->P0, 1, 32); act(&N->A1, 1, 32); act(&N->C1, 1, 64); act(&N->D1a, 1, 32); act(&N->D1b, 1, 32);
  act(&N->P1, 2, 32); act(&N->A2, 2, 32); act(&N->C2, 2, 64); act(&N->D2a, 2, 32); act(&N->D2b, 2, 32);
  act(&N->P2, 3, 32); act(&N->A3, 3, 48); act(&N->H3, 3, 48);
  if (train) add(&N->OUT, (size_t)(B * n[0] * 6) * sizeof(float));
  for (int l = 0; l < kNumLayers; ++l) {
    const LayerDef& L = N->def[l];
    const size_t nw = (size_t)(L.kind == 0 ? 27 : 1) * (L.kind == 2 ? 8 * L.cout : L.cout_p) * L.cin_p;
    add(&N->fw[l], nw * sizeof(bf16));
    add(&N->bw[l], nw * sizeof(bf16));
  }
  add(&N->lnum, (size_t)kLossBlocks * B * sizeof(double));
  add(&N->lden, (size_t)kLossBlocks * B * sizeof(double));
  add(&N->fac_b, (size_t)B * sizeof(double));
  add(&N->rel_b, (size_t)B * sizeof(double));
  add(&N->sbits, (size_t)B * sizeof(unsigned));
  add(&N->err, sizeof(int));
  if (train) {
    act(&N->dOUT, 0, 16); act(&N->dA0, 0, 32); act(&N->dC0, 0, 64); act(&N->dD0a, 0, 32); act(&N->dD0b, 0, 32);
    act(&N->dP0, 1, 32); act(&N->dA1, 1, 32); act(&N->dC1, 1, 64); act(&N->dD1a, 1, 32); act(&N->dD1b, 1, 32);
    act(&N->dP1, 2, 32); act(&N->dA2, 2, 32); act(&N->dC2, 2, 64); act(&N->dD2a, 2, 32); act(&N->dD2b, 2, 32);
    act(&N->dP2, 3, 32); act(&N->dA3, 3, 48); act(&N->dH3, 3, 48);
    // weight-gradient partials: at most 152*8 blocks' worth of one layer's weights, plus bias partials
    N->part_cap = 0;
    for (int l = 0; l < kNumLayers; ++l) {
      const LayerDef& L = N->def[l];
      const long long taps = L.kind == 0 ? 27 : 1;
      const long long per = taps * (L.kind == 2 ? 8 * L.cout : L.cout_p) * L.cin_p;
      const long long mch = L.kind == 2 ? 8 * L.cout / 64 : 1;
      const long long nch = std::max<long long>(1, ceil_div(152 * 8, taps * mch));
      N->part_cap = std::max(N->part_cap, std::max(nch, 152LL) * per + 1024LL * 64);
    }
    add(&N->part, (size_t)N->part_cap * sizeof(float));
  }
  size_t total = 0;
  for (auto& r : req) total += (r.second + 255) / 256 * 256;
  if (cudaMalloc((void**)&N->base, total) != cudaSuccess) {
    cudaGetLastError();
    delete N;
    return BFCS_ERR_OOM;
  }
  size_t pos = 0;
  for (auto& r : req) {
    *r.first = N->base + pos;
    pos += (r.second + 255) / 256 * 256;
  }
  if (conv3_init() != cudaSuccess || wgrad3_init() != cudaSuccess ||
      wgrad1_init() != cudaSuccess) {
    cudaGetLastError();
    free_net(N);
    return BFCS_ERR_CUDA;
  }
  // zero everything once: padded input channels stay zero
  if (cudaMemsetAsync(N->base, 0, total, N->st) != cudaSuccess) { free_net(N); return BFCS_ERR_CUDA; }
  *out = N;
  return BFCS_OK;
}

int bfcs_net_status(bfcs_net N) {
  if (N == nullptr) return BFCS_ERR_INVALID_ARG;
  int h = 0;
  if (cudaMemcpyAsync(&h, N->err, sizeof(int), cudaMemcpyDeviceToHost, N->st) != cudaSuccess ||
      cudaStreamSynchronize(N->st) != cudaSuccess)
    return BFCS_ERR_CUDA;
  return h ? BFCS_ERR_TIMEOUT : BFCS_OK;
}

int bfcs_net_destroy(bfcs_net N) {
  if (N == nullptr) return BFCS_ERR_INVALID_ARG;
  cudaStreamSynchronize(N->st);
  free_net(N);
  return BFCS_OK;
}

int bfcs_net_prepare(bfcs_net N, int precision, const void* b, const int8_t* phase, int nphases,
                     const bfcs_lame* phases, const void* eps, float* x_out, float* target_out) {
  if (N == nullptr || b == nullptr || phase == nullptr || x_out == nullptr || (eps != nullptr && target_out == nullptr) ||
      (precision != BFCS_FP32 && precision != BFCS_FP64) || !valid_phases(nphases, phases))
    return BFCS_ERR_INVALID_ARG;
  MuTab mt;
  mu_table(nphases, phases, &mt);
  const long long n = N->n[0];
  cudaMemsetAsync(N->sbits, 0, sizeof(unsigned), N->st);
  if (precision == BFCS_FP64) {
    SampleArgs<double> sa{};
    sa.b[0] = (const double*)b;
    launch_chain(true, k_absmax<double>, std::min(304, grid_for(3 * n)), 256, 0, N->st, sa, 3 * n, N->sbits);
    launch_chain(true, k_prepare<double>, grid_for(n), 256, 0, N->st, (const double*)b, phase, mt, N->sbits,
                 (const double*)eps, x_out, target_out, n);
  } else {
    SampleArgs<float> sa{};
    sa.b[0] = (const float*)b;
    launch_chain(true, k_absmax<float>, std::min(304, grid_for(3 * n)), 256, 0, N->st, sa, 3 * n, N->sbits);
    launch_chain(true, k_prepare<float>, grid_for(n), 256, 0, N->st, (const float*)b, phase, mt, N->sbits,
                 (const float*)eps, x_out, target_out, n);
  }
  count_launches(2);
  return status_of(cudaGetLastError());
}

int bfcs_net_forward(bfcs_net N, const float* params, int batch, const float* x, float* y) {
  if (N == nullptr || params == nullptr || x == nullptr || y == nullptr || batch < 1 || batch > N->maxb)
    return BFCS_ERR_INVALID_ARG;
  cudaError_t e = pack_all(N, params);
  if (e == cudaSuccess) {
    launch_chain(true, k_features_in, grid_for(N->n[0] * batch), 256, 0, N->st, x, N->X0, N->n[0], batch);
    count_launches(1);
    e = forward(N, params, batch);
  }
  if (e == cudaSuccess) e = head_planar(N, params, batch, y);
  return status_of(e);
}

int bfcs_net_grad(bfcs_net N, const float* params, int batch, const float* x, const float* target, float* grad,
                  double* loss_dev) {
  if (N == nullptr || params == nullptr || x == nullptr || target == nullptr || grad == nullptr || batch < 1 ||
      batch > N->maxb || (N->flags & BFCS_NET_TRAIN) == 0)
    return BFCS_ERR_INVALID_ARG;
  cudaError_t e = pack_all(N, params);
  if (e == cudaSuccess) {
    launch_chain(true, k_features_in, grid_for(N->n[0] * batch), 256, 0, N->st, x, N->X0, N->n[0], batch);
    count_launches(1);
    e = forward(N, params, batch);
  }
  if (e == cudaSuccess) e = head_planar(N, params, batch, N->OUT);
  if (e == cudaSuccess) e = loss_and_grad(N, batch, target, loss_dev);
  if (e == cudaSuccess) e = backward(N, grad, batch);
  return status_of(e);
}

int bfcs_net_adam(bfcs_net N, float* params, const float* grad, float* m, float* v, long long t, float lr) {
  if (N == nullptr || params == nullptr || grad == nullptr || m == nullptr || v == nullptr || t < 1 ||
      !(lr > 0.f) || !std::isfinite(lr))
    return BFCS_ERR_INVALID_ARG;
  const float c1 = (float)(1.0 - std::pow(0.9, (double)t)), c2 = (float)(1.0 - std::pow(0.999, (double)t));
  const long long n = param_count();
  launch_chain(true, k_adam, grid_for(n), 256, 0, N->st, params, grad, m, v, n, lr, 0.9f, 0.999f, 1e-8f, c1, c2);
  count_launches(1);
  return status_of(cudaGetLastError());
}

int bfcs_net_train_step(bfcs_net N, float* params, float* grad, float* m, float* v, long long t, float lr, int batch,
                        const float* x, const float* target, double* loss_dev) {
  const int s = bfcs_net_grad(N, params, batch, x, target, grad, loss_dev);
  if (s != BFCS_OK) return s;
  return bfcs_net_adam(N, params, grad, m, v, t, lr);
}

int bfcs_net_predict(bfcs_net N, const float* params, int precision, int batch, const void* const* b,
                     const int8_t* const* phase, int nphases, const bfcs_lame* phases, void* const* eps_out) {
  if (N == nullptr || params == nullptr || batch < 1 || b == nullptr || phase == nullptr || eps_out == nullptr ||
      (precision != BFCS_FP32 && precision != BFCS_FP64) || !valid_phases(nphases, phases))
    return BFCS_ERR_INVALID_ARG;
  for (int i = 0; i < batch; ++i)
    if (b[i] == nullptr || phase[i] == nullptr || eps_out[i] == nullptr) return BFCS_ERR_INVALID_ARG;
  return precision == BFCS_FP64 ? predict<double>(N, params, batch, (const double* const*)b, phase, nphases, phases,
                                                  (double* const*)eps_out)
                                : predict<float>(N, params, batch, (const float* const*)b, phase, nphases, phases,
                                                 (float* const*)eps_out);
}

}  // extern "C"
