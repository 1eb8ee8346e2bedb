// The network's pointwise GEMMs: the 2^3 stride-2 transposed convolutions (a GEMM to
// 8 C columns and a pixel shuffle) and their data gradient (a gather and a GEMM), the
// 1^3 head and its data gradient.  All are streaming work of a few flops per byte,
// bound by HBM: a warp takes 32 rows (voxels) at a time on mma.sync m16n8k16 (BF16,
// FP32 accumulators), reads its operands straight from global memory and writes whole
// 32-byte sectors.
//
// The K order inside a block of 16 channels is permuted so that a lane's four values
// are neighbours (channel 16 s + 4 t + i for MMA indices 2t, 2t+1, 2t+8, 2t+9), the
// weights alike: an A fragment is one 8-byte load per row, a quad covering a 32-byte
// sector.  Columns are permuted within groups of 32 (MMA tile j, column 2t + e is
// channel 8 t + 2 j + e), so that a lane ends with 8 neighbouring channels of its row:
// one 16-byte store, a quad covering 64 bytes.  Weights sit in shared memory in
// fragment order (8 bytes a lane, conflict-free).
#include "unet_kernels.h"

#include <algorithm>

namespace bfcs {
namespace net {

namespace {

constexpr int kRowWarps = 8;
constexpr int kRowsPerWarp = 32;

}  // namespace

// KS blocks of 16 input channels, NG groups of 32 output columns (columns past
// cout_p are zero and not stored).  GATHER: K runs over the 8 fine voxels of a coarse
// one (up_c channels each), else over the row's channels.  SHUFFLE: group o goes to
// fine voxel 2u + o.  gate as in ConvArgs.
template <int KS, int NG, bool GATHER, bool SHUFFLE>
__global__ void __launch_bounds__(kRowWarps * 32) k_rows(ConvArgs a, unsigned rows) {
  extern __shared__ __align__(16) uint2 wfrag[];      // [KS][NG][4][32]
  __shared__ float bias_s[NG * 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  const int K = a.cin;
  for (int i = tid; i < KS * NG * 128; i += blockDim.x) {
    const int l = i & 31, j = (i >> 5) & 3, grp = (i >> 7) % NG, s = i / (128 * NG);
    const int col = grp * 32 + 8 * ((l >> 2) >> 1) + 2 * j + ((l >> 2) & 1);
    uint2 w = make_uint2(0u, 0u);
    if (col < a.cout_p) w = __ldcg(reinterpret_cast<const uint2*>(a.w + (long long)col * K + 16 * s + 4 * (l & 3)));
    wfrag[i] = w;
  }
  if (tid < NG * 32) bias_s[tid] = a.bias != nullptr && tid < a.cout_p ? __ldcg(a.bias + tid % a.bias_mod) : 0.f;
  chain_wait();
  __syncthreads();
  const unsigned nx = a.v.nx, ny = a.v.ny;
  const long long FX = 2 * nx, FY = 2 * ny;
  const unsigned step = gridDim.x * (kRowWarps * kRowsPerWarp);
  for (unsigned r0 = (blockIdx.x * kRowWarps + warp) * kRowsPerWarp; r0 < rows; r0 += step) {
    const bf16* rp[4];
    long long fine[4];                                // fine voxel 2u of the row (batch included)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned r = min(r0 + q * 8 + g, rows - 1);
      if (GATHER || SHUFFLE) {
        const unsigned x = r % nx, yz = r / nx, y = yz % ny, zb = yz / ny;   // zb = b nz + z
        fine[q] = ((long long)(2 * zb) * FY + 2 * y) * FX + 2 * x;
      }
      rp[q] = a.in + (GATHER ? fine[q] : (long long)r) * a.ldi + a.offi + 4 * t;
    }
    auto load = [&](int s, unsigned (&af)[2][4]) {
      long long ko;
      if (GATHER) {
        const int per = a.up_c >> 4, o = s / per;
        ko = ((long long)(o >> 2) * FY + ((o >> 1) & 1)) * FX * a.ldi + (long long)(o & 1) * a.ldi + 16 * (s - o * per);
      } else {
        ko = 16 * s;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint2 v = *reinterpret_cast<const uint2*>(rp[q] + ko);
        af[q >> 1][q & 1] = v.x;
        af[q >> 1][2 + (q & 1)] = v.y;
      }
    };
    auto store = [&](int grp, float (&acc)[2][4][4]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const unsigned r = r0 + q * 8 + g;
        const int col = grp * 32 + 8 * t;
        if (r >= rows || col >= a.cout_p) continue;
        __align__(16) __nv_bfloat162 o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float v0 = acc[q >> 1][j][2 * (q & 1)], v1 = acc[q >> 1][j][2 * (q & 1) + 1];
          if (a.bias != nullptr) { v0 += bias_s[col + 2 * j]; v1 += bias_s[col + 2 * j + 1]; }
          o[j] = __floats2bfloat162_rn(v0, v1);
        }
        if (a.gate != nullptr)
          gate8(o, *reinterpret_cast<const uint4*>(a.gate + (long long)r * a.ldg + a.offg + col));
        bf16* dst;
        if (SHUFFLE) {
          const long long fv = fine[q] + ((long long)(grp >> 2) * FY + ((grp >> 1) & 1)) * FX + (grp & 1);
          dst = (bf16*)a.out + fv * a.ldo + a.offo + 8 * t;
        } else {
          dst = (bf16*)a.out + (long long)r * a.ldo + a.offo + col;
        }
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(o);
      }
    };
    if constexpr (NG > KS) {
      // few K blocks, many columns: the rows stay in registers
      unsigned af[KS][2][4];
#pragma unroll
      for (int s = 0; s < KS; ++s) load(s, af[s]);
#pragma unroll 1
      for (int grp = 0; grp < NG; ++grp) {
        float acc[2][4][4] = {};
#pragma unroll
        for (int s = 0; s < KS; ++s)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint2 b = wfrag[((s * NG + grp) * 4 + j) * 32 + lane];
            mma16816(acc[0][j], af[s][0], b.x, b.y);
            mma16816(acc[1][j], af[s][1], b.x, b.y);
          }
        store(grp, acc);
        __syncwarp();
      }
    } else {
      float acc[NG][2][4][4] = {};
#pragma unroll 4
      for (int s = 0; s < KS; ++s) {
        unsigned af[2][4];
        load(s, af);
#pragma unroll
        for (int grp = 0; grp < NG; ++grp)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint2 b = wfrag[((s * NG + grp) * 4 + j) * 32 + lane];
            mma16816(acc[grp][0][j], af[0], b.x, b.y);
            mma16816(acc[grp][1][j], af[1], b.x, b.y);
          }
      }
#pragma unroll
      for (int grp = 0; grp < NG; ++grp) store(grp, acc[grp]);
      __syncwarp();
    }
  }
}

// (out of line: inlined it is computed for every value and selected)
__device__ __noinline__ float scaled_f64(float y, double f) { return (float)((double)y * f); }

// The head: 32 channels to 6 strain components, written planar (sample b's component
// c of voxel v at out[b][c n + v]) as FP32 (mode 0), or as the strain prediction
// y s_b / mu_max in R (mode 1).
template <typename R, bool PREDICT>
__global__ void __launch_bounds__(kRowWarps * 32) k_head(HeadArgs<R> a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  uint2 w[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) w[s] = __ldcg(reinterpret_cast<const uint2*>(a.w + g * 32 + 16 * s + 4 * t));   // column g
  const float b0 = 2 * t < 6 ? __ldcg(a.bias + 2 * t) : 0.f, b1 = 2 * t + 1 < 6 ? __ldcg(a.bias + 2 * t + 1) : 0.f;
  chain_wait();
  const int b = blockIdx.y;
  const bf16* in = a.in + (long long)b * a.n * 32;
  R* out = a.out[b];
  double fd = 0.0;
  ff fs = ff(0.0f);
  bool fast = false;
  if (PREDICT) {
    fd = (double)__uint_as_float(a.sbits[b]) / a.mu_max;
    fs = ff(fd);
    fast = fd > 1e-18 && fd < 1e18;
  }
  // y s / mu_max.  FP32 fields: from float-float arithmetic where it rounds as FP64 does;
  // FP64 multiplies and conversions of every value would bind the pass to the FP64 pipe (16
  // us a 64^3 sample), so they serve only the other values (one in 2^18) and those whose
  // product's parts could leave the FP32 range.
  auto value = [&](float y) -> R {
    if constexpr (!PREDICT) return y;
    else if constexpr (sizeof(R) == 8) return (double)y * fd;
    else {
      const float m = fabsf(y);
      const ff r = ff(y) * fs;
      return fast && m > 1e-12f && m < 1e15f && ff_rounds_as_fp64(r) ? r.hi : scaled_f64(y, fd);
    }
  };
  const unsigned n = (unsigned)a.n;
  const unsigned step = gridDim.x * (kRowWarps * kRowsPerWarp);
  for (unsigned r0 = (blockIdx.x * kRowWarps + warp) * kRowsPerWarp; r0 < n; r0 += step) {
    unsigned af[2][2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bf16* rp = in + (long long)min(r0 + q * 8 + g, n - 1) * 32 + 4 * t;
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const uint2 v = *reinterpret_cast<const uint2*>(rp + 16 * s);
        af[s][q >> 1][q & 1] = v.x;
        af[s][q >> 1][2 + (q & 1)] = v.y;
      }
    }
    float acc[2][4] = {};
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      mma16816(acc[0], af[s][0], w[s].x, w[s].y);
      mma16816(acc[1], af[s][1], w[s].x, w[s].y);
    }
    if (t < 3) {                                      // columns 6 and 7 are padding
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const unsigned r = r0 + q * 8 + g;
        if (r >= n) continue;
        const float v0 = acc[q >> 1][2 * (q & 1)] + b0, v1 = acc[q >> 1][2 * (q & 1) + 1] + b1;
        R* o = out + (long long)(2 * t) * a.n + r;
        o[0] = value(v0);
        o[a.n] = value(v1);
      }
    }
    __syncwarp();
  }
}

namespace {

template <int KS, int NG, bool GATHER, bool SHUFFLE>
cudaError_t rows_launch(const ConvArgs& a, unsigned rows, int sms, cudaStream_t st) {
  const unsigned blocks = std::min<unsigned>((rows + kRowWarps * kRowsPerWarp - 1) / (kRowWarps * kRowsPerWarp), 4u * sms);
  launch_chain(true, k_rows<KS, NG, GATHER, SHUFFLE>, blocks, kRowWarps * 32, KS * NG * 128 * sizeof(uint2), st, a, rows);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

// The shapes of the network's pointwise layers: up-convolutions 48 -> 8 x 32 and
// 32 -> 8 x 32, their data gradients 8 x 32 -> 48 (two column groups) and 32, and the
// head's data gradient 16 -> 32.
bool rows_ok(const ConvArgs& a) {
  if (a.ksize != 1 || a.act || a.ldi % 8 || a.offi % 8 || a.ldo % 8 || a.offo % 8) return false;
  if (a.out_mode == OUT_SHUFFLE_UP && a.in_mode == IN_CONV)
    return a.up_c == 32 && a.cout_p == 256 && (a.cin == 32 || a.cin == 48);
  if (a.out_mode != OUT_BF16) return false;
  if (a.in_mode == IN_GATHER_UP) return a.up_c == 32 && a.cin == 256 && (a.cout_p == 32 || a.cout_p == 48);
  return a.cin == 16 && a.cout_p == 32;
}

cudaError_t launch_rows(const ConvArgs& a, int sms, cudaStream_t st) {
  const unsigned rows = (unsigned)((long long)a.v.nx * a.v.ny * a.v.nz * a.batch);
  if (a.out_mode == OUT_SHUFFLE_UP)
    return a.cin == 48 ? rows_launch<3, 8, false, true>(a, rows, sms, st) : rows_launch<2, 8, false, true>(a, rows, sms, st);
  if (a.in_mode == IN_GATHER_UP)
    return a.cout_p == 48 ? rows_launch<16, 2, true, false>(a, rows, sms, st)
                          : rows_launch<16, 1, true, false>(a, rows, sms, st);
  return rows_launch<1, 1, false, false>(a, rows, sms, st);
}

template <typename R>
cudaError_t launch_head(const HeadArgs<R>& a, int batch, bool predict, int sms, cudaStream_t st) {
  const long long per = kRowWarps * kRowsPerWarp;
  const unsigned bx = (unsigned)std::max<long long>(1, std::min((a.n + per - 1) / per, (long long)(8 * sms / batch + 1)));
  if (predict) {
    launch_chain(true, k_head<R, true>, dim3(bx, batch), kRowWarps * 32, 0, st, a);
  } else {
    if constexpr (sizeof(R) == 4) launch_chain(true, k_head<R, false>, dim3(bx, batch), kRowWarps * 32, 0, st, a);
    else return cudaErrorInvalidValue;
  }
  count_launches(1);
  return cudaGetLastError();
}
template cudaError_t launch_head<float>(const HeadArgs<float>&, int, bool, int, cudaStream_t);
template cudaError_t launch_head<double>(const HeadArgs<double>&, int, bool, int, cudaStream_t);

}  // namespace net
}  // namespace bfcs
