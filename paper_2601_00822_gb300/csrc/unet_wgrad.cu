// Weight gradients of the 3^3 circular convolutions on tcgen05 (32 output channels):
// dW[dz, dy, dx][co][ci] = sum over voxels v of dY[v][co] X[v + d][ci].
//
// With w = v + dx one MMA covers the nine pairs (dz, dx) of a row of taps dy at once:
//   A = X over four consecutive planes of one 8 x 16 voxel column (M = 128 rows: plane
//       dz, 32 input channels; the fourth plane's rows are not used),
//   B = three copies of the dY plane, copy dx shifted by dx - 1 along x (N = 96
//       columns: dx, 32 output channels),
//   K = the plane's 128 voxels in blocks of 16 (two rows of 8).
// dy is a row offset of A's start address (whole rows of 8 voxels, so every start keeps
// the swizzle's 512-byte alignment).  Both operands are MN-major in the 64-byte swizzle:
// voxel v's 32 channels are 64 contiguous bytes at 64 v, 8-channel chunk c at 16-byte slot
// c ^ ((v >> 1) & 3); eight voxels are one atom, the next eight 512 B further (SBO), the
// next 32 channels one plane or copy further (LBO).  A voxel's four 16-byte copies land
// side by side, which the copies need: in the chunk-planar layout of the convolutions
// each fetched its 32-byte sector alone, twice the traffic from L2, and at 72 KB a tile
// that bound the pass (209 us for the level-0 layer of 8 samples at 64^3).  Three
// accumulators (dy) of 96 TMEM columns.
//
// The tensor core truncates when it accumulates, and a sum over a block's whole run
// (860 steps for 8 samples of 64^3) came out 1.7e-5 off.  So every kFlush tiles the
// worker warps add the accumulators to FP32 sums in registers, rounding to nearest, and
// the next tile starts from zero.
//
// A block marches along z over a run of tiles like k_conv3.  The four planes must lie
// one after another, so planes are staged in segments of up to kSeg tiles (kSeg + 2 planes
// in kSeg + 3 slots, the last one never written: it only feeds unused rows), and the slots
// of finished tiles take the next segment's planes.  Voxels outside the grid (partial
// tiles) have their dY zero-filled.  At the end the block writes its partial sums; they
// are added in block order (k_reduce_grad).
//
// What bounds it: an MMA reads (128 + 96) * 32 B of shared memory, 56 clocks at 128 B a
// clock; 24 per tile, so 1344 clocks against 9 * 8 * 40 = 2880 with one MMA per (dy,
// dx) on a plain dY plane, and staging three dY copies adds about 270 clocks of writes.
// The 3^3 layers of a gradient over 8 samples of 64^3 take 0.79 ms together, 3.48 ms with
// nine warps of mma.sync and sums over the blocks as a launch of their own.  A thread keeps
// 144 running sums; the ninth warp makes one quarter of an SM hold three, which leaves 168
// registers a thread, and 420 bytes of the staging's state spill (-Xptxas -v).
#include "unet_kernels.h"
#include "unet_tc.cuh"
#include "unet_wgrad_flow.h"

#include <algorithm>

namespace bfcs {
namespace net {

namespace {

constexpr int kGX = 8, kGY = 16, kGV = kGX * kGY;     // tile (one z plane)
constexpr int kGHY = kGY + 2;
constexpr int kSlots = kSeg + 3;
constexpr unsigned kXPlane = kGX * kGHY * 64;         // one staged plane: 8 x 18 voxels
constexpr unsigned kYCopy = kGV * 64, kYTile = 3 * kYCopy;
constexpr unsigned kWgSmem = kSlots * kXPlane + kYRing * kYTile;
constexpr unsigned kWgCols = 512;                     // TMEM allocation (3 x 96 columns used)
constexpr int kXN = (kGX * kGHY * 4 + kTcWorkers - 1) / kTcWorkers;   // X copies per thread and plane
constexpr int kYN = kGV * 12 / kTcWorkers;            // dY copies per thread and tile

// byte offset of channel chunk c of voxel v (64-byte swizzle)
__device__ __forceinline__ unsigned swz(int v, int c) { return (unsigned)v * 64u + (unsigned)((c ^ (v >> 1)) & 3) * 16u; }

}  // namespace

// cin channels of the 32-channel half blockIdx.y (cin = 16: chunks 2 and 3 are zero)
__global__ void __launch_bounds__(kTcWorkers + 32, 1) k_wgrad3(WgArgs a, int* err) {
  chain_wait();
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bars[3 + kYRing];   // full 0/1, done 0..2, drained
  __shared__ unsigned tmem_s;
  __shared__ int fail_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* const fail = &fail_s;
  const unsigned xs = (unsigned)__cvta_generic_to_shared(smem), ys = xs + kSlots * kXPlane;
  const unsigned full = (unsigned)__cvta_generic_to_shared(bars), done = full + 16, drained = done + 8 * kYRing;
  const int ntx = (a.v.nx + kGX - 1) / kGX, nty = (a.v.ny + kGY - 1) / kGY, nz = a.v.nz;
  const long long total = (long long)ntx * nty * nz * a.batch;
  const long long t0 = total * blockIdx.x / gridDim.x, t1 = total * (blockIdx.x + 1) / gridDim.x;
  const int n = (int)(t1 - t0);
  // (sticky error flag as in k_conv3; n >= 1: the grid has at most `total` blocks)
  if (__syncthreads_or(tid == 0 && *(volatile int*)err != 0) || n <= 0) return;
  if (warp == 8) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(&tmem_s);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dst), "r"(kWgCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  if (tid == 0) {
    fail_s = 0;
    for (int i = 0; i < 2 + kYRing; ++i) mbar_init(full + 8 * i, 1);
    mbar_init(drained, kTcWorkers / 32);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  tc_before();
  __syncthreads();
  tc_after();
  const unsigned tmem = tmem_s;

  if (warp == 8) {
    // ---- MMA issue
    const unsigned tm = __shfl_sync(0xffffffffu, tmem, 0);
    int z = (int)(t0 % nz), pos = 0, yr = 0;
    for (int k = 0; k < n; ++k) {
      bool ok = mbar_wait(full + 8 * (k & 1), (unsigned)((k >> 1) & 1), fail);
      if (ok && k > 0 && k % kFlush == 0) ok = mbar_wait(drained, (unsigned)((k / kFlush - 1) & 1), fail);
      if (!ok) {
        if (lane == 0) { *fail = 1; atomicExch(err, 1); }
        break;
      }
      tc_after();
      if (elect_one()) {
        const uint64_t ad0 = sdesc(xs + (unsigned)pos * kXPlane, kXPlane, 512) | kDescSwizzle64;
        const uint64_t bd0 = sdesc(ys + (unsigned)yr * kYTile, kYCopy, 512) | kDescSwizzle64;
        const unsigned acc = k % kFlush != 0 ? 1u : 0u;
#pragma unroll
        for (int ks = 0; ks < kGY / 2; ++ks) {
#pragma unroll
          for (int dy = 0; dy < 3; ++dy) {
            const uint64_t ad = ad0 + (unsigned)((2 * ks + dy) * 32);   // 16-byte units
            const uint64_t bd = bd0 + (unsigned)(2 * ks * 32);
            asm volatile(
                "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tm + 96u * dy),
                "l"(ad), "l"(bd), "r"(idesc_bf16(128, 96) | kIdescMnMajorAB), "r"(ks > 0 ? 1u : acc));
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                         done + 8u * (unsigned)yr)
                     : "memory");
      }
      __syncwarp();
      pos = wg_next_pos(z, nz, pos);
      z = z + 1 == nz ? 0 : z + 1;
      yr = yr + 1 == kYRing ? 0 : yr + 1;
    }
  } else {
    // ---- staging
    const long long nvox = (long long)a.v.nx * a.v.ny * nz, plane = (long long)a.v.nx * a.v.ny;
    const int c0 = blockIdx.y * 4;                     // first chunk of this half
    // this thread's copies in plane 0 of the loading column, as offsets in 16-byte units
    // from the sample's first voxel
    const bf16 *xbase = nullptr, *ybase = nullptr;
    unsigned xsrc[kXN], ysrc[kYN], yvalid = 0;
    const unsigned ldx8 = a.ldx / 8, ldd8 = a.ldd / 8;
    auto set_column = [&](long long col) {
      const int x0 = (int)(col % ntx) * kGX;
      col /= ntx;
      const int y0 = (int)(col % nty) * kGY, b = (int)(col / nty);
      xbase = a.x + (long long)b * nvox * a.ldx + a.offx;
      ybase = a.dy + (long long)b * nvox * a.ldd + a.offd;
#pragma unroll
      for (int j = 0; j < kXN; ++j) {
        const int i = tid + j * kTcWorkers, v = i / 4, c = i % 4;
        // (rows and voxels past the grid read wrapped values; their dY is zero)
        const int gx = (x0 + v % kGX) % a.v.nx, gy = (y0 + v / kGX - 1 + a.v.ny) % a.v.ny;
        xsrc[j] = (unsigned)(gy * a.v.nx + gx) * ldx8 + (unsigned)(c0 + c);
      }
      yvalid = 0;
#pragma unroll
      for (int j = 0; j < kYN; ++j) {
        const int i = tid + j * kTcWorkers, c = i % 4, v = (i / 4) % kGV, dx = i / (4 * kGV);
        const int wx = x0 + v % kGX, wy = y0 + v / kGX;
        if (wx < a.v.nx && wy < a.v.ny) yvalid |= 1u << j;
        const int gx = (wx - (dx - 1) + a.v.nx) % a.v.nx, gy = wy % a.v.ny;
        ysrc[j] = (unsigned)(gy * a.v.nx + gx) * ldd8 + (unsigned)c;
      }
    };
    // where there is nothing to copy zeros are stored
    auto copy = [&](unsigned dst, const bf16* src, bool valid) {
      if (valid) cp16(dst, src);
      else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};\n" ::"r"(dst), "r"(0u) : "memory");
    };
    auto load_x = [&](int z, int slot) {
      const bf16* base = xbase + (long long)wrap(z, nz) * plane * a.ldx;
#pragma unroll
      for (int j = 0; j < kXN; ++j) {
        const int i = tid + j * kTcWorkers, v = i / 4, c = i % 4;
        if (v < kGX * kGHY)
          copy(xs + (unsigned)slot * kXPlane + swz(v, c), base + (long long)xsrc[j] * 8, (c0 + c) * 8 < a.cin);
      }
    };
    auto load_y = [&](int z, int r) {
      const bf16* base = ybase + (long long)z * plane * a.ldd;
#pragma unroll
      for (int j = 0; j < kYN; ++j) {
        const int i = tid + j * kTcWorkers, c = i % 4, v = (i / 4) % kGV, dx = i / (4 * kGV);
        copy(ys + (unsigned)r * kYTile + (unsigned)dx * kYCopy + swz(v, c), base + (long long)ysrc[j] * 8,
             (yvalid >> j) & 1u);
      }
    };
    set_column(t0 / nz);
    auto request = [&](const WgTile& t, int slot) {
      if (t.z == 0) set_column(t.col);                 // a new column
      if (t.pos == 0) { load_x(t.z - 1, 0); load_x(t.z, 1); }
      load_x(t.z + 1, t.pos + 2);
      load_y(t.z, slot);
      cp_commit();
    };
    auto landed = [&](int younger) {
      if (younger >= 2) cp_wait<2>();
      else if (younger == 1) cp_wait<1>();
      else cp_wait<0>();
      fence_async();
    };
    // running sums: TMEM lane = 32 dz + ci, column = 96 dy + 32 dx + co; the two warps of a
    // quarter dz take alternate 16-column slices
    const int dz = warp & 3;
    float sum[9][16] = {};
    // bias gradient: this thread's chunk (tid % 4) of dY over voxels tid / 4 and tid / 4 + 64
    // of every tile, from the unshifted copy, once the tile has landed for all threads
    float bsum[8] = {};
    auto bias = [&](int r) {
      if (blockIdx.y != 0) return;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned off = kSlots * kXPlane + (unsigned)r * kYTile + kYCopy + swz((tid >> 2) + 64 * h, tid & 3);
        const uint4 v = *reinterpret_cast<const uint4*>(smem + off);
#pragma unroll
        for (int q = 0; q < 8; ++q) bsum[q] += __bfloat162float(reinterpret_cast<const bf16*>(&v)[q]);
      }
    };
    auto publish = [&](int k) {
      if (tid == 0) mbar_arrive(full + 8 * (k & 1));
    };
    auto wait_done = [&](int slot, int phase) {
      const bool ok = mbar_wait(done + 8 * slot, (unsigned)phase, fail);
      if (!ok && lane == 0) { *fail = 1; atomicExch(err, 1); }
      return ok;
    };
    auto drain = [&](bool ok) {
      if (ok && dz < 3) {
        tc_after();
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          unsigned v[16];
          tmem_ld16(v, tmem + ((unsigned)(dz * 32) << 16) + 16u * (unsigned)(2 * i + (warp >> 2)));
#pragma unroll
          for (int j = 0; j < 16; ++j) sum[i][j] += __uint_as_float(v[j]);
        }
        tc_before();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(drained);
    };
    const bool ok = wgrad3_workers(n, nz, t0, request, landed, workers_all, publish, bias, wait_done, drain);
    if (ok && blockIdx.y == 0) {                       // threads of a channel added in thread order
      float* red = reinterpret_cast<float*>(smem);     // [tid / 4][32] (every MMA and copy is done)
#pragma unroll
      for (int q = 0; q < 8; ++q) red[(tid >> 2) * 32 + (tid & 3) * 8 + q] = bsum[q];
      workers_all(true);
      if (tid < 32) {
        float t = 0.f;
        for (int q = 0; q < 64; ++q) t += red[q * 32 + tid];
        a.bpart[(long long)blockIdx.x * 32 + tid] = t;
      }
    }
    const int ci = blockIdx.y * 32 + lane;
    if (ok && dz < 3 && ci < a.cin) {
      float* out = a.part + (long long)blockIdx.x * 27 * 32 * a.cin + ci;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const int q = 2 * i + (warp >> 2), dy = q / 6, dx = (q % 6) / 2, co0 = (q & 1) * 16;
#pragma unroll
        for (int j = 0; j < 16; ++j) out[((long long)((dz * 3 + dy) * 3 + dx) * 32 + co0 + j) * a.cin] = sum[i][j];
      }
    }
  }
  // (after an expired wait the last MMAs may still be in flight: see k_conv3)
  tc_before();
  __syncthreads();
  tc_after();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_s), "r"(kWgCols));
}

// Weight gradients of the pointwise layers: the up-convolutions (UP: dW[o 32 + co][ci] =
// sum over coarse voxels u of dY[2u + o][co] X[u][ci], o the 8 sub-voxels) and the head
// (dW[co][ci] over voxels).  A few flops per byte: streaming, bound by HBM.  Each warp
// stages its own 32 rows at a time with cp.async (two stages, no block barriers) and
// transposes them into fragments with ldmatrix; its MMA sums over four stages are added
// to running FP32 sums with rounding (see above).  UP: four warps take two sub-voxels
// each, two row streams per block, one partial per stream; head: eight row streams per
// block, added in warp order into one partial.
namespace {

constexpr int kW1Rows = 32;

// row pitches: 16-byte multiples that put 8 consecutive rows on distinct banks
template <int NP, bool UP> struct W1 {
  static constexpr int MT = UP ? 4 : 1;               // 16-row tiles of this warp's output channels
  static constexpr unsigned AP = UP ? 80 : 48;        // 32 or 16 channels
  static constexpr unsigned XP = NP == 2 ? 80 : 112;  // 32 or 48 channels
  static constexpr unsigned A = (UP ? 2 : 1) * kW1Rows * AP, STAGE = A + kW1Rows * XP;
  static constexpr unsigned SMEM = 8 * 2 * STAGE;     // 8 warps, 2 stages
};

}  // namespace

template <int NP, bool UP>
__global__ void __launch_bounds__(256) k_wgrad1(WgArgs a, unsigned rows) {
  chain_wait();
  using C = W1<NP, UP>;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned buf = (unsigned)__cvta_generic_to_shared(smem) + (unsigned)warp * 2u * C::STAGE;
  const int streams = UP ? 2 : 8, stream = UP ? warp >> 2 : warp;
  const int o0 = UP ? (warp & 3) * 2 : 0;             // first of this warp's two sub-voxels
  const unsigned units = (rows + kW1Rows - 1) / kW1Rows;
  const unsigned s_all = gridDim.x * streams, s_id = blockIdx.x * streams + stream;
  const unsigned u0 = (unsigned)((unsigned long long)units * s_id / s_all);
  const unsigned u1 = (unsigned)((unsigned long long)units * (s_id + 1) / s_all);
  const unsigned nx = a.v.nx, ny = a.v.ny;
  const long long FX = 2 * nx, FY = 2 * ny;
  auto stage = [&](unsigned u, unsigned base) {
    const int c = lane & 3;
#pragma unroll
    for (int q = 0; q < 4; ++q) {                     // 4 lanes to a row: rows lane / 4 + 8 q
      const unsigned lr = (lane >> 2) + 8 * q, row = u * kW1Rows + lr;
      const bool in = row < rows;
      const unsigned r = in ? row : rows - 1;
      if (UP) {
        const unsigned x = r % nx, yz = r / nx, y = yz % ny, zb = yz / ny;
        const long long f = ((long long)(2 * zb) * FY + 2 * y) * FX + 2 * x;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int o = o0 + h;
          const long long fv = f + ((long long)(o >> 2) * FY + ((o >> 1) & 1)) * FX + (o & 1);
          cp16_fill(base + (h * kW1Rows + lr) * C::AP + c * 16u, a.dy + fv * a.ldd + a.offd + c * 8, in);
        }
      } else if (c < 2) {
        cp16_fill(base + lr * C::AP + c * 16u, a.dy + (long long)r * a.ldd + a.offd + c * 8, in);
      }
#pragma unroll
      for (int cc = 0; cc < NP * 2; cc += 4)
        if (cc + c < NP * 2)
          cp16_fill(base + C::A + lr * C::XP + (cc + c) * 16u, a.x + (long long)r * a.ldx + a.offx + (cc + c) * 8, in);
    }
    cp_commit();
  };
  // the bias gradient rides along as one more column tile, dY times a column of ones
  float sum[C::MT][2 * NP + 1][4] = {}, acc[C::MT][2 * NP + 1][4] = {};
  const unsigned ones = 0x3F803F80u;
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < C::MT; ++i)
#pragma unroll
      for (int j = 0; j < 2 * NP + 1; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) { sum[i][j][q] += acc[i][j][q]; acc[i][j][q] = 0.f; }
  };
  if (u0 < u1) stage(u0, buf);
  for (unsigned u = u0; u < u1; ++u) {
    const unsigned base = buf + ((u - u0) & 1) * C::STAGE;
    if (u + 1 < u1) {
      stage(u + 1, buf + ((u + 1 - u0) & 1) * C::STAGE);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncwarp();
    const int mi = lane >> 3, rr = lane & 7;
#pragma unroll
    for (int ks = 0; ks < kW1Rows; ks += 16) {
      unsigned bq[NP][4];
#pragma unroll
      for (int p = 0; p < NP; ++p)
        ldsm_x4_trans(bq[p], base + C::A + (ks + (mi & 1) * 8 + rr) * C::XP + (p * 16 + (mi >> 1) * 8) * 2u);
#pragma unroll
      for (int i = 0; i < C::MT; ++i) {
        unsigned af[4];
        ldsm_x4_trans(af, base + ((i >> 1) * kW1Rows + ks + (mi >> 1) * 8 + rr) * C::AP + ((i & 1) * 16 + (mi & 1) * 8) * 2u);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          mma16816(acc[i][2 * p], af, bq[p][0], bq[p][1]);
          mma16816(acc[i][2 * p + 1], af, bq[p][2], bq[p][3]);
        }
        mma16816(acc[i][2 * NP], af, ones, ones);
      }
    }
    if (((u - u0) & 3) == 3) flush();
    __syncwarp();                                     // the stage is read before the next copies into it
  }
  flush();
  const int g = lane >> 2, t = lane & 3;
  const int cin = NP * 16;
  if (UP) {
    float* out = a.part + (long long)s_id * a.cout_p * cin;
#pragma unroll
    for (int i = 0; i < C::MT; ++i)
#pragma unroll
      for (int j = 0; j < 2 * NP; ++j) {
        const int co = o0 * 32 + i * 16 + g, ci = j * 8 + 2 * t;
        *reinterpret_cast<float2*>(out + co * cin + ci) = make_float2(sum[i][j][0], sum[i][j][1]);
        *reinterpret_cast<float2*>(out + (co + 8) * cin + ci) = make_float2(sum[i][j][2], sum[i][j][3]);
      }
    // bias: the two sub-voxels of a warp, then the warps in order
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);      // [warp][32]
    if (t == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        red[warp * 32 + i * 16 + g] = sum[i][2 * NP][0] + sum[i + 2][2 * NP][0];
        red[warp * 32 + i * 16 + g + 8] = sum[i][2 * NP][2] + sum[i + 2][2 * NP][2];
      }
    }
    __syncthreads();
    if (tid < 32) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[w * 32 + tid];
      a.bpart[(long long)blockIdx.x * 32 + tid] = s;
    }
  } else {
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);      // [warp][16][32], then [warp][16]
    if (t == 0) {
      red[4096 + warp * 16 + g] = sum[0][2 * NP][0];
      red[4096 + warp * 16 + g + 8] = sum[0][2 * NP][2];
    }
#pragma unroll
    for (int j = 0; j < 2 * NP; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) red[warp * 512 + (g + (q >> 1) * 8) * 32 + j * 8 + 2 * t + (q & 1)] = sum[0][j][q];
    __syncthreads();
    for (int i = tid; i < 512; i += 256) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[w * 512 + i];
      a.part[(long long)blockIdx.x * 512 + i] = s;
    }
    if (tid < 16) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[4096 + w * 16 + tid];
      a.bpart[(long long)blockIdx.x * 16 + tid] = s;
    }
  }
}

// up-convolutions with 32 or 48 input channels, the head (16 padded output channels)
bool wgrad1_ok(const WgArgs& a) {
  if (a.ksize != 1 || a.ldd % 8 || a.offd % 8 || a.ldx % 8 || a.offx % 8) return false;
  return a.up_c == 32 ? a.cout_p == 256 && (a.cin == 32 || a.cin == 48) : a.up_c == 0 && a.cout_p == 16 && a.cin == 32;
}

cudaError_t wgrad1_init() {
  cudaError_t e = cudaFuncSetAttribute(k_wgrad1<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W1<2, true>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad1<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W1<3, true>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad1<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W1<2, false>::SMEM);
  return e;
}

static int wgrad1_blocks(const WgArgs& a, int sms) {
  const long long units = ((long long)a.v.nx * a.v.ny * a.v.nz * a.batch + kW1Rows - 1) / kW1Rows;
  const int streams = a.up_c ? 2 : 8;
  return (int)std::max<long long>(1, std::min<long long>((units + streams - 1) / streams, a.up_c ? sms : 2 * sms));
}
int wgrad1_chunks(const WgArgs& a, int sms) { return wgrad1_blocks(a, sms) * (a.up_c ? 2 : 1); }

cudaError_t launch_wgrad1(const WgArgs& a, int sms, cudaStream_t st) {
  const unsigned rows = (unsigned)((long long)a.v.nx * a.v.ny * a.v.nz * a.batch);
  const int blocks = wgrad1_blocks(a, sms);
  if (a.up_c == 0) launch_chain(true, k_wgrad1<2, false>, blocks, 256, W1<2, false>::SMEM, st, a, rows);
  else if (a.cin == 32) launch_chain(true, k_wgrad1<2, true>, blocks, 256, W1<2, true>::SMEM, st, a, rows);
  else launch_chain(true, k_wgrad1<3, true>, blocks, 256, W1<3, true>::SMEM, st, a, rows);
  count_launches(1);
  return cudaGetLastError();
}

bool wgrad3_ok(const WgArgs& a) {
  return a.ksize == 3 && a.up_c == 0 && a.cout_p == 32 && (a.cin == 16 || a.cin == 32 || a.cin == 64) &&
         a.ldd % 8 == 0 && a.offd % 8 == 0 && a.ldx % 8 == 0 && a.offx % 8 == 0;
}

cudaError_t wgrad3_init() {
  return cudaFuncSetAttribute(k_wgrad3, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWgSmem);
}

int wgrad3_chunks(const WgArgs& a, int sms) {
  const long long tiles = (long long)((a.v.nx + kGX - 1) / kGX) * ((a.v.ny + kGY - 1) / kGY) * a.v.nz * a.batch;
  return (int)std::min<long long>(tiles, sms / (a.cin > 32 ? a.cin / 32 : 1));
}

cudaError_t launch_wgrad3(const WgArgs& a, int chunks, int* err, cudaStream_t st) {
  launch_chain(true, k_wgrad3, dim3(chunks, a.cin > 32 ? a.cin / 32 : 1), kTcWorkers + 32, kWgSmem, st, a, err);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace net
}  // namespace bfcs
