// 3^3 circular convolutions of the network on the 5th-generation tensor cores
// (tcgen05.mma kind::f16, BF16 operands, FP32 accumulators in tensor memory).
//
// A block owns a run of 128-voxel tiles (8 x-voxels x 16 y-rows x one z plane) in
// z-fastest order and marches along z.  It keeps the layer's weights and a ring of
// four input planes (10 x 18 voxels, circular halo, all input channels) in shared
// memory: three planes feed the tile at hand and the fourth receives the next
// tile's, so a step loads one plane where a tile on its own loads three.
//
// Operand layout: canonical K-major, no swizzle.  8-channel chunk c of halo voxel v
// of a plane at byte (c * PV + v) * 16: eight consecutive x-voxels are one 8 x 16 B
// core matrix, the next tile row 10 voxels further (SBO) and the next chunk PV
// voxels further (LBO), so every tap's A operand is the same descriptor at another
// start address.  PV (>= 180) spreads the cp.async writes of a quarter warp over all
// banks.  Weights: chunk c of output channel n of tap t at ((t KC + c) N + n) * 16
// (SBO 128 B, LBO 16 N B).
//
// Roles: warps 0-7 stage planes with cp.async and drain the accumulators (tcgen05.ld,
// bias, leaky ReLU or the gate of a data gradient, BF16 store); one elected thread of warp 8 issues the 27 KC / 2
// MMAs of a tile.  Two accumulators: the epilogue and the next plane's copies run
// under the next tile's MMAs.  Barriers (mbarrier, two of each, used by alternate
// tiles): full = operands staged, done = MMAs complete (tcgen05.commit), empty =
// accumulator drained.  Each wait is bounded; an expired one sets *err (sticky, see
// the kernel's exit) and every role leaves.
//
// What bounds it: a 128 x N x 16 MMA reads (128 + N) * 32 B of shared memory at 128 B
// per clock: 40 clocks at N = 32 and 48 at N = 64 (measured), against 16-32 clocks of
// tensor-core arithmetic, so a tile of a 32 -> 32 layer takes at least 54 * 40 = 2160
// clocks.  Issuing the MMAs costs as much again unless descriptors are formed from
// compile-time tap offsets on the uniform data path: a rolled tap loop on thread 0
// measured 122 clocks per MMA, the unrolled loop under elect.sync 48.
//
// Measured over a prediction of 16 samples of 64^3, averages of the launches: 32 -> 32
// layers 358 -> 97 us, 64 -> 32 layers 966 -> 231 us, against one tile's halo staged at a
// time and MMAs issued by thread 0.  The level-0 layers take 143 us (121 by the MMA bound
// above) and 565 us (486; their weights leave room for one block an SM).
#include "unet_kernels.h"
#include "unet_tc.cuh"

#include <algorithm>

namespace bfcs {
namespace net {

namespace {

constexpr int kCX = 8, kCY = 16;                      // tile
constexpr int kCHX = kCX + 2, kCHY = kCY + 2;         // halo plane
constexpr int kCHalo = kCHX * kCHY;
constexpr int kRing = 4;
constexpr int kWorkers = kTcWorkers;                  // warps 0-7
constexpr int kConv3Threads = kWorkers + 32;

template <int KC, int N> struct C3 {
  // plane pitch in voxels: chunk stride 16 PV such that the 16-byte writes of 8 / KC
  // voxels x KC chunks fall on distinct banks (16 PV mod 128 = 64, 96, 80 for KC = 2, 4, 8)
  static constexpr int PV = KC == 2 ? 180 : KC == 4 ? 182 : 181;
  static constexpr unsigned PLANE = KC * PV * 16u;
  static constexpr unsigned WBYTES = 27u * KC * N * 16u;
  static constexpr unsigned SMEM = kRing * PLANE + WBYTES;
  // blocks per SM by shared memory (227 KB, 1 KB reserved per block); a second block
  // keeps the tensor pipe busy across a block's column changes
  static constexpr int BLOCKS = SMEM + 1536 <= 75u * 1024 ? 3 : SMEM + 1536 <= 113u * 1024 ? 2 : 1;
  static constexpr int ACC = N <= 32 ? 32 : 64;       // TMEM columns of one accumulator (a power of two in all)
  static constexpr int NJ = (kCHalo * KC + kWorkers - 1) / kWorkers;   // plane copies per thread
};

// column col of tiles (x fastest, then y, then the sample)
__device__ __forceinline__ void conv3_column(const ConvArgs& a, long long col, int& b, int& x0, int& y0) {
  const int ntx = (a.v.nx + kCX - 1) / kCX, nty = (a.v.ny + kCY - 1) / kCY;
  x0 = (int)(col % ntx) * kCX;
  col /= ntx;
  y0 = (int)(col % nty) * kCY;
  b = (int)(col / nty);
}

// worker tid's copies in plane 0 of column col
template <int KC, int NJ>
__device__ __forceinline__ void conv3_sources(const ConvArgs& a, long long col, int tid, const bf16* (&src)[NJ]) {
  int b, x0, y0;
  conv3_column(a, col, b, x0, y0);
  const bf16* inb = a.in + (long long)b * ((long long)a.v.nx * a.v.ny * a.v.nz) * a.ldi + a.offi;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int i = tid + j * kWorkers;
    const int v = i / KC, c = i % KC;
    // (a partial tile's rows past the grid read wrapped voxels; they are not stored)
    const int gx = (x0 + v % kCHX - 1 + a.v.nx) % a.v.nx, gy = (y0 + v / kCHX - 1 + a.v.ny) % a.v.ny;
    src[j] = inb + ((long long)gy * a.v.nx + gx) * a.ldi + c * 8;
  }
}

// requests plane z into ring slot id
template <int KC, int N>
__device__ __forceinline__ void conv3_load_plane(const ConvArgs& a, unsigned ring, int z, unsigned id, int tid,
                                                 const bf16* const (&src)[C3<KC, N>::NJ]) {
  using C = C3<KC, N>;
  const long long off = (long long)wrap(z, a.v.nz) * ((long long)a.v.nx * a.v.ny * a.ldi);
  const unsigned base = ring + (id & (kRing - 1)) * C::PLANE;
#pragma unroll
  for (int j = 0; j < C::NJ; ++j) {
    const int i = tid + j * kWorkers;
    if (i < kCHalo * KC) cp16(base + (unsigned)((i % KC) * C::PV + i / KC) * 16u, src[j] + off);
  }
}

}  // namespace

template <int KC, int N>
__global__ void __launch_bounds__(kConv3Threads, C3<KC, N>::BLOCKS) k_conv3(ConvArgs a, int* err) {
  using C = C3<KC, N>;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bars[6];   // full 0/1, done 0/1, empty 0/1
  __shared__ unsigned tmem_s;
  __shared__ int fail_s;
  __shared__ float bias_s[N];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* const fail = &fail_s;
  const unsigned ring = (unsigned)__cvta_generic_to_shared(smem);
  const unsigned wsm = ring + kRing * C::PLANE;
  const unsigned full = (unsigned)__cvta_generic_to_shared(bars), done = full + 16, empty = full + 32;
  const int ntx = (a.v.nx + kCX - 1) / kCX, nty = (a.v.ny + kCY - 1) / kCY, nz = a.v.nz;
  const long long total = (long long)ntx * nty * nz * a.batch;
  const long long t0 = total * blockIdx.x / gridDim.x, t1 = total * (blockIdx.x + 1) / gridDim.x;
  const int n = (int)(t1 - t0);
  // The parameters, ahead of the wait for the predecessor (they were written before it,
  // see chain_wait): one 32^3 sample 189 -> 160 us, sixteen of 64^3 1982 -> 1916 us.  The
  // first tile's planes right after the wait, before the flag and the allocation, took
  // 153 us at 32^3 but 2253 us for the batch: their addresses spill.
  if (warp != 8 && n > 0) {
    for (int i = tid; i < 27 * N * KC; i += kWorkers) {   // weights (core-matrix layout)
      const int c = i % KC, m = (i / KC) % N, tap = i / (KC * N);
      cp16(wsm + (unsigned)((tap * KC + c) * N + m) * 16u, a.w + ((long long)tap * N + m) * a.cin + c * 8);
    }
    if (tid < N) bias_s[tid] = a.bias != nullptr ? __ldcg(a.bias + tid % a.bias_mod) : 0.f;
    cp_commit();
  }
  chain_wait();
  // the warp's role once more, as a value of its own: with the test above repeated the
  // compiler joins the parts of a role and spills
  const bool issuer = __shfl_sync(0xffffffffu, warp, 0) == 8;
  // a network whose tensor-core wait once expired launches no more tensor-core work:
  // the flag is sticky until the context is destroyed (one thread reads it, so that
  // every thread of the block takes the same branch)
  if (__syncthreads_or(tid == 0 && *(volatile int*)err != 0) || n <= 0) {
    cp_wait<0>();
    return;
  }

  if (warp == 8) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(&tmem_s);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(dst), "r"(2 * C::ACC));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  if (tid == 0) {
    fail_s = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(full + 8 * i, 1);
      mbar_init(done + 8 * i, 1);
      mbar_init(empty + 8 * i, kWorkers / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  tc_before();
  __syncthreads();
  tc_after();

  if (issuer) {
    // ---- MMA issue
    const unsigned tmem = __shfl_sync(0xffffffffu, tmem_s, 0);
    unsigned q = 0;                                    // ring index of the tile's lowest plane
    int z = (int)(t0 % nz);
    for (int k = 0; k < n; ++k) {
      bool ok = mbar_wait(full + 8 * (k & 1), (unsigned)((k >> 1) & 1), fail);
      if (ok && k >= 2) ok = mbar_wait(empty + 8 * (k & 1), (unsigned)(((k >> 1) - 1) & 1), fail);
      if (!ok) {
        if (lane == 0) { *fail = 1; atomicExch(err, 1); }
        break;
      }
      tc_after();
      if (elect_one()) {
        const unsigned d = tmem + (unsigned)((k & 1) * C::ACC);
        const uint64_t bd0 = sdesc(wsm, N * 16, 128);
#pragma unroll
        for (int dz = 0; dz < 3; ++dz) {
          const uint64_t ad0 = sdesc(ring + ((q + dz) & (kRing - 1)) * C::PLANE, C::PV * 16, kCHX * 16);
#pragma unroll
          for (int t9 = 0; t9 < 9; ++t9) {
#pragma unroll
            for (int kk = 0; kk < KC; kk += 2) {
              // later taps and chunks only move the start address (16-byte units; it
              // never carries out of its 14 bits)
              const uint64_t ad = ad0 + (unsigned)((t9 / 3) * kCHX + t9 % 3 + kk * C::PV);
              const uint64_t bd = bd0 + (unsigned)(((dz * 9 + t9) * KC + kk) * N);
              asm volatile(
                  "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                  "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                  "l"(ad), "l"(bd), "r"(idesc_bf16(128, N)), "r"((dz | t9 | kk) ? 1u : 0u));
            }
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                         done + 8u * (unsigned)(k & 1))
                     : "memory");
      }
      __syncwarp();
      if (++z == nz) { z = 0; q += 3; } else { q += 1; }
    }
  } else {
    // ---- plane staging and epilogue
    const long long nvox = (long long)a.v.nx * a.v.ny * nz;
    const bf16* src[C::NJ];                            // this thread's copies in plane 0 of the loading column
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;               // TMEM lane = tile voxel (x = row % 8, y = row / 8)
    const unsigned tmem = tmem_s;

    long long col = t0 / nz;
    int z = (int)(t0 - col * nz);
    asm volatile("" : "+l"(col));
    conv3_sources<KC>(a, col, tid, src);
    unsigned id = 0;                                   // ring index of tile k's lowest plane
    for (int d = 0; d < 3; ++d) conv3_load_plane<KC, N>(a, ring, z - 1 + d, d, tid, src);
    cp_commit();
    if (n > 1 && z + 1 < nz) conv3_load_plane<KC, N>(a, ring, z + 2, 3, tid, src);
    cp_commit();
    cp_wait<1>();
    fence_async();
    bool ok = workers_all(true);
    if (tid == 0) mbar_arrive(full);
    int eb, ex, ey;
    conv3_column(a, col, eb, ex, ey);
    for (int k = 0; k < n; ++k) {
      const bool more = k + 1 < n, newcol = more && z + 1 == nz;
      if (more && !newcol) {                           // tile k + 1's plane, requested one tile ago
        cp_wait<0>();
        fence_async();
        ok = workers_all(ok);
        if (!ok) break;
        if (tid == 0) mbar_arrive(full + 8 * ((k + 1) & 1));
      }
      ok = mbar_wait(done + 8 * (k & 1), (unsigned)((k >> 1) & 1), fail) && ok;
      tc_after();
      const unsigned idn = id + (newcol ? 3u : 1u);
      if (ok) {
        // tile k's lowest plane is free: request what tiles k + 1 and k + 2 still need
        if (newcol) {
          conv3_sources<KC>(a, col + 1, tid, src);
          for (int d = 0; d < 3; ++d) conv3_load_plane<KC, N>(a, ring, d - 1, idn + d, tid, src);
        }
        const int zn = newcol ? 0 : z + 1;
        if (k + 2 < n && zn + 1 < nz) conv3_load_plane<KC, N>(a, ring, zn + 2, idn + 3, tid, src);
        cp_commit();
        // epilogue of tile k
        const int x = ex + row % kCX, y = ey + row / kCX;
        const bool store = x < a.v.nx && y < a.v.ny;
        const long long vox = (long long)eb * nvox + ((long long)z * a.v.ny + y) * a.v.nx + x;
        bf16* orow = (bf16*)a.out + vox * a.ldo + a.offo;
        const bf16* grow = a.gate != nullptr && store ? a.gate + vox * a.ldg + a.offg : nullptr;
#pragma unroll
        for (int c0 = 0; c0 < N; c0 += 32) {           // this warp's 16-column slices
          const int cc = c0 + half * 16;
          if (cc >= N) break;
          unsigned v[16];
          const unsigned taddr = tmem + ((unsigned)(quarter * 32) << 16) + (unsigned)((k & 1) * C::ACC + cc);
          tmem_ld16(v, taddr);
#pragma unroll
          for (int q8 = 0; q8 < 16; q8 += 8) {
            __align__(16) __nv_bfloat162 o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int j = q8 + 2 * u;
              float f0 = __uint_as_float(v[j]), f1 = __uint_as_float(v[j + 1]);
              if (a.bias != nullptr) { f0 += bias_s[cc + j]; f1 += bias_s[cc + j + 1]; }
              if (a.act) {
                f0 = f0 > 0.f ? f0 : kSlope * f0;
                f1 = f1 > 0.f ? f1 : kSlope * f1;
              }
              o[u] = __floats2bfloat162_rn(f0, f1);
            }
            if (grow != nullptr) gate8(o, *reinterpret_cast<const uint4*>(grow + cc + q8));
            if (store) *reinterpret_cast<uint4*>(orow + cc + q8) = *reinterpret_cast<const uint4*>(o);
          }
        }
        tc_before();
      } else {
        if (lane == 0) { *fail = 1; atomicExch(err, 1); }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + 8 * (k & 1));
      if (newcol) {
        cp_wait<0>();
        fence_async();
        ok = workers_all(ok);
        if (!ok) break;
        if (tid == 0) mbar_arrive(full + 8 * ((k + 1) & 1));
        ++col;
        z = 0;
        conv3_column(a, col, eb, ex, ey);
      } else {
        ++z;
      }
      id = idn;
    }
    cp_wait<0>();
  }
  // After an expired wait the MMAs of the last commit may still be in flight when the
  // columns are released below: the contents of this CTA's TMEM columns are then
  // undefined, and so would be a later CTA's accumulator placed in them.  The error
  // flag is set before this point and is sticky, so no later tensor-core launch of
  // this network runs and bfcs_net_status reports BFCS_ERR_TIMEOUT from then on.
  tc_before();
  __syncthreads();
  tc_after();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_s), "r"(2 * C::ACC));
}

// The layer shapes of the network: (input channels / 8, output channels).  The
// padded input layer, the 32- and 48-channel layers, the layers on concatenated
// inputs, and the data gradients of each.
#define BFCS_CONV3_SHAPES(X) X(2, 32) X(4, 32) X(4, 48) X(6, 32) X(6, 48) X(8, 32) X(4, 64)

bool conv3_ok(const ConvArgs& a) {
  if (a.ksize != 3 || a.in_mode != IN_CONV || a.out_mode != OUT_BF16) return false;
  if (a.ldi % 8 != 0 || a.offi % 8 != 0 || a.ldo % 8 != 0 || a.offo % 8 != 0) return false;
#define BFCS_X(KC, N) if (a.cin == 8 * KC && a.cout_p == N) return true;
  BFCS_CONV3_SHAPES(BFCS_X)
#undef BFCS_X
  return false;
}

cudaError_t conv3_init() {
#define BFCS_X(KC, N)                                                                                          \
  {                                                                                                            \
    const cudaError_t e = cudaFuncSetAttribute(k_conv3<KC, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,    \
                                               (int)C3<KC, N>::SMEM);                                          \
    if (e != cudaSuccess) return e;                                                                            \
  }
  BFCS_CONV3_SHAPES(BFCS_X)
#undef BFCS_X
  return cudaSuccess;
}

cudaError_t launch_conv3(const ConvArgs& a, int sms, int* err, cudaStream_t st) {
  const long long tiles = (long long)((a.v.nx + kCX - 1) / kCX) * ((a.v.ny + kCY - 1) / kCY) * a.v.nz * a.batch;
#define BFCS_X(KC, N)                                                                                          \
  if (a.cin == 8 * KC && a.cout_p == N) {                                                                      \
    const int blocks = (int)std::min<long long>(tiles, (long long)sms * C3<KC, N>::BLOCKS);                    \
    launch_chain(true, k_conv3<KC, N>, blocks, kConv3Threads, C3<KC, N>::SMEM, st, a, err);                    \
    count_launches(1);                                                                                         \
    return cudaGetLastError();                                                                                 \
  }
  BFCS_CONV3_SHAPES(BFCS_X)
#undef BFCS_X
  return cudaErrorInvalidValue;
}

}  // namespace net
}  // namespace bfcs
