// Interfaces shared by the network's translation units (internal).
#pragma once
#include "kernels.h"

#include <cuda_bf16.h>

namespace bfcs {
namespace net {

typedef __nv_bfloat16 bf16;

constexpr float kSlope = 0.1f;

struct Vol { int nx, ny, nz; };

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

// c += a b of one warp (m16n8k16, BF16 operands, FP32 accumulators)
__device__ __forceinline__ void mma16816(float* c, const unsigned* a, unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// four transposed 8 x 8 matrices from the rows at the lanes' shared-memory addresses
__device__ __forceinline__ void ldsm_x4_trans(unsigned* r, unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

enum InMode : int { IN_CONV = 0, IN_GATHER_UP = 1 };
enum OutMode : int { OUT_BF16 = 0, OUT_SHUFFLE_UP = 1 };

struct ConvArgs {
  const bf16* in;     // channels-last input: element (voxel, k) at in[voxel * ldi + offi + k]
  int ldi, offi;
  int cin;            // GEMM K per tap (multiple of 16)
  const bf16* w;      // [tap][cout_p][cin], K fastest
  const float* bias;  // bias[col % bias_mod], or null
  int bias_mod;
  int cout_p;         // GEMM columns (multiple of 8)
  int ksize;          // 1 or 3 (circular)
  Vol v;              // grid of the GEMM rows (coarse grid for the gather / shuffle modes)
  int batch;
  int act;            // 1: leaky ReLU
  int in_mode, out_mode;
  void* out;          // channels-last output, element (voxel, col) at out[voxel * ldo + offo + col]
  int ldo, offo;
  int up_c;           // gather / shuffle: channels per sub-voxel (multiple of 16)
  // data gradients: the activation's derivative at the layer below, from the sign of its
  // saved output (voxel, col) at gate[voxel * ldg + offg + col]; null: none
  const bf16* gate;
  int ldg, offg;
};

// 8 values times act'(y) of the 8 saved outputs in y: the BF16 values are scaled and
// rounded again, as a pass of its own over them would
__device__ __forceinline__ void gate8(__nv_bfloat162* o, uint4 y) {
  const bf16* y8 = reinterpret_cast<const bf16*>(&y);
  bf16* o8 = reinterpret_cast<bf16*>(o);
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (!(__bfloat162float(y8[k]) > 0.f)) o8[k] = __float2bfloat16(__bfloat162float(o8[k]) * kSlope);
}

// Whether r, a product of float-float arithmetic, rounds to FP32 (r.hi) as the product in
// FP64 does: true unless the value lies within 2^-43 of a boundary between two floats.
// The two products differ by less than 2^-44 (a factor cut to 47 bits, two roundings of
// 2^-47 and the product of the low parts; the FP64 form rounds at 2^-53), so the few
// values that fail (2^-18 of them) are formed in FP64 and every result is that of FP64.
__device__ __forceinline__ bool ff_rounds_as_fp64(ff r) {
  const float w = fabsf(r.hi) * 1.1368683772161603e-13f;   // 2^-43
  return __fadd_rn(r.hi, __fadd_rn(r.lo, w)) == r.hi && __fadd_rn(r.hi, __fsub_rn(r.lo, w)) == r.hi;
}

constexpr int kSampleArgs = 64;      // samples whose pointers travel in one launch's arguments

template <typename R> struct HeadArgs {
  const bf16* in;                    // [sample][n][32]
  const bf16* w;                     // [16][32], rows 6.. zero
  const float* bias;                 // 6
  long long n;                       // voxels of a sample
  const unsigned* sbits;             // prediction: per-sample max |b| (bits of a float)
  float mu_max;
  R* out[kSampleArgs];               // 6 x n each
};

// 3^3 circular convolution on the tensor cores (unet_conv.cu); conv3_ok: the layer
// shapes it is compiled for.  err is set by an expired wait.
bool conv3_ok(const ConvArgs& a);
cudaError_t conv3_init();   // once per network context: shared-memory limits
cudaError_t launch_conv3(const ConvArgs& a, int sms, int* err, cudaStream_t st);

// weight gradients (see k_wgrad in unet.cu): partial[chunk][tap][cout_p][cin] in FP32
struct WgArgs {
  const bf16* dy; int ldd, offd;   // output gradient (pre-activation)
  const bf16* x; int ldx, offx;    // layer input
  int cin, cout_p;                 // multiples of 16; cin <= 128; cout_p <= 64 or a multiple of 64
  int ksize;
  Vol v;                           // grid of the GEMM K index (coarse grid for the up mode)
  int batch;
  int up_c;
  long long chunk;                 // voxels per block (multiple of 64)
  float* part;
  float* bpart;                    // bias gradient partials of the fused forms: [block][channels]
};
// tcgen05 form of the 3^3 layers with 32 output channels (unet_wgrad.cu): wgrad3_chunks
// partials, one per block
bool wgrad3_ok(const WgArgs& a);
cudaError_t wgrad3_init();
int wgrad3_chunks(const WgArgs& a, int sms);
cudaError_t launch_wgrad3(const WgArgs& a, int chunks, int* err, cudaStream_t st);

// the up-convolutions and the head
bool wgrad1_ok(const WgArgs& a);
cudaError_t wgrad1_init();
int wgrad1_chunks(const WgArgs& a, int sms);
cudaError_t launch_wgrad1(const WgArgs& a, int sms, cudaStream_t st);

// pointwise GEMMs (unet_gemm.cu): up-convolutions, their data gradients, the head's
// data gradient; rows_ok: the layer shapes they are compiled for
bool rows_ok(const ConvArgs& a);
cudaError_t launch_rows(const ConvArgs& a, int sms, cudaStream_t st);
// the head for up to kSampleArgs samples
template <typename R>
cudaError_t launch_head(const HeadArgs<R>& a, int batch, bool predict, int sms, cudaStream_t st);

}  // namespace net
}  // namespace bfcs
