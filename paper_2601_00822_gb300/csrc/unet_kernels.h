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

enum InMode : int { IN_CONV = 0, IN_GATHER_UP = 1 };
enum OutMode : int { OUT_BF16 = 0, OUT_SHUFFLE_UP = 1, OUT_F32 = 2 };

struct ConvArgs {
  const bf16* in;     // channels-last input: element (voxel, k) at in[voxel * ldi + offi + k]
  int ldi, offi;
  int cin;            // GEMM K per tap (multiple of 16)
  const bf16* w;      // [tap][cout_p][cin], K fastest
  const float* bias;  // bias[col % bias_mod], or null
  int bias_mod;
  int cout_p;         // GEMM columns (multiple of 8)
  int cout;           // columns stored (OUT_F32)
  int ksize;          // 1 or 3 (circular)
  Vol v;              // grid of the GEMM rows (coarse grid for the gather / shuffle modes)
  int batch;
  int act;            // 1: leaky ReLU
  int in_mode, out_mode;
  void* out;          // channels-last output, element (voxel, col) at out[voxel * ldo + offo + col]
  int ldo, offo;
  int up_c;           // gather / shuffle: channels per sub-voxel (multiple of 16)
};

// 3^3 circular convolution on the tensor cores (unet_conv.cu); conv3_ok: the layer
// shapes it is compiled for.  err is set by an expired wait.
bool conv3_ok(const ConvArgs& a);
cudaError_t conv3_init();   // once per network context: shared-memory limits
cudaError_t launch_conv3(const ConvArgs& a, int sms, int* err, cudaStream_t st);

}  // namespace net
}  // namespace bfcs
