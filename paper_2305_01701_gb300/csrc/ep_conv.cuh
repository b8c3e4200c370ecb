// ep_conv.cuh -- the warm-start network's convolutions: training in FP32
// (ep_conv_fp32.cu), inference on the tensor cores (ep_conv_tc.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace ep {

struct ConvArgs32 {
  const float *x;             // N x cin x [Z x] Y x X
  const float *w;             // the layer's packed weights in this direction (conv32_pack)
  const float *b;             // cout (nullable)
  float *y;                   // N x cout x [Z x] Y x X
  const float *mask;          // nullable, the shape of y: y is 0 where it is <= 0
  int N, cin, cout, X, Y, Z, relu;
};
struct WgradArgs {
  const float *x, *dy;        // N x cin x ..., N x cout x ...
  float *partial;             // conv32_wgrad_floats
  int N, cin, cout, X, Y, Z, nq;
};

// the layers whose weights are packed for the tensor cores (ep_conv_tc.cu), as
// one launch's arguments
struct PackTable {
  int n, taps;
  int cin[24], cout[24];
  long long src[24], dst[24];   // offsets of a layer's weights and of their packed copy
  long long total;              // packed elements of all layers
};
void conv_tc_pack_weights(const PackTable &P, const __nv_bfloat16 *w, __nv_bfloat16 *out, cudaStream_t st);

cudaError_t conv32_configure();
// FP32 copies of the 3^D layers' weights in the order the kernels read them, for
// the forward pass and for the data gradient
struct Pack32 {
  int n, taps;
  int cin[24], cout[24];
  long long src[24], fwd[24], bwd[24];   // offsets of the weights and of their packed copies
};
__host__ __device__ constexpr int conv32_cinp(int cin) { return (cin + 7) / 8 * 8; }
long long conv32_packed(int D, int cin, int cout);   // floats of one direction
void conv32_pack(const Pack32 &P, const __nv_bfloat16 *w, float *out, cudaStream_t st);
// 3^D convolution with zero padding, forward or data gradient
void conv32(int D, const ConvArgs32 &A, cudaStream_t st);
// weight and bias gradient of a k^D convolution (k = 1 or 3): overwrites dw, db
long long conv32_wgrad_floats(int D, int k, int N, int X, int Y, int Z, int cin, int cout);
void conv32_wgrad(int D, int k, WgradArgs A, float *dw, float *db, cudaStream_t st);

}  // namespace ep
