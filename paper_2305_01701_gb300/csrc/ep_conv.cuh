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

// Where a tensor-core convolution's output goes (any of them may be null).
// Blocked tensors are BF16 [n][channel / 8][z][y][x][8].
struct TcOut {
  int relu;
  float *f32;                    // N x cout x V; with a head, its N x head_c x V output
  __nv_bfloat16 *b16;            // the output in blocks b16_off .. of a tensor of b16_ch blocks
  int b16_ch, b16_off;
  __nv_bfloat16 *pool;           // its 2^D average
  __nv_bfloat16 *up;             // its nearest upsample, the first blocks of a tensor of up_ch blocks
  int up_ch;
  const __nv_bfloat16 *head_w;   // the 1^D head on the FP32 output: head_c x cout, times scale
  const float *head_b;
  int head_c;
  float scale;
};
// shared-memory limits of the kernels, per device (at every network's creation)
cudaError_t conv_tc_configure();
bool conv_tc_supported(int k, int cout);
__host__ __device__ constexpr int conv_tc_cinp(int cin) { return (cin + 15) / 16 * 16; }
// FP32 N x C x V -> blocks of conv_tc_cinp(C) channels
void conv_tc_to_blocks(const float *x, int N, int C, long long nv, __nv_bfloat16 *out, cudaStream_t st);
cudaError_t conv_tc_forward(int D, const __nv_bfloat16 *xb, int N, int X, int Y, int Z, int cin,
                            const __nv_bfloat16 *wpk, const float *bias, int cout, const TcOut &out, int *err,
                            cudaStream_t st);

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
