// ep_conv_fp32.cu -- the warm-start network's 3^D convolutions in FP32 on the
// CUDA cores: forward and data gradient (k_conv_tile) and weight gradient
// (k_conv_wgrad_tile), for training.
//
// FP32 activations and gradients, BF16 weights, FP32 sums.  The tensor cores
// are left out here on purpose: their FP32 accumulation loses more than an FP32
// FMA chain does (measured on 2592-term sums split into BF16 parts: 1.9e-6 to
// 4.4e-6 relative, against 6.5e-7), and training keeps FP32's accuracy.
//
// Bound: FP32 FMA issue.  Both kernels work on register tiles fed from shared
// memory, with the FMAs packed two to an instruction (FFMA2 on float2).
//   k_conv_tile: a block of 128 threads computes 512 voxels x 16 output
//   channels; a thread 4 voxels along x times 16 channels (8 pairs).  Per input
//   channel and row of taps it reads 6 inputs (2 loads) and 12 broadcast vectors
//   of weights for 96 packed FMAs.  Input channels come 4 at a time, copied
//   with cp.async (zero fill is the padding) while the previous 4 are used.
//   k_conv_wgrad_tile: a block of 256 threads holds, in registers, the gradients
//   of up to 32 x 32 (output, input) channels and all taps -- a lane one input
//   channel, a warp four output channels -- and walks over tiles of voxels; the
//   voxel tiles are split over enough blocks to fill the chip.  Each block
//   writes its partial sums, and k_wgrad_sum adds them in a fixed order (the
//   gradient is the same bit for bit on every call).
// Measured on the 64^3 network (base 32, two samples): forward and backward
// 18.85 ms against 223 ms with one thread per voxel (or weight) reading global
// memory (58 - 60 % of the issue slots, the FMA pipe's throttle the first stall); the 32 -> 32 convolution of 524,288 voxels 0.69 ms = 42 TFLOP/s, its
// weight gradient 0.72 ms.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "ep_conv.cuh"

namespace ep {

namespace {

__device__ __forceinline__ unsigned su32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
// 4-byte asynchronous copy; zero when !ok
__device__ __forceinline__ void cp4(float *dst, const float *src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(su32(dst)), "l"(src), "r"(ok ? 4 : 0));
}
__device__ __forceinline__ void cp16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(su32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int n>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(n));
}

// ---- forward and data gradient --------------------------------------------
constexpr int CO = 16;   // output channels per block
constexpr int CT = 128;  // threads
constexpr int TX = 16;   // voxels along x
constexpr int PX = 20;   // pitch of a row of TX + 2 inputs

// KS = 1: 512 voxels per block, every thread sums over all input channels.
// KS = 4: 128 voxels per block; each warp takes every fourth input channel and
// the four partial sums are added at the end.
template <int D, int KS>
struct Tile {
  static constexpr int CK = KS == 1 ? 4 : 8;   // input channels per stage
  static constexpr int TY = D == 3 ? (KS == 1 ? 8 : 4) : (KS == 1 ? 32 : 8);
  static constexpr int TZ = D == 3 ? (KS == 1 ? 4 : 2) : 1;
  static constexpr int RY = TY + 2, RZ = D == 3 ? TZ + 2 : 1;   // rows with the halo
  static constexpr int TAPS = D == 3 ? 27 : 9;
  static constexpr int ROWS = CK * RZ * RY;
  static constexpr int WN = CK * TAPS * CO;   // weights per stage
  static constexpr size_t stages = 2 * (size_t)(ROWS * PX + WN) * sizeof(float);
  static constexpr size_t sums = KS == 1 ? 0 : (size_t)CT * CO * 4 * sizeof(float);
  static constexpr size_t bytes = stages > sums ? stages : sums;
};

// y[n, co, v] = b[co] + sum over ci, tap of W(co, ci, tap) x[n, ci, v + tap - 1]
// The data gradient is the same with the weights packed the other way round
// (channels swapped, taps mirrored) and no bias.  relu: max(y, 0).  mask (nullable): y is 0 where mask[n, co, v] <= 0 (the
// ReLU of the layer that produced the tensor whose gradient y is).
template <int D, int KS>
__global__ void __launch_bounds__(CT, 3) k_conv_tile(const ConvArgs32 A) {
  using L = Tile<D, KS>;
  constexpr int CK = L::CK;
  extern __shared__ __align__(16) float sm[];
  auto xs = [&](int k) { return sm + k * (L::ROWS * PX); };
  auto ws = [&](int k) { return sm + 2 * L::ROWS * PX + k * L::WN; };
  const int tid = threadIdx.x;
  const int vt = tid % (CT / KS), kpart = tid / (CT / KS);
  const int tx = vt & 3, ty = (vt >> 2) % L::TY, tz = (vt >> 2) / L::TY;
  const int X = A.X, Y = A.Y, Z = A.Z, cin = A.cin, cout = A.cout;
  const int nbx = (X + TX - 1) / TX, nby = (Y + L::TY - 1) / L::TY;
  const int x0 = (blockIdx.x % nbx) * TX, y0 = (blockIdx.x / nbx % nby) * L::TY, z0 = blockIdx.x / (nbx * nby) * L::TZ;
  const int co0 = blockIdx.y * CO, n = blockIdx.z;
  const long long nvox = (long long)X * Y * Z;
  const float *xn = A.x + (long long)n * cin * nvox;

  auto fetch_x = [&](int c0, float *dst) {
    for (int e = tid; e < L::ROWS * (TX + 2); e += CT) {
      const int row = e / (TX + 2), xx = e - row * (TX + 2);
      const int c = row / (L::RZ * L::RY), rz = row / L::RY % L::RZ, ry = row % L::RY;
      const int gx = x0 + xx - 1, gy = y0 + ry - 1, gz = D == 3 ? z0 + rz - 1 : 0;
      const bool ok = c0 + c < cin && gx >= 0 && gx < X && gy >= 0 && gy < Y && gz >= 0 && gz < Z;
      cp4(dst + row * PX + xx, ok ? xn + (long long)(c0 + c) * nvox + ((long long)gz * Y + gy) * X + gx : xn, ok);
    }
  };
  // a stage's weights are one run of the packed array: [ci][tap][16 co]
  const float *wn = A.w + (long long)blockIdx.y * conv32_cinp(cin) * L::TAPS * CO;
  auto fetch_w = [&](int c0, float *dst) {
    const float *src = wn + (long long)c0 * L::TAPS * CO;
    for (int e = tid; e < L::WN / 4; e += CT) cp16(dst + 4 * e, src + 4 * e);
  };

  float2 acc[CO / 2][4];
#pragma unroll
  for (int p = 0; p < CO / 2; ++p) {
    const int c = co0 + 2 * p;
    const float2 b = make_float2(A.b && kpart == 0 && c < cout ? A.b[c] : 0.f,
                                 A.b && kpart == 0 && c + 1 < cout ? A.b[c + 1] : 0.f);
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[p][v] = b;
  }

  fetch_x(0, xs(0));
  fetch_w(0, ws(0));
  cp_commit();
  const int stages = (cin + CK - 1) / CK;
  for (int s = 0; s < stages; ++s) {
    const int cur = s & 1;
    cp_wait<0>();
    __syncthreads();   // stage s has arrived, stage s - 1 is no longer read
    if (s + 1 < stages) {
      fetch_x((s + 1) * CK, xs(cur ^ 1));
      fetch_w((s + 1) * CK, ws(cur ^ 1));
    }
    cp_commit();
    const float *xb = xs(cur) + (tz * L::RY + ty) * PX + 4 * tx, *wb = ws(cur);
    for (int c = kpart; c < CK; c += KS) {
#pragma unroll
      for (int dz = 0; dz < (D == 3 ? 3 : 1); ++dz)
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          const float *xr = xb + ((c * L::RZ + dz) * L::RY + dy) * PX;
          const float4 xa = *reinterpret_cast<const float4 *>(xr);
          const float2 xc = *reinterpret_cast<const float2 *>(xr + 4);
          const float xv[6] = {xa.x, xa.y, xa.z, xa.w, xc.x, xc.y};
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {
            const float4 *wp = reinterpret_cast<const float4 *>(wb + (c * L::TAPS + (dz * 3 + dy) * 3 + dx) * CO);
#pragma unroll
            for (int q = 0; q < CO / 4; ++q) {
              const float4 w4 = wp[q];
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                const float2 xx = make_float2(xv[v + dx], xv[v + dx]);
                acc[2 * q][v] = __ffma2_rn(make_float2(w4.x, w4.y), xx, acc[2 * q][v]);
                acc[2 * q + 1][v] = __ffma2_rn(make_float2(w4.z, w4.w), xx, acc[2 * q + 1][v]);
              }
            }
          }
        }
    }
  }

  // KS = 4: every warp's sums to shared memory, [part][channel, voxel][thread];
  // warp k then adds and writes channels 4k .. 4k + 3
  constexpr int CW = CO / KS;   // channels this thread writes
  const int cw0 = KS == 1 ? 0 : kpart * CW;
  float out[KS == 1 ? 1 : CW][4];
  if constexpr (KS > 1) {
    __syncthreads();   // the last stage is no longer read
#pragma unroll
    for (int c = 0; c < CO; ++c)
#pragma unroll
      for (int v = 0; v < 4; ++v)
        sm[((kpart * CO + c) * 4 + v) * 32 + vt] = (c & 1) ? acc[c / 2][v].y : acc[c / 2][v].x;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < CW; ++c)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float r = sm[((cw0 + c) * 4 + v) * 32 + vt];
#pragma unroll
        for (int k = 1; k < KS; ++k) r += sm[((k * CO + cw0 + c) * 4 + v) * 32 + vt];
        out[c][v] = r;
      }
  }

  const int ox = x0 + 4 * tx, oy = y0 + ty, oz = z0 + tz;
  if (ox >= X || oy >= Y || oz >= Z) return;
  const long long v0 = ((long long)oz * Y + oy) * X + ox;
  const bool vec = (X & 3) == 0;   // then v0 and every channel's offset are multiples of 4
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    const int co = co0 + cw0 + c;
    if (co >= cout) break;
    const long long o = ((long long)n * cout + co) * nvox + v0;
    float r[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      if constexpr (KS == 1) r[v] = (c & 1) ? acc[c / 2][v].y : acc[c / 2][v].x;
      else r[v] = out[c][v];
      if (A.relu && r[v] < 0.f) r[v] = 0.f;
    }
    if (vec) {
      if (A.mask) {
        const float4 m = *reinterpret_cast<const float4 *>(A.mask + o);
        r[0] = m.x <= 0.f ? 0.f : r[0]; r[1] = m.y <= 0.f ? 0.f : r[1];
        r[2] = m.z <= 0.f ? 0.f : r[2]; r[3] = m.w <= 0.f ? 0.f : r[3];
      }
      *reinterpret_cast<float4 *>(A.y + o) = make_float4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
      for (int v = 0; v < 4; ++v)
        if (ox + v < X) A.y[o + v] = A.mask && A.mask[o + v] <= 0.f ? 0.f : r[v];
    }
  }
}

// ---- weight gradient --------------------------------------------------------
constexpr int GT = 256;   // threads: 8 warps
constexpr int GC = 32;    // channels of either kind per block
constexpr int GPX = 33;   // pitch of an input voxel's channels
constexpr int GPY = 36;   // pitch of a gradient voxel's channels

template <int D, int K>
struct GTile {
  static constexpr int TY = 4, TZ = D == 3 ? 2 : 1, R = K / 2;
  static constexpr int HX = TX + 2 * R, HY = TY + 2 * R, HZ = D == 3 ? TZ + 2 * R : 1;
  static constexpr int TAPS = D == 3 ? K * K * K : K * K;
  static constexpr int VOX = TX * TY * TZ, HALO = HX * HY * HZ;
  static constexpr int STAGE = HALO * GPX + VOX * GPY;
  static constexpr size_t bytes = 2 * (size_t)STAGE * sizeof(float);
};

// partial sums of dW[co][ci][tap] = sum over n, v of dy[n, co, v] x[n, ci, v + tap - r]
// and of db[co] = sum of dy.  blockIdx.x: split of the voxel tiles; .y, .z:
// blocks of output / input channels.  A block's warps hold nq quads of output
// channels, and 8 / nq of them share a quad and take every (8 / nq)-th run of 4
// voxels each (a partial sum of its own).
template <int D, int K>
__global__ void __launch_bounds__(GT, 1) k_conv_wgrad_tile(const WgradArgs A) {
  using L = GTile<D, K>;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int X = A.X, Y = A.Y, Z = A.Z, cin = A.cin, cout = A.cout;
  const int co0 = blockIdx.y * GC, ci0 = blockIdx.z * GC;
  const int nci = min(GC, cin - ci0), nco = min(GC, cout - co0);
  const int q = warp % A.nq, part = warp / A.nq, parts = 8 / A.nq;
  const int nbx = (X + TX - 1) / TX, nby = (Y + L::TY - 1) / L::TY, nbz = (Z + L::TZ - 1) / L::TZ;
  const long long nvox = (long long)X * Y * Z, tiles = (long long)A.N * nbx * nby * nbz;

  auto fetch = [&](long long t, float *st) {
    const int bx = (int)(t % nbx), by = (int)(t / nbx % nby), bz = (int)(t / ((long long)nbx * nby) % nbz);
    const int n = (int)(t / ((long long)nbx * nby * nbz));
    const int x0 = bx * TX - L::R, y0 = by * L::TY - L::R, z0 = D == 3 ? bz * L::TZ - L::R : 0;
    const float *xn = A.x + ((long long)n * cin + ci0) * nvox, *gn = A.dy + ((long long)n * cout + co0) * nvox;
    for (int e = tid; e < L::HALO * nci; e += GT) {   // x fastest, then rows, then channels
      const int c = e / L::HALO, r = e - c * L::HALO;
      const int hx = r % L::HX, hy = r / L::HX % L::HY, hz = r / (L::HX * L::HY);
      const int gx = x0 + hx, gy = y0 + hy, gz = z0 + hz;
      const bool ok = gx >= 0 && gx < X && gy >= 0 && gy < Y && gz >= 0 && gz < Z;
      cp4(st + r * GPX + c, ok ? xn + c * nvox + ((long long)gz * Y + gy) * X + gx : xn, ok);
    }
    float *sy = st + L::HALO * GPX;
    for (int e = tid; e < L::VOX * nco; e += GT) {
      const int c = e / L::VOX, r = e - c * L::VOX;
      const int gx = bx * TX + r % TX, gy = by * L::TY + r / TX % L::TY, gz = bz * L::TZ + r / (TX * L::TY);
      const bool ok = gx < X && gy < Y && gz < Z;
      cp4(sy + r * GPY + c, ok ? gn + c * nvox + ((long long)gz * Y + gy) * X + gx : gn, ok);
    }
  };

  // columns of channels beyond the last stay zero
  for (int e = tid; e < 2 * L::STAGE; e += GT) sm[e] = 0.f;
  __syncthreads();
  auto st = [&](int k) { return sm + k * L::STAGE; };

  float2 acc[L::TAPS][2], accb[2];
#pragma unroll
  for (int t = 0; t < L::TAPS; ++t) acc[t][0] = acc[t][1] = make_float2(0.f, 0.f);
  accb[0] = accb[1] = make_float2(0.f, 0.f);

  long long t = blockIdx.x;
  if (t < tiles) fetch(t, st(0));
  cp_commit();
  for (int it = 0; t < tiles; t += gridDim.x, ++it) {
    cp_wait<0>();
    __syncthreads();   // this tile has arrived, the previous one is no longer read
    if (t + gridDim.x < tiles) fetch(t + gridDim.x, st((it & 1) ^ 1));
    cp_commit();
    const float *xs = st(it & 1), *ys = xs + L::HALO * GPX;
    for (int r = part; r < L::VOX / 4; r += parts) {   // runs of 4 voxels along x
      const int vx = (r % (TX / 4)) * 4, vy = r / (TX / 4) % L::TY, vz = r / (TX / 4 * L::TY);
      float2 g[4][2];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const float4 f = *reinterpret_cast<const float4 *>(ys + (r * 4 + v) * GPY + 4 * q);
        g[v][0] = make_float2(f.x, f.y);
        g[v][1] = make_float2(f.z, f.w);
        accb[0] = __fadd2_rn(accb[0], g[v][0]);
        accb[1] = __fadd2_rn(accb[1], g[v][1]);
      }
#pragma unroll
      for (int dz = 0; dz < (D == 3 ? K : 1); ++dz)
#pragma unroll
        for (int dy = 0; dy < K; ++dy) {
          const float *xr = xs + (((vz + dz) * L::HY + vy + dy) * L::HX + vx) * GPX + lane;
#pragma unroll
          for (int h = 0; h < 4 + K - 1; ++h) {
            const float xv = xr[h * GPX];
            const float2 xx = make_float2(xv, xv);
#pragma unroll
            for (int dx = 0; dx < K; ++dx) {
              const int v = h - dx;
              if (v < 0 || v > 3) continue;
              const int tap = (dz * K + dy) * K + dx;
              acc[tap][0] = __ffma2_rn(g[v][0], xx, acc[tap][0]);
              acc[tap][1] = __ffma2_rn(g[v][1], xx, acc[tap][1]);
            }
          }
        }
    }
  }
  // partial sums: [split][co][ci][tap], then the biases' [split][co]
  const long long slot = (long long)blockIdx.x * parts + part;
  const long long per = (long long)cout * cin * L::TAPS;
  float *pw = A.partial + slot * (per + cout);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int co = co0 + 4 * q + c;
    if (co >= cout) break;
    if (lane < nci) {
      float *d = pw + ((long long)co * cin + ci0 + lane) * L::TAPS;
#pragma unroll
      for (int k = 0; k < L::TAPS; ++k) d[k] = (c & 1) ? acc[k][c / 2].y : acc[k][c / 2].x;
    }
    if (ci0 == 0 && lane == 0) pw[per + co] = (c & 1) ? accb[c / 2].y : accb[c / 2].x;
  }
}

// s + c += x, the rounding of s + x kept in c (Knuth's two-sum)
__device__ __forceinline__ void add_exact(float &s, float &c, float x) {
  const float t = s + x, b = t - s;
  c += (s - (t - b)) + (x - b);
  s = t;
}

// dw = sum of the partial sums, db likewise: 8 threads per element add every
// eighth split each, then their sums are added, in a fixed order.  Up to 150
// partial sums come one after the other here: plain additions made the last
// layers' gradients up to 1.5 times as far from 64 bits as a tree over all
// threads does; with their roundings kept every layer's is 0.5 to 0.8 times as
// far (a training step of the 48 x 48 network 612 -> 620 us, of 64^3 no change).
__global__ void __launch_bounds__(256) k_wgrad_sum(const float *partial, int slots, long long per, int cout, float *dw,
                                                   float *db) {
  __shared__ float sh[8][32], ch[8][32];
  const int e = threadIdx.x & 31, j = threadIdx.x >> 5;
  const long long i = (long long)blockIdx.x * 32 + e, stride = per + cout;
  float s = 0.f, c = 0.f;
  if (i < stride)
    for (int q = j; q < slots; q += 8) add_exact(s, c, partial[q * stride + i]);
  sh[j][e] = s;
  ch[j][e] = c;
  __syncthreads();
  if (j != 0 || i >= stride) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) {
    add_exact(s, c, sh[q][e]);
    c += ch[q][e];
  }
  if (fabsf(s) < INFINITY) s += c;   // an infinite sum's rounding is no number
  if (i < per) dw[i] = s;
  else db[i - per] = s;
}

template <int D, int K>
void wgrad_launch(const WgradArgs &A, int slots_x, cudaStream_t st) {
  dim3 grid(slots_x, (A.cout + GC - 1) / GC, (A.cin + GC - 1) / GC);
  k_conv_wgrad_tile<D, K><<<grid, GT, GTile<D, K>::bytes, st>>>(A);
}

// quads of output channels that a block's warps hold: 1, 2, 4 or 8
int wgrad_quads(int cout) {
  const int q = (std::min(cout, GC) + 3) / 4;
  return q <= 1 ? 1 : q <= 2 ? 2 : q <= 4 ? 4 : 8;
}

// splits of the voxel tiles: enough blocks for two per SM (152 SMs), no more
// than there are tiles
int wgrad_splits(int D, int N, int X, int Y, int Z, int cin, int cout) {
  const int ty = 4, tz = D == 3 ? 2 : 1;
  const long long tiles = (long long)N * ((X + TX - 1) / TX) * ((Y + ty - 1) / ty) * ((Z + tz - 1) / tz);
  const int blocks = ((cout + GC - 1) / GC) * ((cin + GC - 1) / GC);
  return (int)std::max(1ll, std::min<long long>(tiles, 304 / blocks));
}

}  // namespace

// fewest blocks of the 512-voxel tiling that it is used for; below, the chip is
// filled better by the 128-voxel blocks that split the input channels
constexpr long long KS_BLOCKS = 400;

cudaError_t conv32_configure() {
  cudaError_t e = cudaSuccess;
#define EP_CFG(k, b) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(b));
  EP_CFG((k_conv_tile<2, 1>), (Tile<2, 1>::bytes)) EP_CFG((k_conv_tile<3, 1>), (Tile<3, 1>::bytes))
  EP_CFG((k_conv_tile<2, 4>), (Tile<2, 4>::bytes)) EP_CFG((k_conv_tile<3, 4>), (Tile<3, 4>::bytes))
  EP_CFG((k_conv_wgrad_tile<2, 1>), (GTile<2, 1>::bytes)) EP_CFG((k_conv_wgrad_tile<2, 3>), (GTile<2, 3>::bytes))
  EP_CFG((k_conv_wgrad_tile<3, 1>), (GTile<3, 1>::bytes)) EP_CFG((k_conv_wgrad_tile<3, 3>), (GTile<3, 3>::bytes))
#undef EP_CFG
  return e;
}

namespace {

template <int D, int KS>
dim3 conv_grid(const ConvArgs32 &A) {
  using L = Tile<D, KS>;
  return dim3(((A.X + TX - 1) / TX) * ((A.Y + L::TY - 1) / L::TY) * ((A.Z + L::TZ - 1) / L::TZ), (A.cout + CO - 1) / CO,
              A.N);
}

template <int D>
void conv_launch(const ConvArgs32 &A, cudaStream_t st) {
  const dim3 g = conv_grid<D, 1>(A);
  if ((long long)g.x * g.y * g.z >= KS_BLOCKS) k_conv_tile<D, 1><<<g, CT, Tile<D, 1>::bytes, st>>>(A);
  else k_conv_tile<D, 4><<<conv_grid<D, 4>(A), CT, Tile<D, 4>::bytes, st>>>(A);
}

// BF16 cout x cin x taps -> FP32 [block of 16 output channels][ci][tap][16],
// forward (even blockIdx.y) and transposed (odd); channels beyond the last are
// zero, input channels are padded to a multiple of 8
__global__ void k_pack32(const Pack32 P, const __nv_bfloat16 *w, float *out) {
  const int l = blockIdx.y >> 1, tr = blockIdx.y & 1, taps = P.taps;
  const int cin = tr ? P.cout[l] : P.cin[l], cout = tr ? P.cin[l] : P.cout[l], cinp = conv32_cinp(cin);
  const int total = (cout + CO - 1) / CO * cinp * taps * CO;
  float *dst = out + (tr ? P.bwd[l] : P.fwd[l]);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int tap = i / CO % taps, ci = i / (CO * taps) % cinp, co = i / (CO * taps * cinp) * CO + i % CO;
    float v = 0.f;
    if (ci < cin && co < cout)
      v = __bfloat162float(w[P.src[l] + (tr ? ((long long)ci * cout + co) * taps + taps - 1 - tap
                                            : ((long long)co * cin + ci) * taps + tap)]);
    dst[i] = v;
  }
}

}  // namespace

long long conv32_packed(int D, int cin, int cout) {
  return (long long)((cout + CO - 1) / CO) * conv32_cinp(cin) * (D == 3 ? 27 : 9) * CO;
}

void conv32_pack(const Pack32 &P, const __nv_bfloat16 *w, float *out, cudaStream_t st) {
  k_pack32<<<dim3(96, 2 * P.n), 256, 0, st>>>(P, w, out);
}

void conv32(int D, const ConvArgs32 &A, cudaStream_t st) {
  if (D == 3) conv_launch<3>(A, st);
  else conv_launch<2>(A, st);
}

long long conv32_wgrad_floats(int D, int k, int N, int X, int Y, int Z, int cin, int cout) {
  const long long taps = D == 3 ? (long long)k * k * k : (long long)k * k;
  return (long long)wgrad_splits(D, N, X, Y, Z, cin, cout) * (8 / wgrad_quads(cout)) * (cout * cin * taps + cout);
}

void conv32_wgrad(int D, int k, WgradArgs A, float *dw, float *db, cudaStream_t st) {
  A.nq = wgrad_quads(A.cout);
  const int sx = wgrad_splits(D, A.N, A.X, A.Y, A.Z, A.cin, A.cout);
  if (D == 3) {
    if (k == 3) wgrad_launch<3, 3>(A, sx, st); else wgrad_launch<3, 1>(A, sx, st);
  } else {
    if (k == 3) wgrad_launch<2, 3>(A, sx, st); else wgrad_launch<2, 1>(A, sx, st);
  }
  const long long taps = D == 3 ? (long long)k * k * k : (long long)k * k, per = (long long)A.cout * A.cin * taps;
  k_wgrad_sum<<<(unsigned)((per + A.cout + 31) / 32), 256, 0, st>>>(A.partial, sx * (8 / A.nq), per, A.cout, dw, db);
}

}  // namespace ep
