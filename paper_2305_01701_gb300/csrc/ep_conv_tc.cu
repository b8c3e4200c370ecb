// ep_conv_tc.cu -- the warm-start network's 3^D convolutions as implicit GEMMs
// on the 5th-generation tensor cores (tcgen05), for its forward pass.
//
// Activations between the convolutions are BF16 in blocks of 8 channels,
// [n][channel / 8][z][y][x][8]: 16 bytes per voxel and block.  One CTA computes
// a brick of 8 x 16 x TZ output voxels (TZ = 4 or 2 slabs in 3D, 1 in 2D) for
// NB output channels: per slab, D[128 x NB] = sum over taps and input channels of
// A[128 x Cin] B[Cin x NB].
//   * A: 32 (or 16) input channels of the brick and its halo of one voxel arrive
//     as one TMA box (cp.async.bulk.tensor; zero fill outside the volume is the
//     convolution's padding) and serve all 27 taps: in shared memory a run of 8
//     voxels along x is a core matrix (8 rows of 16 bytes), the 16 runs of a
//     slab lie one halo row apart (stride offset), and a tap is only another
//     start address.
//   * B: the weights of a row of 3 taps for those channels, packed in the operand
//     layout and in the order they are used, by one bulk copy (cp.async.bulk) into
//     a ring.
//   * One elected thread issues tcgen05.mma (kind::f16, BF16 x BF16, FP32
//     accumulation in tensor memory), every slab of a tap from the same B.
// The epilogue (four warps, one accumulator row per thread) adds the bias,
// applies the ReLU and writes what the next layer reads: BF16 blocks, the 2^D
// average (FP32 sums), the nearest upsample, each straight into its place in the
// decoder's concatenation, or the 1^D head's FP32 output.
// Bound: one CTA of four warps per SM goes through its phases one after the other
// (the first box, the MMAs, the epilogue), so the tensor pipe is active 12 - 21 % of the
// time on the 64^3 layers and 36 - 41 % on the 16^3 ones (16 CTAs of 152); within the MMAs
// at NB = 32 the read of A from shared memory (4 KB per 32 cycles; L1 at 31 - 53 % of its
// rate over the kernel) allows half the tensor peak.  Measured on the 64^3 network (base
// 32): 0.417 ms for the pass (32 -> 32 channels 52 us, 96 -> 32 104 us), against 2.3 ms
// with a box of 8 channels per tap and FP32 tensors between the layers.
// Every wait is bounded; a wait that runs out sets the error word, the block
// waits (bounded) for the copies it issued, frees its tensor memory and ends.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "ep_conv.cuh"
#include "ep_internal.cuh"

namespace ep {

namespace {

constexpr int BX = 8, BY = 16;             // voxels of a slab: the accumulator's 128 rows
constexpr int HX = BX + 2, HY = BY + 2;    // with the halo
constexpr int ROWB = HX * 16;              // bytes of a halo row (one block of 8 channels)
constexpr int A_STAGES = 2, B_MAX = 8;   // B stages (a row of 3 taps each): as many as fit, up to B_MAX
constexpr int HEAD = 12;   // head outputs at a time
constexpr long long WAIT_LIMIT = 1ll << 31;   // SM cycles, about a second

__device__ __forceinline__ unsigned su32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mb_init(unsigned long long *b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_expect(unsigned long long *b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mb_try(unsigned long long *b, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mb_wait(unsigned long long *b, unsigned parity) {
  if (mb_try(b, parity)) return true;
  const long long t0 = clock64();
  while (!mb_try(b, parity))
    if (clock64() - t0 > WAIT_LIMIT) return false;
  return true;
}

template <int D>
__device__ __forceinline__ void tma_box(void *dst, const CUtensorMap *map, int x, int y, int z, int c,
                                        unsigned long long *bar) {
  if (D == 3)
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(su32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(c), "r"(su32(bar))
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n" ::"r"(su32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(c), "r"(su32(bar))
        : "memory");
}

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}

__device__ __forceinline__ void mma_commit(unsigned long long *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(su32(bar))
               : "memory");
}

// Shared-memory matrix descriptors, K-major without swizzle: address / 16 in
// bits 0 - 13, the stride between 8-channel blocks / 16 in bits 16 - 29, between
// 8-row groups / 16 in bits 32 - 45, bit 46 set.
// instruction descriptor: D FP32, A and B BF16, both K-major, M = 128, N = n
__host__ __device__ constexpr unsigned idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}

// what a CTA's shared memory holds after the A stages
struct Ctl {
  unsigned long long a_full[A_STAGES], a_empty[A_STAGES], b_full[B_MAX], b_empty[B_MAX], done;
  unsigned tmem_base;
  int fail, a_used, b_used;   // b_used, a_used: stages whose MMAs were issued
};

struct TcArgs {
  const __nv_bfloat16 *wpk;
  const float *bias;
  int *err;
  TcOut o;
  int X, Y, Z, cinp, cout, kc, bst, ncol;
};

__device__ __forceinline__ uint4 pack8(const float *v) {
  __nv_bfloat162 h[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
  return *reinterpret_cast<uint4 *>(h);
}

template <int D, int TZ, int KQ>
__global__ void __launch_bounds__(128, 1) k_conv_tc(const __grid_constant__ CUtensorMap map, const TcArgs A) {
  constexpr int HZ = D == 3 ? TZ + 2 : 1, TAPS = D == 3 ? 27 : 9;
  constexpr int CHB = HX * HY * HZ * 16;   // bytes of one block of 8 channels with the halo
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  constexpr int kc = 16 * KQ, kb = kc / 8;   // input channels per A stage
  const int nb = A.cout, nchunk = A.cinp / kc, bst = A.bst;
  const unsigned a_bytes = (unsigned)(kb * CHB), b_bytes = (unsigned)(3 * kc * nb * 2);
  const unsigned a_pitch = (a_bytes + 127u) & ~127u;
  unsigned char *sa = sm, *sb = sm + A_STAGES * a_pitch;
  __shared__ Ctl S;
  __shared__ __align__(16) float hw[128 * HEAD];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nbx = (A.X + BX - 1) / BX, nby = (A.Y + BY - 1) / BY;
  const int x0 = (int)(blockIdx.x % nbx) * BX, y0 = (int)(blockIdx.x / nbx % nby) * BY,
            z0 = (int)(blockIdx.x / (nbx * nby)) * TZ;
  const int n = blockIdx.y;

  if (threadIdx.x == 0) {
    for (int s = 0; s < A_STAGES; ++s) { mb_init(&S.a_full[s], 1); mb_init(&S.a_empty[s], 1); }
    for (int s = 0; s < bst; ++s) { mb_init(&S.b_full[s], 1); mb_init(&S.b_empty[s], 1); }
    mb_init(&S.done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    S.fail = 0;
    S.a_used = S.b_used = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(&S.tmem_base)),
                 "r"(A.ncol)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = S.tmem_base;
  volatile int *fail = &S.fail;

  if (warp == 0 && lane == 0) {
    // A producer: the halo brick of kc channels per stage
    int issued = 0;
    for (int c = 0; c < nchunk; ++c) {
      const int s = c % A_STAGES;
      if (c >= A_STAGES && !mb_wait(&S.a_empty[s], (unsigned)(c / A_STAGES - 1) & 1u)) { atomicExch(&S.fail, 1); break; }
      if (*fail) break;
      mb_expect(&S.a_full[s], a_bytes);
      tma_box<D>(sa + s * a_pitch, &map, (x0 - 1) * 8, y0 - 1, z0 - 1, n * (A.cinp / 8) + c * kb, &S.a_full[s]);
      issued = c + 1;
    }
    if (*fail)   // wait (bounded) for what was issued but not consumed
      for (int c = *(volatile int *)&S.a_used; c < issued; ++c)
        mb_wait(&S.a_full[c % A_STAGES], (unsigned)(c / A_STAGES) & 1u);
  } else if (warp == 2 && lane == 0) {
    // B producer: a row of 3 taps of kc input channels per stage
    int issued = 0, bs = 0;
    unsigned bph = 1;   // the first round's stages are empty
    const unsigned char *src = reinterpret_cast<const unsigned char *>(A.wpk);
    for (int it = 0; it < nchunk * (TAPS / 3); ++it, src += b_bytes) {
      if (it >= bst && !mb_wait(&S.b_empty[bs], bph)) { atomicExch(&S.fail, 1); break; }
      if (*fail) break;
      mb_expect(&S.b_full[bs], b_bytes);
      bulk_copy(sb + bs * b_bytes, src, b_bytes, &S.b_full[bs]);
      issued = it + 1;
      if (++bs == bst) { bs = 0; bph ^= 1u; }
    }
    if (*fail)
      for (int it = *(volatile int *)&S.b_used; it < issued; ++it)
        mb_wait(&S.b_full[it % bst], (unsigned)(it / bst) & 1u);
  } else if (warp == 1 && lane == 0) {
    // MMA issuer.  One thread issues every MMA, so its own instructions bound the
    // rate: descriptors are one 32-bit add each (their low words hold the address
    // and the leading stride, and no carry leaves them)
    const unsigned id = idesc_bf16(nb);
    const unsigned a_hi = (unsigned)(ROWB >> 4) | (1u << 14), b_hi = (128u >> 4) | (1u << 14);
    const unsigned a_lbo = (unsigned)(CHB >> 4) << 16, b_lbo = (unsigned)nb << 16, b_step = 2u * (unsigned)nb;
    bool ok = true;
    int it = 0, bs = 0;
    unsigned bph = 0;
    for (int c = 0; c < nchunk && ok; ++c) {
      const int as = c % A_STAGES;
      if (*fail || !mb_wait(&S.a_full[as], (unsigned)(c / A_STAGES) & 1u)) { ok = false; break; }
      const unsigned a0 = (su32(sa + as * a_pitch) >> 4) | a_lbo;
      for (int row = 0; row < TAPS / 3 && ok; ++row) {
        const unsigned ar = a0 + (unsigned)(((D == 3 ? row / 3 * HY : 0) + row % 3) * (ROWB / 16));
        if (!mb_wait(&S.b_full[bs], bph)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const unsigned bt = (su32(sb + bs * b_bytes) >> 4) | b_lbo;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
          for (int q = 0; q < KQ; ++q)
#pragma unroll
            for (int z = 0; z < TZ; ++z) {
              const unsigned al = ar + (unsigned)(dx + ((z * HY * ROWB + 2 * q * CHB) >> 4)), bl = bt + (dx * KQ + q) * b_step;
              asm volatile(
                  "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
                  " setp.ne.b32 p, %6, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(
                      tmem + (unsigned)(z * nb)),
                  "r"(al), "r"(a_hi), "r"(bl), "r"(b_hi), "r"(id), "r"(dx + q > 0 ? 1 : it)
                  : "memory");
            }
        mma_commit(&S.b_empty[bs]);
        ++it;
        *(volatile int *)&S.b_used = it;
        if (++bs == bst) { bs = 0; bph ^= 1u; }
      }
      if (ok) {
        mma_commit(&S.a_empty[as]);
        *(volatile int *)&S.a_used = c + 1;
      }
    }
    if (!ok) atomicExch(&S.fail, 1);
    mma_commit(&S.done);
  }
  __syncwarp();

  // epilogue: warp w reads accumulator rows 32 w .. 32 w + 31 of every slab
  if (!mb_wait(&S.done, 0u)) atomicExch(&S.fail, 1);
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const int m = warp * 32 + lane;
  const int vx = x0 + m % BX, vy = y0 + m / BX;
  const bool in_xy = vx < A.X && vy < A.Y && !*fail;
  const TcOut &O = A.o;
  auto ld16 = [&](int z, int c0, float *v) {
    unsigned r[16];
    const unsigned ta = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(z * nb + c0);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(ta)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float f = __uint_as_float(r[e]) + A.bias[c0 + e];
      v[e] = O.relu && f < 0.f ? 0.f : f;
    }
  };
  // 8 channels of a voxel into a blocked tensor of ch blocks and size (X, Y, Z)
  auto put = [&](__nv_bfloat16 *dst, int ch, int cb, int X, int Y, int Z, int x, int y, int z, const float *v) {
    const size_t e = ((((size_t)n * ch + cb) * Z + z) * Y + y) * X + x;
    *reinterpret_cast<uint4 *>(dst + e * 8) = pack8(v);
  };
  const long long nv = (long long)A.X * A.Y * A.Z;
  if (O.head_w) {
    // the 1^D head on the FP32 activations: a voxel's channels per thread, 12
    // outputs at a time, their weights as FP32 in shared memory [channel][12]
    for (int h0 = 0; h0 < O.head_c; h0 += HEAD) {
      __syncthreads();
      for (int i = threadIdx.x; i < nb * HEAD; i += 128) {
        const int h = h0 + i % HEAD;
        hw[i] = h < O.head_c ? __bfloat162float(O.head_w[(size_t)h * nb + i / HEAD]) : 0.f;
      }
      __syncthreads();
      for (int z = 0; z < TZ; ++z) {
        const bool in = in_xy && z0 + z < A.Z;
        const long long vox = ((long long)(z0 + z) * A.Y + vy) * A.X + vx;
        float acc[HEAD];
#pragma unroll
        for (int h = 0; h < HEAD; ++h) acc[h] = h0 + h < O.head_c ? O.head_b[h0 + h] : 0.f;
        for (int c0 = 0; c0 < nb; c0 += 16) {
          float v[16];
          ld16(z, c0, v);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float4 *w = reinterpret_cast<const float4 *>(hw + (c0 + e) * HEAD);
#pragma unroll
            for (int q = 0; q < HEAD / 4; ++q) {
              const float4 f = w[q];
              acc[4 * q] += f.x * v[e];
              acc[4 * q + 1] += f.y * v[e];
              acc[4 * q + 2] += f.z * v[e];
              acc[4 * q + 3] += f.w * v[e];
            }
          }
        }
        if (in)
#pragma unroll
          for (int h = 0; h < HEAD; ++h)
            if (h0 + h < O.head_c) O.f32[((long long)n * O.head_c + h0 + h) * nv + vox] = O.scale * acc[h];
      }
    }
  } else {
    for (int c0 = 0; c0 < nb; c0 += 16) {
      float pool[16];
      for (int z = 0; z < TZ; ++z) {
        float v[16];
        ld16(z, c0, v);
        const int gz = z0 + z;
        const bool in = in_xy && gz < A.Z;
        const int cb = c0 / 8;
        if (in && O.f32) {
          const long long vox = ((long long)gz * A.Y + vy) * A.X + vx;
#pragma unroll
          for (int e = 0; e < 16; ++e) O.f32[((long long)n * nb + c0 + e) * nv + vox] = v[e];
        }
        if (in && O.b16) {
          put(O.b16, O.b16_ch, O.b16_off + cb, A.X, A.Y, A.Z, vx, vy, gz, v);
          put(O.b16, O.b16_ch, O.b16_off + cb + 1, A.X, A.Y, A.Z, vx, vy, gz, v + 8);
        }
        if (in && O.up) {   // nearest upsample: this voxel's 2^D fine ones
          for (int f = 0; f < (D == 3 ? 8 : 4); ++f)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              put(O.up, O.up_ch, cb + h, 2 * A.X, 2 * A.Y, D == 3 ? 2 * A.Z : 1, 2 * vx + (f & 1), 2 * vy + (f >> 1 & 1),
                  D == 3 ? 2 * gz + (f >> 2) : 0, v + 8 * h);
        }
        if (O.pool) {   // mean of 2^D voxels: z here, then x and y across lanes
          if (D == 2 || (z & 1) == 0)
#pragma unroll
            for (int e = 0; e < 16; ++e) pool[e] = v[e];
          else
#pragma unroll
            for (int e = 0; e < 16; ++e) pool[e] += v[e];
          if (D == 2 || (z & 1)) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              pool[e] += __shfl_xor_sync(0xffffffffu, pool[e], 1);
              pool[e] += __shfl_xor_sync(0xffffffffu, pool[e], 8);
              pool[e] *= D == 3 ? 0.125f : 0.25f;
            }
            if (in && !(lane & 1) && !(lane & 8)) {
              const int pz = D == 3 ? gz / 2 : 0, pZ = D == 3 ? A.Z / 2 : 1;
              put(O.pool, nb / 8, cb, A.X / 2, A.Y / 2, pZ, vx / 2, vy / 2, pz, pool);
              put(O.pool, nb / 8, cb + 1, A.X / 2, A.Y / 2, pZ, vx / 2, vy / 2, pz, pool + 8);
            }
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && S.fail) atomicExch(A.err, 1);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(A.ncol) : "memory");
  }
}

// FP32 N x C x V -> BF16 blocks N x Cp/8 x V x 8 (channels >= C zero)
__global__ void k_to_blocks(const float *x, int N, int C, long long nv, int cp, __nv_bfloat16 *out) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)N * (cp / 8) * nv) return;
  const long long v = t % nv, b = t / nv;
  const int cb = (int)(b % (cp / 8));
  const long long n = b / (cp / 8);
  float f[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) f[q] = 8 * cb + q < C ? x[(n * C + 8 * cb + q) * nv + v] : 0.f;
  *reinterpret_cast<uint4 *>(out + t * 8) = pack8(f);
}

// BF16 co x ci x taps -> the B stages in the order they are used, per layer:
// [chunk of kc input channels][tap][8-channel block][co][8 channels]; channels
// >= ci are zero
__host__ __device__ constexpr int chunk_of(int cinp) { return cinp % 32 == 0 ? 32 : 16; }
__global__ void k_pack_weights(const PackTable P, const __nv_bfloat16 *w, __nv_bfloat16 *out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.total) return;
  int l = 0;
  while (l + 1 < P.n && i >= P.dst[l + 1]) ++l;
  const int cin = P.cin[l], cout = P.cout[l], kc = chunk_of(conv_tc_cinp(cin));
  const int t = (int)(i - P.dst[l]);   // taps * cinp * cout elements
  const int e = t % 8, co = t / 8 % cout, cb = t / (8 * cout) % (kc / 8), tap = t / (kc * cout) % P.taps;
  const int ci = t / (kc * cout * P.taps) * kc + 8 * cb + e;
  out[i] = ci < cin ? w[P.src[l] + ((long long)co * cin + ci) * P.taps + tap] : __float2bfloat16_rn(0.f);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    return ok ? (EncodeTiledFn)p : nullptr;
  }();
  return fn;
}

constexpr size_t SMEM_MAX = 216 * 1024;   // beside the static arrays

template <int D, int TZ, int KQ>
cudaError_t tc_launch(const CUtensorMap &map, TcArgs A, int N, cudaStream_t st) {
  // shared memory: two A stages, and as many B stages as fit
  const size_t a = ((size_t)(A.kc / 8) * HX * HY * (D == 3 ? TZ + 2 : 1) * 16 + 127) / 128 * 128;
  const size_t b = 3 * (size_t)A.kc * A.cout * 2;
  A.bst = (int)std::min<size_t>(B_MAX, (SMEM_MAX - 128 - A_STAGES * a) / b);
  A.ncol = 32;
  while (A.ncol < TZ * A.cout) A.ncol *= 2;
  const unsigned bricks = (unsigned)(((A.X + BX - 1) / BX) * ((A.Y + BY - 1) / BY) * ((A.Z + TZ - 1) / TZ));
  dim3 grid(bricks, (unsigned)N);
  k_conv_tc<D, TZ, KQ><<<grid, 128, A_STAGES * a + A.bst * b + 128, st>>>(map, A);
  return cudaGetLastError();
}

}  // namespace

cudaError_t conv_tc_configure() {
  cudaError_t e = cudaSuccess;
#define EP_CFG(d, tz, kq)                                                                                       \
  if (e == cudaSuccess)                                                                                         \
    e = cudaFuncSetAttribute(k_conv_tc<d, tz, kq>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
  EP_CFG(2, 1, 1) EP_CFG(2, 1, 2) EP_CFG(3, 2, 1) EP_CFG(3, 2, 2) EP_CFG(3, 4, 1) EP_CFG(3, 4, 2)
#undef EP_CFG
  return e;
}

bool conv_tc_supported(int k, int cout) { return k == 3 && cout >= 16 && cout <= 128 && cout % 16 == 0; }

void conv_tc_to_blocks(const float *x, int N, int C, long long nv, __nv_bfloat16 *out, cudaStream_t st) {
  const int cp = conv_tc_cinp(C);
  const long long total = (long long)N * nv * (cp / 8);
  k_to_blocks<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(x, N, C, nv, cp, out);
}

void conv_tc_pack_weights(const PackTable &P, const __nv_bfloat16 *w, __nv_bfloat16 *out, cudaStream_t st) {
  k_pack_weights<<<(unsigned)((P.total + 255) / 256), 256, 0, st>>>(P, w, out);
}

cudaError_t conv_tc_forward(int D, const __nv_bfloat16 *xb, int N, int X, int Y, int Z, int cin,
                            const __nv_bfloat16 *wpk, const float *bias, int cout, const TcOut &out, int *err,
                            cudaStream_t st) {
  const EncodeTiledFn fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  TcArgs A{};
  A.wpk = wpk; A.bias = bias; A.err = err; A.o = out;
  A.X = X; A.Y = Y; A.Z = D == 3 ? Z : 1; A.cinp = conv_tc_cinp(cin); A.cout = cout;
  A.kc = chunk_of(A.cinp);
  // slabs per CTA: 4 share a halo and the weights best; 2 (pooling needs pairs)
  // where 4 would leave SMs idle
  const long long cols = (long long)((X + BX - 1) / BX) * ((Y + BY - 1) / BY) * N;
  const int tz = D == 2 ? 1 : cols * ((A.Z + 3) / 4) >= 152 ? 4 : 2;
  CUtensorMap map;
  const int ch = A.cinp / 8;
  CUresult r;
  if (D == 3) {
    cuuint64_t dims[4] = {(cuuint64_t)X * 8, (cuuint64_t)Y, (cuuint64_t)A.Z, (cuuint64_t)N * ch};
    cuuint64_t strides[3] = {(cuuint64_t)X * 16, (cuuint64_t)X * Y * 16, (cuuint64_t)X * Y * A.Z * 16};
    cuuint32_t box[4] = {HX * 8, HY, (cuuint32_t)(tz + 2), (cuuint32_t)(A.kc / 8)}, es[4] = {1, 1, 1, 1};
    r = fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16 *>(xb), dims, strides, box, es,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    cuuint64_t dims[3] = {(cuuint64_t)X * 8, (cuuint64_t)Y, (cuuint64_t)N * ch};
    cuuint64_t strides[2] = {(cuuint64_t)X * 16, (cuuint64_t)X * Y * 16};
    cuuint32_t box[3] = {HX * 8, HY, (cuuint32_t)(A.kc / 8)}, es[3] = {1, 1, 1};
    r = fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16 *>(xb), dims, strides, box, es,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  if (A.kc == 32) {
    if (D == 2) return tc_launch<2, 1, 2>(map, A, N, st);
    return tz == 4 ? tc_launch<3, 4, 2>(map, A, N, st) : tc_launch<3, 2, 2>(map, A, N, st);
  }
  if (D == 2) return tc_launch<2, 1, 1>(map, A, N, st);
  return tz == 4 ? tc_launch<3, 4, 1>(map, A, N, st) : tc_launch<3, 2, 1>(map, A, N, st);
}

}  // namespace ep
