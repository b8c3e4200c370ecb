// ep_fused3d_reg.cu -- the fused 3D iteration with the z-march held in
// registers.
//
// Same arithmetic and z-march as ep_fused3d.cu (spin, relaxed trial, centre
// return, edge return, velocity update; Eqs. A5, A23ssP, A2ssP, A6121lambda,
// A22S, A22P), mapped so that little but a plane's inputs goes through shared
// memory:
//   * a block covers a window of 32 x H columns (x, y) of the box and walks
//     them through a chunk of z-planes; the inner 28 x (H-4) columns are
//     written (the iteration couples columns two apart);
//   * FP32: a thread owns two adjacent x columns as one float2 and half a
//     warp owns a row (H = 24: 384 threads of 168 registers, the whole file);
//     FP64: a thread owns one column, a warp a row;
//   * a plane's 23 inputs arrive as TMA boxes (cp.async.bulk.tensor, zero
//     outside the box) in one of two stages: plane t + 2 is asked for when
//     every warp has read plane t, a whole plane before it is needed; each
//     warp's elected thread issues its share;
//   * x +- 1 neighbours are warp shuffles of registers (one per pair);
//   * y +- 1 neighbours are rows of shared memory, each written once by its
//     owner (two plane slots where a value is read one plane later);
//   * z - 1 neighbours are registers carried from the previous plane.
// Plane t of the march computes spins at plane t, edge trials at face t and
// plane t-1, centres t-1, edges t-1 and velocities t-2.  Three block barriers
// separate the steps of a plane.
// Bound: HBM in principle (132 B per cell); in fact the latency of a plane's
// three steps at 12 warps per SM.  Measured (FP32, one sweep): 127^3 80.5 us,
// 383^3 1611 us (4.6 TB/s), against 126.9 and 2312 us of the form with one
// column per thread (16 warps, 600 instructions per warp and plane, register
// prefetch).  Packing the pairs alone, with the register prefetch (8 warps of
// 255 registers), halved the instructions and gained nothing: the loads'
// latency showed.  cp.async in place of TMA cost 5 shared-memory wavefronts
// per 8-byte copy (the window starts off a 32-byte sector): 131 and 2164 us.
// With a per-cell shear modulus (31 inputs, 16 rows) 95^3 takes 56 us, the five
// staged kernels 100 to 124.
// Instruction count:
//   * FP32 arithmetic is packed (add/mul/fma on float2: one instruction per
//     pair);
//   * a mean of four neighbours is a sum of two pair sums: the pair sum along
//     x or z is formed once by its owner and shared (shuffle, shared row or
//     carried register) by the two or three means that need it, and the
//     factors 1/2, 1/4, 1/8 are folded into the coefficients (exact powers of
//     two);
//   * walls are factors of 0 and 1 per column on the spins, the trials and the
//     velocity step, and blocks whose whole window lies inside the domain run
//     a copy of the body without them: what a window's outermost columns and
//     rows compute is never read by a written point;
//   * the march is unrolled by two planes, so the stage and the slot of each
//     copy are compile-time constants;
//   * offsets within an array are 32-bit when the box has fewer than 2^31
//     points (FP32);
//   * warps whose rows are never written skip the steps that only written
//     rows need.
// Waits are bounded (ep_solver_opts.wait_cycles): one that runs out marks the grid's
// record (status 4), the block waits, with the default bound, for the copies in flight
// and returns.
// Check iterations (FP32, CHK = true) also reduce the stopping measures of
// Eqs. Convergence1-3 over the points each block writes, the same point sets
// and the same snapshot updates as the staged check iteration: max|sigma|,
// max|tau - tau_chk|, max|p - p_chk| at centres and edges, max|R|,
// max|u - u_chk| and max|v0 + u| at faces, and they store the centre scales
// (held when plasticity freezes).  One atomic per block and measure.  The
// snapshot values a thread checks in a plane are copied to shared memory with
// cp.async at the plane's start and read after the second barrier, so that
// their memory latency hides behind the plane's first steps.
#include <cuda.h>
#include <math.h>

#include <type_traits>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"

namespace ep {

namespace {

constexpr int WX = 32;       // window columns
constexpr int OX = WX - 4;   // written columns per block
constexpr unsigned FULL = 0xffffffffu;

// ---- the columns of one thread -------------------------------------------
// LaneF: two adjacent FP32 columns, 16 threads per row, H_ rows per block.
// LaneD: one FP64 column, 32 threads per row, 8 rows per block.
template <int H_>
struct LaneF {
  using T = float;
  using V = float2;
  static constexpr int N = 2, LPR = 16, H = H_;
};
struct LaneD {
  using T = double;
  using V = double;
  static constexpr int N = 1, LPR = 32, H = 8;
};

// v off the domain's boundary, 0 on it: m holds 1 or 0 per column.  INT
// windows have no boundary columns.
template <bool INT, typename V>
__device__ __forceinline__ V keep(V m, V v) {
  return INT ? v : vmul(m, v);
}

// One plane slot of a value per thread, as rows of the window
template <typename L>
struct Rows {
  typename L::V r[L::H * L::LPR];
};

// inputs of a plane: face/edge arrays of plane t, centre arrays of plane t - 1
enum {
  I_U0, I_U1, I_U2, I_RQ0, I_RQ1, I_RQ2, I_RD0, I_RD1, I_SOXZ, I_SOYZ, I_TBXZ, I_TBYZ,
  I_SON0, I_SON1, I_SON2, I_TBN0, I_TBN1, I_TBN2, I_SOXY, I_TBXY, I_SOP, I_PB, I_YC,
  I_COUNT,
  // with a per-cell shear modulus also 2 eta_ve and c2 of the points of plane t - 1
  // (centres, xy) and plane t (xz, yz)
  I_GEN = I_COUNT, I_GCN, I_GEXY, I_GCXY, I_GEXZ, I_GCXZ, I_GEYZ, I_GCYZ,
  I_COUNT_G
};
template <bool GC>
constexpr int inputs() { return GC ? I_COUNT_G : I_COUNT; }

// columns of a TMA box: the window and two more on either side, so that its
// first column is a multiple of 16 bytes
constexpr int BX = WX + 4;

template <typename L, bool GC>
struct SmemR {
  alignas(128) typename L::T in[2][inputs<GC>()][L::H * BX];   // inputs of planes t and t + 1 (then t + 2)
  static_assert(sizeof(in[0][0]) % 128 == 0, "a TMA box lands on a 128-byte boundary");
  Rows<L> A, D, I, K;               // sums of neighbouring inputs
  Rows<L> B, E, wxz, M, pyz;        // pair sums of spins and rotation products
  Rows<L> Q, Sz, U, Vs;             // pair sums of the edge trials and of the scales
  Rows<L> syy[2], nxy[2], nyz[2];   // read one plane later
  alignas(8) unsigned long long full[2];   // a stage's copies have arrived
};

template <bool GC>
struct Maps {
  CUtensorMap m[inputs<GC>()];
};

template <typename T>
struct Args {
  T *snn[3], *sns[3], *snp, *uo[3];
  T *s;   // centre return scales (read when plasticity is frozen, written by checks)
  bool keep_s;   // written by this iteration too (GC: the last one of a chunk)
  T *cn[3], *cs[3], *cp, *uchk[3];   // state at the previous check (check iterations)
  const double *v0[3];               // start velocity (check iterations)
};

// a check iteration's snapshot values, one slot per thread, after SmemR
template <typename L>
struct ChkSlots {
  static constexpr int NT = L::LPR * L::H;
  double v0[3][NT * L::N];
  typename L::V cn[3][NT], cs[3][NT], cp[NT], uchk[3][NT];
};

template <int BYTES>
__device__ __forceinline__ void cp_async_el(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"(BYTES));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::); }

__device__ __forceinline__ unsigned su32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_expect(unsigned long long *b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(b)), "r"(bytes) : "memory");
}
// bounded wait for a phase of b: gives up after the grid's bound (sc null: the default, far
// above any copy's latency).  A bound below the default polls with test_wait, which does
// not suspend the thread, so that the bound decides when the wait gives up.
__device__ __forceinline__ bool bar_test(unsigned long long *b, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool bar_wait(unsigned long long *b, unsigned parity, const Scal *sc) {
  if (bar_test(b, parity)) return true;
  const long long limit = sc ? wait_limit(sc) : WAIT_DEFAULT, t0 = clock64();
  do {
    unsigned ok;
    if (limit < WAIT_DEFAULT)
      ok = bar_test(b, parity);
    else
      asm volatile(
          "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
          : "=r"(ok)
          : "r"(su32(b)), "r"(parity)
          : "memory");
    if (ok) return true;
  } while (clock64() - t0 <= limit);
  return false;
}
__device__ __forceinline__ void tma_load(void *dst, const CUtensorMap *map, int x, int y, int z,
                                         unsigned long long *b) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::
          "r"(su32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(su32(b))
      : "memory");
}

template <typename T>
__device__ __forceinline__ T maxt(T a, T b) { return (a > b || a != a) ? a : b; }
__device__ __forceinline__ float absv(float x) { return fabsf(x); }

// block-wide max of a non-negative value as its IEEE bits (integer order; a
// NaN sorts above infinity), one atomic per block
__device__ __forceinline__ void block_max_bits(double v, unsigned long long *slot) {
  __shared__ unsigned long long part[32];
  unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(FULL, b, o);
    b = b > w ? b : w;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) part[wid] = b;
  __syncthreads();
  if (wid == 0) {
    b = lane < (int)(blockDim.x >> 5) ? part[lane] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(FULL, b, o);
      b = b > w ? b : w;
    }
    if (lane == 0 && b) atomicMax(slot, b);
  }
}

// INT: every column of the block's window lies strictly inside the domain
// (1 <= x, y index <= n - 1), so the domain-boundary tests fold away.
// Off: the integer type of offsets within an array.  CHK: a check iteration.
// GC: a per-cell shear modulus.
template <typename L, bool GC, bool INT, typename Off, bool CHK>
__device__ __forceinline__ void reg_body(const Maps<GC> &M, const Args<typename L::T> &A, const Geo &g, const Scal *sc, DevInfo *di,
                                         bool frozen, int kz, unsigned char *smem_raw) {
  using T = typename L::T;
  using V = typename L::V;
  constexpr int N = L::N, H = L::H, LPR = L::LPR;
  SmemR<L, GC> &S = *reinterpret_cast<SmemR<L, GC> *>(smem_raw);
  ChkSlots<L> &C = *reinterpret_cast<ChkSlots<L> *>(smem_raw + sizeof(SmemR<L, GC>));   // CHK only
  const int a = threadIdx.x % LPR, b = threadIdx.x / LPR;
  const int i0 = blockIdx.x * OX, j0 = blockIdx.y * (H - 4);
  const int gi = i0 - 2 + N * a, gj = j0 - 2 + b;   // first column of the thread, row
  const int kb = blockIdx.z * kz, ke = min(kb + kz, g.pz);
  const int nx = g.nx, ny = g.ny, nz = g.nz, pz = g.pz;
  const Off px = (Off)g.px, plane = (Off)g.plane;
  // inside the domain: x1, y1 a vertex/edge line off the walls; x0, y0 a centre
  auto in_x1 = [&](int e) { return INT || (gi + e >= 1 && gi + e <= nx - 1); };
  auto in_x0 = [&](int e) { return INT || (gi + e >= 0 && gi + e < nx); };
  const bool gy1 = INT || (gj >= 1 && gj <= ny - 1), gy0 = INT || (gj >= 0 && gj < ny);
  auto mask = [](bool e0, bool e1, T v) -> V {
    if constexpr (N == 2) return make_float2(e0 ? v : (T)0, e1 ? v : (T)0);
    else return e0 ? v : (T)0;
  };
  const V m_xy = mask(in_x1(0) && gy1, in_x1(1) && gy1, (T)1), m_xz = mask(in_x1(0) && gy0, in_x1(1) && gy0, (T)1),
          m_yz = mask(in_x0(0) && gy1, in_x0(1) && gy1, (T)1);
  const bool inb = INT || (gi >= 0 && gi < g.px && gj >= 0 && gj < g.py);   // px is a multiple of N
  // this thread's offset in a plane, clamped into the box; every store and the
  // frozen-scale read are guarded by in-box tests, where it is the exact one
  const Off col = (Off)min(max(gj, 0), g.py - 1) * px + (Off)min(max(gi, 0), g.px - N);

  const bool out_col = N * a >= 2 && N * a < WX - 2 && b >= 2 && b < H - 2 && inb;
  // rows of this warp: which steps some written row needs
  constexpr int RPW = 32 / LPR;
  const int b0 = (int)(threadIdx.x >> 5) * RPW, b1 = b0 + RPW - 1;
  const bool w_edge = b1 >= 2, w_vel = b1 >= 2 && b0 < H - 2;

  const SweepScal<T> &Q = sweep_scal<T>(sc);
  const T rdx = Q.rdx, rdy = Q.rdy, rdz = Q.rdz;
  const T eta = Q.eta, two_eta = Q.two_eta, bt = Q.bt, ob = Q.ob;
  const T bp = Q.bp, obp = Q.obp, KDt = Q.KDt, Acoef = Q.A;
  const T vs = Q.vstep, qr = (T)0.25, e8 = (T)0.125, e32 = (T)0.03125;
  // velocity step of x-, y- and z-faces: 0 on the walls and off the extent
  const V st0 = mask(in_x1(0) && gy0, in_x1(1) && gy0, vs), st1 = mask(in_x0(0) && gy1, in_x0(1) && gy1, vs),
          st2 = mask(in_x0(0) && gy0, in_x0(1) && gy0, vs);
  auto bc = [](T v) -> V { return Splat<V>::of(v); };   // the same value in every column
  const V zero = bc((T)0);
  // this thread's place in a Rows slot, and its row neighbours' (clamped: the
  // window's first and last rows read a value that no written point uses)
  const int bm = max(b - 1, 0), bq = min(b + 1, H - 1);
  const int q0 = b * LPR + a, qm = bm * LPR + a, qp = bq * LPR + a;
  const int p0 = b * BX + 2 + N * a, pm = bm * BX + 2 + N * a, pp = bq * BX + 2 + N * a;   // the same in a stage

  auto ldv = [&](const T *p, Off e) -> V { return __ldg(reinterpret_cast<const V *>(p + e)); };
  auto stv = [&](T *p, Off e, V v) { *reinterpret_cast<V *>(p + e) = v; };
  auto lev = [&](int k) -> Off { return (Off)min(max(k, 0), pz - 1) * plane + col; };

  // the elected thread of each warp copies its share of a plane's input boxes
  // into a stage: face/edge arrays of plane t, centre arrays of plane t - 1
  constexpr int NW = LPR * H / 32;
  constexpr unsigned BOX = H * BX * sizeof(T);
  const int warp = threadIdx.x >> 5;
  const bool elected = (threadIdx.x & 31) == 0;
  auto fetch = [&](int t, const int stage) {
    if (!elected) return;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    constexpr int NI = inputs<GC>();
    bar_expect(&S.full[stage], (unsigned)((NI - warp + NW - 1) / NW) * BOX);
    for (int k = warp; k < NI; k += NW)
      tma_load(S.in[stage][k], &M.m[k], i0 - 4, j0 - 2, k < I_SON0 || k >= I_GEXZ ? t : t - 1, &S.full[stage]);
  };
  if (threadIdx.x == 0) {
    for (int q = 0; q < 2; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(&S.full[q])), "r"(NW) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();

  // plane history (suffix: _1 plane t-1, _2 plane t-2, _3 plane t-3)
  V u0 = zero, u1 = zero, u2 = zero, u0_1 = zero, u1_1 = zero, u2_1 = zero, u0_2 = zero, u1_2 = zero, u2_2 = zero;
  V rq0 = zero;
  V D_1 = zero, E_1 = zero, F_1 = zero, G_1 = zero, J_1 = zero, L_1 = zero, M_1 = zero, N_1 = zero, O_1 = zero;
  V wxy_1 = zero, qxy_1 = zero, gxy_1 = zero, g1_1 = zero, tsxz_1 = zero, tsyz_1 = zero;
  V s_2 = zero, U_2 = zero;                                // quarter scale and its x pair sum, plane t-2
  V sxx_2 = zero, syy_2 = zero, szz_2 = zero, szz_3 = zero;   // centre stress minus pressure
  V nxy_2 = zero, nxz_2 = zero, nyz_2 = zero;              // edge stress, level t-2
  // check iterations: the stopping measures over this block's points
  T c_sig = 0, c_dtau = 0, c_dp = 0, c_r = 0, c_du = 0;
  double c_vm = 0.0;

  fetch(kb - 2, 0);
  fetch(kb - 1, 1);
  unsigned ph[2] = {0u, 0u};   // the phase of each stage that is waited for next
  // wait until a stage's copies have arrived; false once a wait has run out
  // anywhere in the block: the record then says so and the copies in flight
  // (a plane in each stage at most) have been waited for
  auto arrived = [&](const int stage, bool other) -> bool {
    const bool ok = bar_wait(&S.full[stage], ph[stage], sc);
    ph[stage] ^= 1u;
    if (!__syncthreads_or(!ok)) return true;
    if (threadIdx.x == 0 && di != nullptr) di->done = 4;
    if (!ok) bar_wait(&S.full[stage], ph[stage] ^ 1u, nullptr);
    if (other) bar_wait(&S.full[stage ^ 1], ph[stage ^ 1], nullptr);
    return false;
  };
  if (!arrived(0, true)) return;
  // the march unrolled by two planes: the slot parity of each copy is a
  // compile-time constant
  auto plane_step = [&](const int t, auto slc) -> bool {
    constexpr int sl = decltype(slc)::value, sl1 = sl ^ 1;  // plane slots of t and t - 1
    auto own = [&](int k) -> V { return *reinterpret_cast<const V *>(&S.in[sl][k][p0]); };
    auto below = [&](int k) -> V { return *reinterpret_cast<const V *>(&S.in[sl][k][pm]); };   // row y - 1
    auto above = [&](int k) -> V { return *reinterpret_cast<const V *>(&S.in[sl][k][pp]); };   // row y + 1
    // ---- 0. take this plane's inputs (they lie in its stage) ----
    u0_2 = u0_1; u1_2 = u1_1; u2_2 = u2_1;
    u0_1 = u0; u1_1 = u1; u2_1 = u2;
    u0 = own(I_U0); u1 = own(I_U1); u2 = own(I_U2);
    const V rq0_1 = rq0, rq1 = own(I_RQ1), rq2 = own(I_RQ2);
    rq0 = own(I_RQ0);
    // sums of inputs: A = rq0 over planes t-1, t; D = rq2, I = rd0, J = rd1
    // over columns x-1, x; K = rd1 - rd0
    const V rd0 = own(I_RD0), rd1 = own(I_RD1);
    const V vA = vadd(rq0_1, rq0), D = vadd(rq2, xm<LPR>(rq2)), vI = vadd(rd0, xm<LPR>(rd0)), J = vadd(rd1, xm<LPR>(rd1));
    const V vK = vsub(rd1, rd0);
    S.A.r[q0] = vA; S.D.r[q0] = D; S.I.r[q0] = vI; S.K.r[q0] = vK;
    if constexpr (CHK) {   // the snapshot values checked at this plane: levels t-1 (centres, edges), t-2 (faces)
      const int tid = threadIdx.x;
      const Off e1 = lev(t - 1), e2 = lev(t - 2);
      constexpr int VB = (int)sizeof(V);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        cp_async_el<VB>(&C.cn[d][tid], A.cn[d] + e1);
        cp_async_el<VB>(&C.cs[d][tid], A.cs[d] + e1);
        cp_async_el<VB>(&C.uchk[d][tid], A.uchk[d] + e2);
        cp_async_el<8 * N>(&C.v0[d][N * tid], A.v0[d] + e2);
      }
      cp_async_el<VB>(&C.cp[tid], A.cp + e1);
      cp_async_commit();
    }
    const bool zf = t >= 1 && t <= nz - 1;   // face t carries xz/yz edges inside the domain

    // ---- 1. shear strain rates g = 2 eps and spins w = 2 omega at plane t
    //         (xy) / face t (xz, yz) ----
    V gxy, wxy, gxz, wxz, gyz, wyz;
    {
      const V u0_ym = below(I_U0), u2_ym = below(I_U2);
      V x = vmul(vsub(u0, u0_ym), bc(rdy)), y = vsub(u1, xm<LPR>(u1));
      gxy = vfma(y, bc(rdx), x);
      wxy = keep<INT>(m_xy, vfma(y, bc(-rdx), x));
      x = vmul(vsub(u0, u0_1), bc(rdz)); y = vsub(u2, xm<LPR>(u2));
      gxz = vfma(y, bc(rdx), x);
      wxz = keep<INT>(m_xz, vfma(y, bc(-rdx), x));
      x = vmul(vsub(u1, u1_1), bc(rdz)); y = vsub(u2, u2_ym);
      gyz = vfma(y, bc(rdy), x);
      wyz = keep<INT>(m_yz, vfma(y, bc(-rdy), x));
      if (t < 0 || t >= nz) wxy = zero;
      if (!zf) { wxz = zero; wyz = zero; }
    }
    // rotation products (2 rq omega) and the pair sums that their means and
    // the spin means share
    const V pxy = vmul(rq0, wxy), pxz = vmul(rq1, wxz), pyz = vmul(rq2, wyz);
    const V vB = vadd(wxy_1, wxy), vE = vadd(wyz, xm<LPR>(wyz)), vM = vadd(pxy, xp<LPR>(pxy)), vN = vadd(pxz, xp<LPR>(pxz));
    S.B.r[q0] = vB; S.E.r[q0] = vE; S.wxz.r[q0] = wxz; S.M.r[q0] = vM; S.pyz.r[q0] = pyz;
    __syncthreads();

    // ---- 2. relaxed trials: faces t (xz, yz), plane t-1 (xy, centres) ----
    const int lc = t - 1;
    const bool zc = lc >= 0 && lc < nz;
    // an edge's trial: base + eta g + rotation r (in units of sc), each point's
    // own 2 eta_ve and c2 with a per-cell modulus
    auto trial = [&](V r, T unit, V gs, int tb, int ge) -> V {
      if constexpr (GC) return vfma(vmul(r, bc(unit)), own(ge + 1), vfma(vmul(gs, bc((T)0.5)), own(ge), own(tb)));
      else return vfma(r, bc(unit), vfma(gs, bc(eta), own(tb)));
    };
    V tsxz, tsyz, tsxy, c0v, c1v, c2v, div;
    const V sop = own(I_SOP), pb = own(I_PB), yc = own(I_YC);
    {
      const V F = vadd(rq1, below(I_RQ1)), G = vadd(wxz, S.wxz.r[qm]);   // over rows y-1, y
      const V Lz = vadd(vK, S.K.r[qm]), dyx = vadd(vI, S.I.r[qm]);
      {   // xz: w dzx + (Tyz Wxy - Txy Wyz) / 4, in units of 1/8
        const V Dz = vadd(J_1, J), Tyz = vadd(D, S.D.r[qp]), Wyz = vadd(vE, S.E.r[qp]);
        const V Txy = vadd(vA, S.A.r[qp]), Wxy = vadd(vB, S.B.r[qp]);
        const V r1 = vsub(vmul(Tyz, Wxy), vmul(Txy, Wyz));
        const V r = vfma(r1, bc(qr), vmul(wxz, Dz));
        const V tr = trial(r, e8, gxz, I_TBXZ, I_GEXZ);
        tsxz = keep<INT>(m_xz, vfma(own(I_SOXZ), bc(bt), vmul(tr, bc(ob))));
      }
      {   // yz: w dzy - (Txy Wxz + Txz Wxy) / 4
        const V Dz = vadd(L_1, Lz), Txy = vadd(vA, xp<LPR>(vA)), Wxy = vadd(vB, xp<LPR>(vB));
        const V Txz = vadd(F, xp<LPR>(F)), Wxz = vadd(G, xp<LPR>(G));
        const V r1 = vfma(Txz, Wxy, vmul(Txy, Wxz));
        const V r = vfma(r1, bc(-qr), vmul(wyz, Dz));
        const V tr = trial(r, e8, gyz, I_TBYZ, I_GEYZ);
        tsyz = keep<INT>(m_yz, vfma(own(I_SOYZ), bc(bt), vmul(tr, bc(ob))));
      }
      if (!zf) { tsxz = zero; tsyz = zero; }
      {   // xy of plane t-1: w dyx + (Tyz Wxz + Txz Wyz) / 4
        const V Tyz = vadd(D_1, D), Wyz = vadd(E_1, vE), Txz = vadd(F_1, F), Wxz = vadd(G_1, G);
        const V r1 = vfma(Tyz, Wxz, vmul(Txz, Wyz));
        V tr;
        if constexpr (GC) tr = trial(vfma(r1, bc(qr), qxy_1), e8, gxy_1, I_TBXY, I_GEXY);
        else tr = vfma(r1, bc(e32), vadd(own(I_TBXY), qxy_1));
        tsxy = keep<INT>(m_xy, vfma(own(I_SOXY), bc(bt), vmul(tr, bc(ob))));
        if (!zc) tsxy = zero;
        // this plane's part of the next plane's xy trial
        if constexpr (GC) {
          qxy_1 = vmul(wxy, dyx);
          gxy_1 = gxy;
        } else {
          qxy_1 = vfma(gxy, bc(eta), vmul(vmul(wxy, dyx), bc(e8)));
        }
      }
      {   // centres of plane t-1
        const V g0 = vsub(xp<LPR>(u0_1), u0_1), g1 = g1_1, g2 = vsub(u2, u2_1);
        div = vfma(g2, bc(rdz), vfma(g1, bc(rdy), vmul(g0, bc(rdx))));
        const V O = vadd(pyz, S.pyz.r[qp]);
        const V Pxz = vadd(N_1, vN), Pyz = vadd(O_1, O), Pxy = M_1;
        // the deviatoric rate e - div / 3 is rounded once and scaled after: 2 eta e and
        // -2 eta div / 3 as two terms would round each at the size of the larger
        const V d3 = vmul(div, bc((T)(-1.0 / 3.0)));
        const V d0 = vfma(g0, bc(rdx), d3), d1 = vfma(g1, bc(rdy), d3), d2 = vfma(g2, bc(rdz), d3);
        const V r0 = vadd(Pxy, Pxz), r1 = vsub(Pyz, Pxy), r2 = vadd(Pxz, Pyz);
        V t0, t1, t2;
        if constexpr (GC) {
          const V te = own(I_GEN), q = vmul(own(I_GCN), bc(qr));
          t0 = vfma(r0, q, vfma(d0, te, own(I_TBN0)));
          t1 = vfma(r1, q, vfma(d1, te, own(I_TBN1)));
          t2 = vfma(vsub(zero, r2), q, vfma(d2, te, own(I_TBN2)));
        } else {
          const V te = bc(two_eta);
          t0 = vfma(r0, bc(qr), vfma(d0, te, own(I_TBN0)));
          t1 = vfma(r1, bc(qr), vfma(d1, te, own(I_TBN1)));
          t2 = vfma(r2, bc(-qr), vfma(d2, te, own(I_TBN2)));
        }
        c0v = vfma(own(I_SON0), bc(bt), vmul(t0, bc(ob)));
        c1v = vfma(own(I_SON1), bc(bt), vmul(t1, bc(ob)));
        c2v = vfma(own(I_SON2), bc(bt), vmul(t2, bc(ob)));
        g1_1 = vsub(above(I_U1), u1);
        M_1 = vadd(vM, S.M.r[qp]);
        N_1 = vN; O_1 = O;
      }
      D_1 = D; E_1 = vE; F_1 = F; G_1 = G; J_1 = J; L_1 = Lz;
    }
    const V vQ = vadd(tsxy, xp<LPR>(tsxy)), vS = vadd(tsyz_1, tsyz);
    S.Q.r[q0] = vQ; S.Sz.r[q0] = vS;
    __syncthreads();

    // every read of plane t's inputs lies behind the second barrier: their
    // stage takes plane t + 2
    if (t + 2 < ke + 2) fetch(t + 2, sl);
    if constexpr (CHK) cp_async_wait_all();   // this thread's own snapshot slots

    // ---- 3. pressure and return at the centres of plane t-1 ----
    V s_1, sxx_1, syy_1, szz_1;
    {
      const V pr = vfma(sop, bc(bp), vmul(vfma(div, bc(-KDt), pb), bc(obp)));
      const V R = vadd(tsxz_1, tsxz);
      const V xy = vadd(vQ, S.Q.r[qp]), xz = vadd(R, xp<LPR>(R)), yz = vadd(vS, S.Sz.r[qp]);
      const V j4 = vfma(yz, yz, vfma(xz, xz, vmul(xy, xy)));        // 16 x the shear part
      const V jn = vfma(c2v, c2v, vfma(c1v, c1v, vmul(c0v, c0v)));  // 2 x the normal part
      const V J2 = vfma(j4, bc((T)0.0625), vmul(jn, bc((T)0.5)));
      V sc1;
      if (frozen) sc1 = ldv(A.s, lev(lc));
      else sc1 = vscale(J2, vfma(pr, bc(Acoef), yc));
      const V n0 = vmul(sc1, c0v), n1 = vmul(sc1, c1v), n2 = vmul(sc1, c2v);
      sxx_1 = vsub(n0, pr); syy_1 = vsub(n1, pr); szz_1 = vsub(n2, pr);
      if (out_col && lc >= kb && lc < ke && zc && gy0 && in_x0(0)) {
        const Off ec = (Off)lc * plane + col;
        // the last pair of a row can lie half outside: its second column stays as it is
        auto stc = [&](T *p, V v) {
          if (N == 1 || in_x0(1)) stv(p, ec, v);
          else p[ec] = el<0>(v);
        };
        stc(A.snn[0], n0); stc(A.snn[1], n1); stc(A.snn[2], n2); stc(A.snp, pr);
        if constexpr (CHK) {   // the centres of the box
          if (!frozen) stc(A.s, sc1);
          const int tid = threadIdx.x;
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            if (!in_x0(E)) return;
            const T p_ = el<E>(pr), a0 = el<E>(n0), a1 = el<E>(n1), a2 = el<E>(n2);
            c_sig = maxt(c_sig, maxt(absv(a0 - p_), maxt(absv(a1 - p_), absv(a2 - p_))));
            c_dtau = maxt(c_dtau, maxt(absv(a0 - el<E>(C.cn[0][tid])),
                                       maxt(absv(a1 - el<E>(C.cn[1][tid])), absv(a2 - el<E>(C.cn[2][tid])))));
            c_dp = maxt(c_dp, absv(p_ - el<E>(C.cp[tid])));
            if (isnan(el<E>(sc1)) || isnan(p_)) c_sig = (T)NAN;
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          stc(A.cn[0], n0); stc(A.cn[1], n1); stc(A.cn[2], n2); stc(A.cp, pr);
        } else if constexpr (GC) {
          if (A.keep_s && !frozen) stc(A.s, sc1);
        }
      }
      s_1 = vmul(sc1, bc(qr));
    }
    const V vU = vadd(s_1, xm<LPR>(s_1)), vV = vadd(s_2, s_1);   // quarter scales over x-1, x / planes t-2, t-1
    S.U.r[q0] = vU; S.Vs.r[q0] = vV; S.syy[sl1].r[q0] = syy_1;
    if (t + 1 < ke + 2) {   // plane t + 1 is needed next
      if (!arrived(sl1, t + 2 < ke + 2)) return false;
    } else {
      __syncthreads();
    }

    // ---- 4. new edge deviators at level t-1 ----
    V nxy_1 = zero, nxz_1 = zero, nyz_1 = zero;
    if (w_edge) {
      // the trials are zero on the walls, and so are these
      nxy_1 = vmul(vadd(vU, S.U.r[qm]), tsxy);
      nxz_1 = vmul(vadd(U_2, vU), tsxz_1);
      nyz_1 = vmul(vadd(vV, S.Vs.r[qm]), tsyz_1);
      if (out_col && lc >= kb && lc < ke) {
        const Off e = (Off)lc * plane + col;
        stv(A.sns[0], e, nxy_1); stv(A.sns[1], e, nxz_1); stv(A.sns[2], e, nyz_1);
        if constexpr (CHK) {
          const int tid = threadIdx.x;
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            if (gi + E > nx || gj > ny || lc > nz) return;   // the staged check's edge points
            const T a0 = el<E>(nxy_1), a1 = el<E>(nxz_1), a2 = el<E>(nyz_1);
            c_sig = maxt(c_sig, maxt(absv(a0), maxt(absv(a1), absv(a2))));
            c_dtau = maxt(c_dtau, maxt(absv(a0 - el<E>(C.cs[0][tid])),
                                       maxt(absv(a1 - el<E>(C.cs[1][tid])), absv(a2 - el<E>(C.cs[2][tid])))));
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          if (gi <= nx && gj <= ny && lc <= nz) {   // zero beyond the last edge
            stv(A.cs[0], e, nxy_1); stv(A.cs[1], e, nxz_1); stv(A.cs[2], e, nyz_1);
          }
        }
      }
      S.nxy[sl1].r[q0] = nxy_1; S.nyz[sl1].r[q0] = nyz_1;
    }

    // ---- 5. residual and velocity update of plane t-2 ----
    if (w_vel) {
      const int lu = t - 2;
      const V sxx_2_xm = xm<LPR>(sxx_2), nxy_2_xp = xp<LPR>(nxy_2), nxz_2_xp = xp<LPR>(nxz_2);
      if (out_col && lu >= kb && lu < ke) {
        const V nxy_2_yp = S.nxy[sl].r[qp], syy_2_ym = S.syy[sl].r[qm];
        const V nyz_2_yp = S.nyz[sl].r[qp];
        const Off e = (Off)lu * plane + col;
        const V vx = bc(rdx), vy = bc(rdy), vz = bc(rdz);
        const V R0 = vfma(vsub(nxz_1, nxz_2), vz, vfma(vsub(nxy_2_yp, nxy_2), vy, vmul(vsub(sxx_2, sxx_2_xm), vx)));
        const V R1 = vfma(vsub(nyz_1, nyz_2), vz, vfma(vsub(nxy_2_xp, nxy_2), vx, vmul(vsub(syy_2, syy_2_ym), vy)));
        const V R2 = vfma(vsub(nyz_2_yp, nyz_2), vy, vfma(vsub(nxz_2_xp, nxz_2), vx, vmul(vsub(szz_2, szz_3), vz)));
        // a face off the interior keeps its value
        const bool zu = lu < nz, zw = lu >= 1 && lu <= nz - 1;
        const V un0 = zu ? vfma(R0, st0, u0_2) : u0_2, un1 = zu ? vfma(R1, st1, u1_2) : u1_2;
        const V un2 = zw ? vfma(R2, st2, u2_2) : u2_2;
        stv(A.uo[0], e, un0); stv(A.uo[1], e, un1); stv(A.uo[2], e, un2);
        if constexpr (CHK) {
          const int tid = threadIdx.x;
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            const int x = gi + E;
            const bool x1 = in_x1(E), xl = in_x0(E);
            if (x1 && gy0 && zu) c_r = maxt(c_r, absv(el<E>(R0)));
            if (xl && gy1 && zu) c_r = maxt(c_r, absv(el<E>(R1)));
            if (xl && gy0 && zw) c_r = maxt(c_r, absv(el<E>(R2)));
            // |v0 + u|: a NaN in u also reaches c_du
            if (x <= nx && gj < ny && lu < nz) {
              c_du = maxt(c_du, absv(el<E>(un0) - el<E>(C.uchk[0][tid])));
              c_vm = fmax(c_vm, fabs(C.v0[0][N * tid + E] + (double)el<E>(u0_2)));
            }
            if (x < nx && gj <= ny && lu < nz) {
              c_du = maxt(c_du, absv(el<E>(un1) - el<E>(C.uchk[1][tid])));
              c_vm = fmax(c_vm, fabs(C.v0[1][N * tid + E] + (double)el<E>(u1_2)));
            }
            if (x < nx && gj < ny && lu <= nz) {
              c_du = maxt(c_du, absv(el<E>(un2) - el<E>(C.uchk[2][tid])));
              c_vm = fmax(c_vm, fabs(C.v0[2][N * tid + E] + (double)el<E>(u2_2)));
            }
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          // off a location's extent u stays zero, and so does its snapshot
          stv(A.uchk[0], e, un0); stv(A.uchk[1], e, un1); stv(A.uchk[2], e, un2);
        }
      }
    }

    // ---- carry this plane's values one plane down ----
    wxy_1 = wxy;
    tsxz_1 = tsxz; tsyz_1 = tsyz;
    s_2 = s_1; U_2 = vU;
    sxx_2 = sxx_1; syy_2 = syy_1; szz_3 = szz_2; szz_2 = szz_1;
    nxy_2 = nxy_1; nxz_2 = nxz_1; nyz_2 = nyz_1;
    return true;
  };
  int t = kb - 2;
  for (; t + 1 < ke + 2; t += 2) {
    if (!plane_step(t, std::integral_constant<int, 0>{})) return;
    if (!plane_step(t + 1, std::integral_constant<int, 1>{})) return;
  }
  if (t < ke + 2 && !plane_step(t, std::integral_constant<int, 0>{})) return;
  if constexpr (CHK) {
    block_max_bits((double)c_sig, &di->red[RED_SIG]);
    block_max_bits((double)c_dtau, &di->red[RED_DTAU]);
    block_max_bits((double)c_dp, &di->red[RED_DP]);
    block_max_bits((double)c_r, &di->red[RED_R]);
    block_max_bits((double)c_du, &di->red[RED_DU]);
    block_max_bits(c_vm, &di->red[RED_V]);
  }
}

template <typename L, bool GC, typename Off, bool CHK>
__global__ void __launch_bounds__(L::LPR *L::H, 1)
    k_fused3d_reg(const __grid_constant__ Maps<GC> M, const Args<typename L::T> A, Geo g, const Scal *sc, DevInfo *di, int kz) {
  if (di != nullptr && *(volatile const int *)&di->done != 0) return;
  const bool frozen = di != nullptr && di->frozen;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int i0 = blockIdx.x * OX, j0 = blockIdx.y * (L::H - 4);
  const bool interior = i0 - 2 >= 1 && i0 + WX - 3 <= g.nx - 1 && j0 - 2 >= 1 && j0 + L::H - 3 <= g.ny - 1;
  if (interior) reg_body<L, GC, true, Off, CHK>(M, A, g, sc, di, frozen, kz, smem_raw);
  else reg_body<L, GC, false, Off, CHK>(M, A, g, sc, di, frozen, kz, smem_raw);
}

typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    return ok ? (EncodeTiled)p : nullptr;
  }();
  return fn;
}

// tensor maps of the stage's input arrays: boxes of BX x H x 1, zero outside
template <typename L, bool GC>
bool encode_maps(Maps<GC> *M, const Geo &g, const Stage<typename L::T> &S) {
  using T = typename L::T;
  const T *src[I_COUNT_G] = {S.u[0],   S.u[1],   S.u[2],   S.rq[0],  S.rq[1],  S.rq[2],  S.rd[0],  S.rd[1],
                             S.sos[1], S.sos[2], S.tbs[1], S.tbs[2], S.son[0], S.son[1], S.son[2], S.tbn[0],
                             S.tbn[1], S.tbn[2], S.sos[0], S.tbs[0], S.sop,    S.pb,     S.yc,     S.ge[0],
                             S.gc[0],  S.ge[1],  S.gc[1],  S.ge[2],  S.gc[2],  S.ge[3],  S.gc[3]};
  const EncodeTiled fn = encoder();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)g.px, (cuuint64_t)g.py, (cuuint64_t)g.pz};
  cuuint64_t strides[2] = {(cuuint64_t)g.px * sizeof(T), (cuuint64_t)g.plane * sizeof(T)};
  cuuint32_t box[3] = {(cuuint32_t)BX, (cuuint32_t)L::H, 1}, es[3] = {1, 1, 1};
  for (int k = 0; k < inputs<GC>(); ++k)
    if (fn(&M->m[k], sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3,
           const_cast<T *>(src[k]), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
  return true;
}

template <typename L, bool GC, bool CHK>
constexpr size_t lane_bytes() { return sizeof(SmemR<L, GC>) + (CHK ? sizeof(ChkSlots<L>) : 0); }

template <typename L, bool GC, bool CHK>
cudaError_t configure_lane() {
  const cudaError_t e = cudaFuncSetAttribute(k_fused3d_reg<L, GC, int, CHK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)lane_bytes<L, GC, CHK>());
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(k_fused3d_reg<L, GC, long long, CHK>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)lane_bytes<L, GC, CHK>());
}

// the columns to write: 0 .. nx (the row's padding stays zero)
Geo extent(Geo g) {
  g.px = g.nx + 1;
  return g;
}

template <typename L, bool GC, typename Off, bool CHK>
bool launch_lane(const Stage<typename L::T> &S, const Args<typename L::T> &A, const Geo &g, const Scal *sc, DevInfo *di,
                 int kz, cudaStream_t st) {
  Maps<GC> M;
  if (!encode_maps<L, GC>(&M, g, S)) return false;
  if (kz <= 0) kz = fused3d_kz(extent(g), OX, L::H - 4, 0);
  dim3 grid((g.nx + OX) / OX, (g.py + L::H - 5) / (L::H - 4), (g.pz + kz - 1) / kz);
  k_fused3d_reg<L, GC, Off, CHK><<<grid, L::LPR * L::H, lane_bytes<L, GC, CHK>(), st>>>(M, A, g, sc, di, kz);
  return true;
}

template <typename L, bool GC, bool CHK>
bool launch_off(const Stage<typename L::T> &S, const Args<typename L::T> &A, const Geo &g, const Scal *sc, DevInfo *di,
                int kz, cudaStream_t st) {
  return (long long)g.pz * g.plane < (1LL << 31) ? launch_lane<L, GC, int, CHK>(S, A, g, sc, di, kz, st)
                                                  : launch_lane<L, GC, long long, CHK>(S, A, g, sc, di, kz, st);
}

}  // namespace

// One fused iteration, register z-march flavour: reads buffer b of the
// stage, writes 1 - b.  check (FP32 only): a check iteration, which also
// reduces the stopping measures into di and updates the check snapshots.
// last: the last iteration of a chunk, whose return scales a commit of the
// undecided solve reads (stored with a per-cell modulus).
// Returns false if a tensor map could not be made.
template <typename T>
bool launch_fused3d_reg(const Geo &g, const Stage<T> &S, const Scal *sc, DevInfo *di, int kz, cudaStream_t st,
                        bool check, bool last) {
  Args<T> A;
  for (int d = 0; d < 3; ++d) {
    A.snn[d] = S.snn[d]; A.sns[d] = S.sns[d]; A.uo[d] = S.uo[d];
    A.cn[d] = S.cn[d]; A.cs[d] = S.cs[d]; A.uchk[d] = S.uchk[d]; A.v0[d] = S.v0[d];
  }
  A.snp = S.snp; A.s = S.s; A.keep_s = last; A.cp = S.cp;
  if constexpr (sizeof(T) == 8) {
    return launch_off<LaneD, false, false>(S, A, g, sc, di, kz, st);
  } else if (S.ge[0]) {
    return check ? launch_off<LaneF<16>, true, true>(S, A, g, sc, di, kz, st)
                 : launch_off<LaneF<16>, true, false>(S, A, g, sc, di, kz, st);
  } else if (check) {   // the snapshots' slots take the room of eight rows
    return launch_off<LaneF<16>, false, true>(S, A, g, sc, di, kz, st);
  } else {
    // a plane takes a 16-row block 1.5 us and a 24-row one 2.0 us; the 24 rows write
    // 20 of theirs, the 16 rows 12, but need fewer planes per block where the grid is
    // small (90x40x24 13.0 against 16.6 us a sweep, 63^3 21.2 / 23.4; 127^3 95.8 / 79.5,
    // 383^3 1814 / 1619)
    long long c16 = 0, c24 = 0;
    const int k16 = fused3d_kz(extent(g), OX, 12, kz, 1, &c16), k24 = fused3d_kz(extent(g), OX, 20, kz, 1, &c24);
    if (3 * c16 < 4 * c24) return launch_off<LaneF<16>, false, false>(S, A, g, sc, di, k16, st);
    return launch_off<LaneF<24>, false, false>(S, A, g, sc, di, k24, st);
  }
}

bool fused3d_reg_cell_g_fits(const Geo &g, int kz) {
  constexpr int rows = LaneF<16>::H - 4;
  return (g.py + rows - 1) / rows <= 65535 && (kz <= 0 || (g.pz + kz - 1) / kz <= 65535);
}

cudaError_t fused3d_reg_configure() {
  const cudaError_t e[] = {configure_lane<LaneF<24>, false, false>(), configure_lane<LaneF<16>, false, false>(),
                           configure_lane<LaneF<16>, false, true>(),  configure_lane<LaneF<16>, true, false>(),
                           configure_lane<LaneF<16>, true, true>(),   configure_lane<LaneD, false, false>()};
  for (cudaError_t q : e)
    if (q != cudaSuccess) return q;
  return cudaSuccess;
}

template bool launch_fused3d_reg<float>(const Geo &, const Stage<float> &, const Scal *, DevInfo *, int, cudaStream_t,
                                        bool, bool);
template bool launch_fused3d_reg<double>(const Geo &, const Stage<double> &, const Scal *, DevInfo *, int,
                                         cudaStream_t, bool, bool);

}  // namespace ep
