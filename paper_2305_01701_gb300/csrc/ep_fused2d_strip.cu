// ep_fused2d_strip.cu -- the batched 2D iteration with one warp per strip.
//
// Same arithmetic as ep_fused2d.cu (vertex spin and strain rate, relaxed
// trials at vertices and centres with the Jaumann term, pressure and
// Drucker-Prager return at centres, vertex deviators, momentum residual and
// velocity update; Eqs. A41, A5, A23ssP, A2ssP, A61, A6121lambda, A22S,
// A22P), mapped without shared memory or block barriers:
//   * a work item is (instance, strip of columns, segment of `seg` rows).  FP32: a
//     thread owns two adjacent columns as one float2 and the warp covers 64
//     (60 written); FP64: one column, 32 (28 written);
//   * the warp marches the rows y = j0 - 2 .. j1 + 1 of its segment: at row
//     t it forms the vertex quantities of row t, the centres of row t - 1,
//     the vertex deviators of row t - 1 and the velocities of row t - 2;
//   * x +- 1 neighbours are warp shuffles (of pair sums where a mean of four
//     allows), y - 1 neighbours are registers carried from the previous row;
//     inputs are loaded one row ahead;
//   * check iterations reduce the residual norms per warp (one atomic per
//     warp, item and norm).
// The deviatoric rate e - div / 3 is rounded once and scaled after (2 eta e and -2 eta div / 3
// as two terms round each at the size of the larger); its two registers more would leave an
// SM three FP32 blocks (519 us a sweep), so the compiler is held to 128.
// Warps take items independently, so a block never waits for another warp.
// 256 grids of 127^2 .. 511^2, one sweep: FP32 is bound by the 20 arrays it
// moves, 464 us (5.6 TB/s; one column a thread and two rows ahead: 773 us; two
// columns and two rows ahead 168 registers, 12 warps an SM: 511 us, at 128
// registers with spills 638 us); FP64 (64 grids) by the FP64 pipe.
#include <math.h>

#include <type_traits>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"

namespace ep {

namespace {

constexpr int SWARPS = 4;       // warps per block
constexpr unsigned FULL = 0xffffffffu;

template <typename T>
struct Strip;
template <>
struct Strip<float> {
  using V = float2;
  static constexpr int N = 2;
};
template <>
struct Strip<double> {
  using V = double;
  static constexpr int N = 1;
};

template <typename T>
__device__ __forceinline__ T maxt(T a, T b) { return (a > b || a != a) ? a : b; }
// |a - b|, formed in FP64
__device__ __forceinline__ double gap(double a, double b) { return fabs(a - b); }

// warp-wide max of |v| (NaN kept: its bit pattern is above +inf), one atomic
__device__ __forceinline__ void warp_max(double v, unsigned long long *slot) {
  unsigned long long x = (unsigned long long)__double_as_longlong(fabs(v));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(FULL, x, o);
    x = x > w ? x : w;
  }
  if ((threadIdx.x & 31) == 0 && x) atomicMax(slot, x);
}

template <typename T, bool CHK>
__global__ void __launch_bounds__(32 * SWARPS, sizeof(T) == 4 && !CHK ? 4 : 0)
    k_fused2d_strip(const Inst2<T> *insts, const int4 *items, int n_items, int b, int seg) {
  using V = typename Strip<T>::V;
  constexpr int N = Strip<T>::N, SW = 32 * N, SO = SW - 4;   // columns covered and written
  const int a = threadIdx.x & 31;
  const int warps = gridDim.x * SWARPS;
  const int o = 1 - b;
  auto bc = [](T v) -> V { return Splat<V>::of(v); };
  const V zero = bc((T)0);
  for (int it = blockIdx.x * SWARPS + (threadIdx.x >> 5); it < n_items; it += warps) {
    const int4 item = items[it];
    const Inst2<T> &I = insts[item.x];
    if (*(volatile const int *)&I.di->done != 0) continue;   // uniform per warp
    const bool frozen = I.di->frozen != 0;
    const Geo &g = I.g;
    const SweepScal<T> &Q = sweep_scal<T>(I.sc);
    const int nx = g.nx, ny = g.ny, px = g.px, py = g.py;
    const int i0 = item.y * SO, j0 = item.z * seg, j1 = min(j0 + seg, py);
    const int gi = i0 - 2 + N * a;   // first column of the thread
    // x1: an interior vertex line; x0: a centre.  What the strip's outermost
    // columns compute is never read by a written one.
    auto in_x1 = [&](int e) { return gi + e >= 1 && gi + e <= nx - 1; };
    auto in_x0 = [&](int e) { return gi + e >= 0 && gi + e < nx; };
    auto mask = [](bool e0, bool e1, T v) -> V {
      if constexpr (N == 2) return make_float2(e0 ? v : (T)0, e1 ? v : (T)0);
      else return e0 ? v : (T)0;
    };
    const bool out = N * a >= 2 && N * a < SW - 2 && gi >= 0 && gi < px;   // px is a multiple of N
    const V m1 = mask(in_x1(0), in_x1(1), (T)1);
    const V stx = mask(in_x1(0), in_x1(1), Q.vstep), sty = mask(in_x0(0), in_x0(1), Q.vstep);
    const V rdx = bc(Q.rdx), rdy = bc(Q.rdy), nrdx = bc(-Q.rdx), bt = bc(Q.bt), ob = bc(Q.ob);
    const V eta = bc(Q.eta), two_eta = bc(Q.two_eta), m3 = bc((T)(-1.0 / 3.0)), qr = bc((T)0.25);
    const T *u0 = I.u[b][0], *u1 = I.u[b][1];
    // loads read the nearest in-box columns and row without a test: a value
    // outside the box only ever enters masked expressions.  A 2D box that fits
    // the device has fewer than 2^31 points.
    const int gic = min(max(gi, 0), px - N);
    auto ld = [&](const T *p, int e) -> V { return *reinterpret_cast<const V *>(p + e); };
    auto st = [&](T *p, int e, V v) { *reinterpret_cast<V *>(p + e) = v; };

    // inputs one row ahead (vertex / face arrays of row r, centre arrays of
    // row r - 1): `next` holds row t + 1
    struct Row {
      V vx, vy, rq, rd, tbs, ss, tbn0, tbn1, sn0, sn1, sp, pb, yc;
    };
    auto load_row = [&](int r, Row &w) {
      const int e = min(max(r, 0), py - 1) * px + gic, c = min(max(r - 1, 0), py - 1) * px + gic;
      w.vx = ld(u0, e); w.vy = ld(u1, e); w.rq = ld(I.rq, e); w.rd = ld(I.rd, e);
      w.tbs = ld(I.tbs, e); w.ss = ld(I.ss[b], e);
      w.tbn0 = ld(I.tbn[0], c); w.tbn1 = ld(I.tbn[1], c); w.sn0 = ld(I.sn[b][0], c); w.sn1 = ld(I.sn[b][1], c);
      w.sp = ld(I.sp[b], c); w.pb = ld(I.pb, c); w.yc = ld(I.yc, c);
    };
    Row next;

    // row history (suffix _1: row t - 1, _2: row t - 2, _3: row t - 3)
    V vx = zero, vy = zero, vx_1 = zero, vy_1 = zero, vx_2 = zero, vy_2 = zero, rd = zero;
    V P = zero, ts = zero, s_1 = zero, sxx_1 = zero, syy_1 = zero, syy_2 = zero, nxy_1 = zero;
    double sig = 0.0, dtau = 0.0, dp = 0.0, rmax = 0.0, du = 0.0, vm = 0.0;   // the stopping measures, in FP64

    load_row(j0 - 2, next);
    for (int t = j0 - 2; t < j1 + 2; ++t) {
      const int c = t - 1, u = t - 2;
      vx_2 = vx_1; vy_2 = vy_1; vx_1 = vx; vy_1 = vy;
      const V rd_1 = rd, P_1 = P, ts_1 = ts, s_2 = s_1, sxx_2 = sxx_1, syy_3 = syy_2, nxy_2 = nxy_1;
      syy_2 = syy_1;
      vx = next.vx; vy = next.vy; rd = next.rd;
      const V rq = next.rq, tbs = next.tbs, ssv = next.ss;
      const V tbn0 = next.tbn0, tbn1 = next.tbn1, sn0 = next.sn0, sn1 = next.sn1, sp = next.sp, pb = next.pb,
              yc = next.yc;
      if (t + 1 < j1 + 2) load_row(t + 1, next);

      // ---- vertex (gi, t): shear rate g = 2 eps, spin w = 2 omega, relaxed trial ----
      const V J = vadd(rd_1, rd);
      const V x = vmul(vsub(vx, vx_1), rdy), y = vsub(vy, xm<32>(vy));
      const V w = vmul(m1, vfma(y, nrdx, x));
      const V dyx = vadd(J, xm<32>(J));
      const V tr = vfma(vmul(w, dyx), bc((T)0.125), vfma(vfma(y, rdx, x), eta, tbs));
      ts = vmul(m1, vfma(ssv, bt, vmul(tr, ob)));
      P = vmul(rq, w);
      if (t < 1 || t > ny - 1) { ts = zero; P = zero; }   // walls

      // ---- centre (gi, t - 1): relaxed trial, pressure, return ----
      const V Pc = vadd(P_1, P), tc = vadd(ts_1, ts);
      const V xy = vadd(Pc, xp<32>(Pc)), txy = vadd(tc, xp<32>(tc));
      const V ux = vsub(xp<32>(vx_1), vx_1), uy = vsub(vy, vy_1);
      const V div = vfma(uy, rdy, vmul(ux, rdx)), d3 = vmul(div, m3), d0 = vfma(ux, rdx, d3), d1 = vfma(uy, rdy, d3);
      const V q = vmul(xy, qr);
      const V t0 = vadd(vfma(d0, two_eta, tbn0), q), t1 = vsub(vfma(d1, two_eta, tbn1), q);
      const V c0 = vfma(sn0, bt, vmul(t0, ob)), c1 = vfma(sn1, bt, vmul(t1, ob));
      const V pr = vfma(sp, bc(Q.bp), vmul(vfma(div, bc(-Q.KDt), pb), bc(Q.obp)));
      const bool row_c = c >= 0 && c < ny, own_c = out && c >= j0 && c < j1;
      if (frozen) {   // frozen plasticity: the held scale (Sec. 3.3)
        s_1 = ld(I.s, min(max(c, 0), py - 1) * px + gic);
      } else {
        const V J2 = vfma(vmul(txy, txy), bc((T)0.0625), vmul(vfma(c1, c1, vmul(c0, c0)), bc((T)0.5)));
        s_1 = vscale(J2, vfma(pr, bc(Q.A), yc));
      }
      const V n0 = vmul(s_1, c0), n1 = vmul(s_1, c1);
      sxx_1 = vsub(n0, pr);
      syy_1 = vsub(n1, pr);
      if (own_c && row_c && in_x0(0)) {
        const int e = c * px + gi;
        // the last pair of a row can lie half outside: its second column stays as it is
        auto stc = [&](T *p, V v) {
          if (N == 1 || in_x0(1)) st(p, e, v);
          else p[e] = el<0>(v);
        };
        stc(I.sn[o][0], n0); stc(I.sn[o][1], n1); stc(I.sp[o], pr);
        if (!frozen) stc(I.s, s_1);
        if constexpr (CHK) {
          const V k0 = ld(I.cn[0], e), k1 = ld(I.cn[1], e), kp = ld(I.cp, e);
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            if (!in_x0(E)) return;
            sig = maxt(sig, maxt(fabs((double)el<E>(sxx_1)), fabs((double)el<E>(syy_1))));
            dtau = maxt(dtau, maxt(gap(el<E>(n0), el<E>(k0)), gap(el<E>(n1), el<E>(k1))));
            dp = maxt(dp, gap(el<E>(pr), el<E>(kp)));
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          stc(I.cn[0], n0); stc(I.cn[1], n1); stc(I.cp, pr);
        }
      }

      // ---- vertex (gi, t - 1): deviator from the mean of its centre scales ----
      const V h = vadd(s_2, s_1);
      nxy_1 = vmul(vmul(vadd(h, xm<32>(h)), qr), ts_1);   // the trial is zero on the walls
      if (own_c) {   // rows below py
        const int e = c * px + gi;
        st(I.ss[o], e, nxy_1);
        if constexpr (CHK) {
          const V k = ld(I.cs, e);
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            sig = maxt(sig, fabs((double)el<E>(nxy_1)));
            dtau = maxt(dtau, gap(el<E>(nxy_1), el<E>(k)));
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          st(I.cs, e, nxy_1);
        }
      }

      // ---- faces (gi, t - 2): residual and velocity update ----
      const V sxx_2_xm = xm<32>(sxx_2), nxy_2_xp = xp<32>(nxy_2);
      if (out && u >= j0 && u < j1) {
        const int e = u * px + gi;
        const V R0 = vfma(vsub(nxy_1, nxy_2), rdy, vmul(vsub(sxx_2, sxx_2_xm), rdx));
        const V R1 = vfma(vsub(nxy_2_xp, nxy_2), rdx, vmul(vsub(syy_2, syy_3), rdy));
        const bool ux = u < ny, uy = u >= 1 && u <= ny - 1;
        const V un0 = ux ? vfma(R0, stx, vx_2) : vx_2, un1 = uy ? vfma(R1, sty, vy_2) : vy_2;
        st(I.u[o][0], e, un0);
        st(I.u[o][1], e, un1);
        if constexpr (CHK) {
          const V k0 = ld(I.uchk[0], e), k1 = ld(I.uchk[1], e);
          auto one = [&](auto ic) {
            constexpr int E = decltype(ic)::value;
            if (ux && in_x1(E)) rmax = maxt(rmax, fabs((double)el<E>(R0)));
            if (uy && in_x0(E)) rmax = maxt(rmax, fabs((double)el<E>(R1)));
            if (gi + E <= nx && u < ny) {
              du = maxt(du, gap(el<E>(un0), el<E>(k0)));
              vm = maxt(vm, fabs(I.v0[0][e + E] + (double)el<E>(vx_2)));
            }
            if (gi + E < nx && u <= ny) {
              du = maxt(du, gap(el<E>(un1), el<E>(k1)));
              vm = maxt(vm, fabs(I.v0[1][e + E] + (double)el<E>(vy_2)));
            }
          };
          one(std::integral_constant<int, 0>{});
          if constexpr (N == 2) one(std::integral_constant<int, 1>{});
          st(I.uchk[0], e, un0);   // off a location's extent u and its snapshot stay zero
          st(I.uchk[1], e, un1);
        }
      }
    }
    if constexpr (CHK) {
      warp_max(sig, &I.di->red[RED_SIG]);
      warp_max(dtau, &I.di->red[RED_DTAU]);
      warp_max(dp, &I.di->red[RED_DP]);
      warp_max(rmax, &I.di->red[RED_R]);
      warp_max(du, &I.di->red[RED_DU]);
      warp_max(vm, &I.di->red[RED_V]);
    }
  }
}

}  // namespace

int fused2d_strip_columns(size_t elem) { return elem == 4 ? 60 : 28; }

template <typename T>
void launch_fused2d_strip(int seg, const Inst2<T> *insts, const int4 *items, int n_items, int b, int check,
                          int blocks, cudaStream_t st) {
  if (check) k_fused2d_strip<T, true><<<blocks, 32 * SWARPS, 0, st>>>(insts, items, n_items, b, seg);
  else k_fused2d_strip<T, false><<<blocks, 32 * SWARPS, 0, st>>>(insts, items, n_items, b, seg);
}

template <typename T>
int fused2d_strip_blocks_per_sm() {
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_fused2d_strip<T, false>, 32 * SWARPS, 0);
  return e == cudaSuccess && nb > 0 ? nb : 1;
}

template void launch_fused2d_strip<float>(int, const Inst2<float> *, const int4 *, int, int, int, int, cudaStream_t);
template void launch_fused2d_strip<double>(int, const Inst2<double> *, const int4 *, int, int, int, int,
                                           cudaStream_t);
template int fused2d_strip_blocks_per_sm<float>();
template int fused2d_strip_blocks_per_sm<double>();

}  // namespace ep
