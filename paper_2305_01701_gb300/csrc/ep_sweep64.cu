// ep_sweep64.cu -- the FP64 sweep of a 3D grid with a uniform shear modulus, as
// five stage kernels.
//
// The same iteration as ep_stages.cu (strain, trial, centre return, edge return,
// velocity; Eqs. A41, A5, A23ssP, A2ssP, A6121lambda, A22S, A22P), every quantity
// computed once per point.  Bound: the FP64 pipe (two operations per clock and
// SM, 1.2 TFLOP/s measured on this part), then launch latency on small grids.
// What these kernels leave out of the general ones, which also serve the physical
// response, FP32 and a per-cell modulus:
//   * the means of the old stress around a vertex/edge do not change within an
//     increment: k_rotation_means forms them once, with every factor of 1/2, 1/4
//     and 1/8 of the rotation terms and their signs folded in (exact powers of
//     two), so that an edge's rotation is three FMAs;
//   * spins and shear rates stay unscaled (w = 2 omega, g = 2 eps);
//   * the divergence is formed once, in the trial, and the normal stresses less
//     the pressure once, in the centre return;
//   * the square root and the division of the return run only where J2 is within
//     rounding of Y^2 or above (elsewhere the scale is exactly 1).
// Measured, an iteration at 127^3: 1129 -> 639 us (156 FP64 operations per cell are
// 506 us of the pipe).  A warp covers 32 points along x; blocks hold as many rows as leave every SM some (launch_rows).
#include <math.h>

#include <algorithm>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"
#include "ep_measures.cuh"

namespace ep {

namespace {

struct Pt {
  int i, j, k;
  long long e;
};
// o: the row block and the plane that a launch starts at (launch_parts)
__device__ __forceinline__ Pt point(const Geo &g, int2 o) {
  Pt p;
  p.i = blockIdx.x * 32 + threadIdx.x;
  p.j = (o.x + blockIdx.y) * blockDim.y + threadIdx.y;
  p.k = o.y + blockIdx.z;
  p.e = ((long long)p.k * g.py + p.j) * g.px + p.i;
  return p;
}

// ---- spins, shear rates and rotation products at vertices / edges ------------
__global__ void __launch_bounds__(256) k64_strain(Geo g, int2 o, Stage<double> S, DevInfo *di) {
  if (skip(di)) return;
  const Pt q = point(g, o);
  const int i = q.i, j = q.j, k = q.k, nx = g.nx, ny = g.ny, nz = g.nz;
  if (i > nx || j > ny) return;
  const long long e = q.e, px = g.px, pl = g.plane;
  const bool x1 = i > 0 && i < nx, y1 = j > 0 && j < ny, z1 = k > 0 && k < nz;
  const double u0 = S.u[0][e], u1 = S.u[1][e], u2 = S.u[2][e];
  const auto edge = [&](int c, bool in, double a, double a_m, double ra, double b, double b_m, double rb) {
    double gs = 0.0, w = 0.0, p = 0.0;
    if (in) {
      const double x = (a - a_m) * ra, y = b - b_m;
      gs = fma(y, rb, x);
      w = fma(y, -rb, x);
      p = S.rq[c][e] * w;
    }
    S.es[c][e] = gs;
    S.om[c][e] = w;
    S.pr[c][e] = p;
  };
  const bool in0 = k < nz && x1 && y1;
  edge(0, in0, u0, in0 ? S.u[0][e - px] : 0.0, g.rdy, u1, in0 ? S.u[1][e - 1] : 0.0, g.rdx);
  const bool in1 = j < ny && x1 && z1, in2 = i < nx && y1 && z1;
  edge(1, in1, u0, in1 ? S.u[0][e - pl] : 0.0, g.rdz, u2, in1 ? S.u[2][e - 1] : 0.0, g.rdx);
  edge(2, in2, u1, in2 ? S.u[1][e - pl] : 0.0, g.rdz, u2, in2 ? S.u[2][e - px] : 0.0, g.rdy);
}

// ---- relaxed trials -------------------------------------------------------------
__global__ void __launch_bounds__(256) k64_trial(Geo g, int2 o, Stage<double> S, const Scal *sc, DevInfo *di) {
  if (skip(di)) return;
  const Pt q = point(g, o);
  const int i = q.i, j = q.j, k = q.k, nx = g.nx, ny = g.ny, nz = g.nz;
  if (i > nx || j > ny) return;
  const long long e = q.e, px = g.px, pl = g.plane;
  const double two_eta = sc->two_eta, eta = 0.5 * two_eta, bt = sc->bt, ob = 1.0 - bt;
  if (i < nx && j < ny && k < nz) {
    const double d0 = S.u[0][e + 1] - S.u[0][e], d1 = S.u[1][e + px] - S.u[1][e], d2 = S.u[2][e + pl] - S.u[2][e];
    // the rate e - div / 3 rounded once, then scaled
    const double div = fma(d2, g.rdz, fma(d1, g.rdy, d0 * g.rdx)), d3 = div * (-1.0 / 3.0);
    const double *p0 = S.pr[0];
    const double xy = (p0[e] + p0[e + 1]) + (p0[e + px] + p0[e + px + 1]);
    const double *p1 = S.pr[1], *p2 = S.pr[2];
    const double xz = (p1[e] + p1[e + 1]) + (p1[e + pl] + p1[e + pl + 1]);
    const double yz = (p2[e] + p2[e + px]) + (p2[e + pl] + p2[e + pl + px]);
    const double t0 = fma(0.25, xy + xz, fma(two_eta, fma(d0, g.rdx, d3), S.tbn[0][e]));
    const double t1 = fma(0.25, yz - xy, fma(two_eta, fma(d1, g.rdy, d3), S.tbn[1][e]));
    const double t2 = fma(-0.25, xz + yz, fma(two_eta, fma(d2, g.rdz, d3), S.tbn[2][e]));
    S.Tn[0][e] = fma(bt, S.son[0][e], ob * t0);
    S.Tn[1][e] = fma(bt, S.son[1][e], ob * t1);
    S.Tn[2][e] = fma(bt, S.son[2][e], ob * t2);
    S.dv[e] = div;
  }
  const bool x1 = i > 0 && i < nx, y1 = j > 0 && j < ny, z1 = k > 0 && k < nz;
  // spins summed over the four neighbours of another orientation
  const double *w0 = S.om[0], *w1 = S.om[1], *w2 = S.om[2];
  const auto edge = [&](int c, double wa, double wb) {
    const double tr = fma(S.om[c][e], S.md[c][e],
                          fma(wa, S.ma[c][e], fma(wb, S.mb[c][e], fma(eta, S.es[c][e], S.tbs[c][e]))));
    return fma(bt, S.sos[c][e], ob * tr);
  };
  double v = 0.0;
  if (k < nz && x1 && y1)
    v = edge(0, (w1[e - px] + w1[e]) + (w1[e - px + pl] + w1[e + pl]), (w2[e - 1] + w2[e]) + (w2[e - 1 + pl] + w2[e + pl]));
  S.Ts[0][e] = v;
  v = 0.0;
  if (j < ny && x1 && z1)
    v = edge(1, (w0[e - pl] + w0[e - pl + px]) + (w0[e] + w0[e + px]), (w2[e - 1] + w2[e]) + (w2[e - 1 + px] + w2[e + px]));
  S.Ts[1][e] = v;
  v = 0.0;
  if (i < nx && y1 && z1)
    v = edge(2, (w1[e - px] + w1[e - px + 1]) + (w1[e] + w1[e + 1]), (w0[e - pl] + w0[e - pl + 1]) + (w0[e] + w0[e + 1]));
  S.Ts[2][e] = v;
}

// ---- pressure and return at centres ------------------------------------------------
template <bool CHK>
__global__ void __launch_bounds__(256) k64_centres(Geo g, int2 o, Stage<double> S, const Scal *sc, DevInfo *di) {
  if (skip(di)) return;
  const Pt q = point(g, o);
  const long long e = q.e, px = g.px, pl = g.plane;
  const bool frozen = di != nullptr && di->frozen;
  double sig = 0.0, dtau = 0.0, dp = 0.0;
  if (q.i < g.nx && q.j < g.ny && q.k < g.nz) {
    const double p = fma(sc->bp, S.sop[e], sc->obp * fma(-sc->KDt, S.dv[e], S.pb[e]));
    const double *t0 = S.Ts[0];
    double tn[3] = {S.Tn[0][e], S.Tn[1][e], S.Tn[2][e]};
    const double *t1 = S.Ts[1], *t2 = S.Ts[2];
    const double xy = (t0[e] + t0[e + 1]) + (t0[e + px] + t0[e + px + 1]);
    const double xz = (t1[e] + t1[e + 1]) + (t1[e + pl] + t1[e + pl + 1]);
    const double yz = (t2[e] + t2[e + px]) + (t2[e + pl] + t2[e + pl + px]);
    const double j4 = fma(yz, yz, fma(xz, xz, xy * xy)), jn = fma(tn[2], tn[2], fma(tn[1], tn[1], tn[0] * tn[0]));
    double s = 1.0;
    if (frozen) {
      s = S.s[e];   // frozen plasticity: the held scale (Sec. 3.3)
    } else {
      s = scale_of(fma(0.0625, j4, 0.5 * jn), fma(sc->A, p, S.yc[e]));
      S.s[e] = s;
    }
    S.snp[e] = p;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double t = s * tn[d], sx = t - p;
      S.snn[d][e] = t;
      S.sx[d][e] = sx;
      if (CHK) {
        sig = maxn(sig, fabs(sx));
        dtau = maxn(dtau, fabs(t - S.cn[d][e]));
        S.cn[d][e] = t;
      }
    }
    if (CHK) {
      dp = fabs(p - S.cp[e]);
      S.cp[e] = p;
      if (isnan(s) || isnan(p)) sig = NAN;
    }
  }
  if (CHK && di) {
    block_max(sig, &di->red[RED_SIG]);
    block_max(dtau, &di->red[RED_DTAU]);
    block_max(dp, &di->red[RED_DP]);
  }
}

// ---- new deviators at vertices / edges ------------------------------------------------
template <bool CHK>
__global__ void __launch_bounds__(256) k64_edges(Geo g, int2 o, Stage<double> S, DevInfo *di) {
  if (skip(di)) return;
  const Pt q = point(g, o);
  const int i = q.i, j = q.j, k = q.k, nx = g.nx, ny = g.ny, nz = g.nz;
  const long long e = q.e, px = g.px, pl = g.plane;
  double sig = 0.0, dtau = 0.0;
  if (i <= nx && j <= ny) {
    const double *s = S.s;
    const bool x1 = i > 0 && i < nx, y1 = j > 0 && j < ny, z1 = k > 0 && k < nz;
    double v[3] = {0.0, 0.0, 0.0};
    if (k < nz && x1 && y1)
      v[0] = (s[e - px - 1] + s[e - px] + s[e - 1] + s[e]) * (0.25 * S.Ts[0][e]);
    if (j < ny && x1 && z1) v[1] = (s[e - pl - 1] + s[e - pl] + s[e - 1] + s[e]) * (0.25 * S.Ts[1][e]);
    if (i < nx && y1 && z1) v[2] = (s[e - pl - px] + s[e - pl] + s[e - px] + s[e]) * (0.25 * S.Ts[2][e]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      S.sns[c][e] = v[c];
      if (CHK) {
        sig = maxn(sig, fabs(v[c]));
        dtau = maxn(dtau, fabs(v[c] - S.cs[c][e]));
        S.cs[c][e] = v[c];
      }
    }
  }
  if (CHK && di) {
    block_max(sig, &di->red[RED_SIG]);
    block_max(dtau, &di->red[RED_DTAU]);
  }
}

// ---- residual and velocity update ---------------------------------------------------------
template <bool CHK>
__global__ void __launch_bounds__(256) k64_velocity(Geo g, int2 o, Stage<double> S, const Scal *sc, DevInfo *di) {
  if (skip(di)) return;
  const Pt q = point(g, o);
  const int i = q.i, j = q.j, k = q.k, nx = g.nx, ny = g.ny, nz = g.nz;
  const long long e = q.e, px = g.px, pl = g.plane;
  const double vs = sc->vstep;
  double rmax = 0.0, du = 0.0, vm = 0.0;
  if (i <= nx && j <= ny) {
    // face d: in = inside its extent, in1 = off the walls
    const auto face = [&](int d, bool in, bool in1, double R) {
      const double u = S.u[d][e];
      double un = u;
      if (in1) {
        if (S.f[d]) R += S.f[d][e];
        un = fma(vs, R, u);
        if (CHK) rmax = maxn(rmax, fabs(R));
      }
      S.uo[d][e] = un;
      if (CHK && in) {
        du = maxn(du, fabs(un - S.uchk[d][e]));
        vm = maxn(vm, fabs(S.v0[d][e] + u));
        S.uchk[d][e] = un;
      }
    };
    const bool kc = k < nz;
    const bool ix = j < ny && kc, iy = i < nx && kc, x1 = ix && i > 0 && i < nx, y1 = iy && j > 0 && j < ny;
    double R = 0.0;
    if (x1) {
      R = fma(S.sns[0][e + px] - S.sns[0][e], g.rdy, (S.sx[0][e] - S.sx[0][e - 1]) * g.rdx);
      R = fma(S.sns[1][e + pl] - S.sns[1][e], g.rdz, R);
    }
    face(0, ix, x1, R);
    if (y1) {
      R = fma(S.sns[0][e + 1] - S.sns[0][e], g.rdx, (S.sx[1][e] - S.sx[1][e - px]) * g.rdy);
      R = fma(S.sns[2][e + pl] - S.sns[2][e], g.rdz, R);
    }
    face(1, iy, y1, R);
    const bool iz = i < nx && j < ny, z1 = iz && k > 0 && k < nz;
    if (z1)
      R = fma(S.sns[2][e + px] - S.sns[2][e], g.rdy,
              fma(S.sns[1][e + 1] - S.sns[1][e], g.rdx, (S.sx[2][e] - S.sx[2][e - pl]) * g.rdz));
    face(2, iz, z1, R);
  }
  if (CHK && di) {
    block_max(rmax, &di->red[RED_R]);
    block_max(du, &di->red[RED_DU]);
    block_max(vm, &di->red[RED_V]);
  }
}

// ---- the rotation's coefficients at vertices / edges, once per increment -------------------
// md: of the edge's own w; ma, mb: of the summed w of the two other orientations
// (w = 2 omega; sums of four).  rq = c2 dt tau_hat at edges, rd = c2 dt (tyy - txx),
// c2 dt (tzz - txx) at centres.
__global__ void __launch_bounds__(256) k_rotation_means(Geo g, int2 o, Stage<double> S, double *md0, double *md1,
                                                        double *md2, double *ma0, double *ma1, double *ma2,
                                                        double *mb0, double *mb1, double *mb2) {
  const Pt q = point(g, o);
  const int i = q.i, j = q.j, k = q.k, nx = g.nx, ny = g.ny, nz = g.nz;
  if (i > nx || j > ny) return;
  const long long e = q.e, px = g.px, pl = g.plane;
  const bool x1 = i > 0 && i < nx, y1 = j > 0 && j < ny, z1 = k > 0 && k < nz;
  const double *rd0 = S.rd[0], *rd1 = S.rd[1], *q0 = S.rq[0], *q1 = S.rq[1], *q2 = S.rq[2];
  if (k < nz && x1 && y1) {
    md0[e] = 0.125 * (rd0[e - px - 1] + rd0[e - px] + rd0[e - 1] + rd0[e]);
    // + Tyz Wxz + Txz Wyz
    ma0[e] = 0.03125 * (q2[e - 1] + q2[e] + q2[e - 1 + pl] + q2[e + pl]);
    mb0[e] = 0.03125 * (q1[e - px] + q1[e] + q1[e - px + pl] + q1[e + pl]);
  }
  if (j < ny && x1 && z1) {   // + Tyz Wxy - Txy Wyz
    md1[e] = 0.125 * (rd1[e - pl - 1] + rd1[e - pl] + rd1[e - 1] + rd1[e]);
    ma1[e] = 0.03125 * (q2[e - 1] + q2[e] + q2[e - 1 + px] + q2[e + px]);
    mb1[e] = -0.03125 * (q0[e - pl] + q0[e - pl + px] + q0[e] + q0[e + px]);
  }
  if (i < nx && y1 && z1) {   // - Txy Wxz - Txz Wxy
    md2[e] = 0.125 * ((rd1[e - pl - px] - rd0[e - pl - px]) + (rd1[e - pl] - rd0[e - pl]) +
                      (rd1[e - px] - rd0[e - px]) + (rd1[e] - rd0[e]));
    ma2[e] = -0.03125 * (q0[e - pl] + q0[e - pl + 1] + q0[e] + q0[e + 1]);
    mb2[e] = -0.03125 * (q1[e - px] + q1[e - px + 1] + q1[e] + q1[e + 1]);
  }
}

// rows per block: 8 where that leaves four blocks per SM (152), fewer on smaller
// grids
dim3 launch_rows(const Geo &g, dim3 *block) {
  const int bx = (g.nx + 32) / 32;   // points 0 .. nx
  int rows = 8;
  while (rows > 1 && (long long)bx * ((g.py + rows - 1) / rows) * g.pz < 608) rows /= 2;
  *block = dim3(32, rows);
  return dim3(bx, (g.py + rows - 1) / rows, g.pz);
}

// go(grid, offset) for a grid of row blocks and planes, cut where it is longer than a
// launch can be
template <typename F>
void launch_parts(dim3 gr, F go) {
  constexpr unsigned most = 65535;
  for (unsigned z = 0; z < gr.z; z += most)
    for (unsigned y = 0; y < gr.y; y += most)
      go(dim3(gr.x, std::min(most, gr.y - y), std::min(most, gr.z - z)), make_int2((int)y, (int)z));
}

}  // namespace

void launch_sweep64(const Geo &g, const Stage<double> &S, const Scal *sc, DevInfo *di, bool check, cudaStream_t st,
                   const cudaEvent_t *ev) {
  dim3 bl;
  const dim3 all = launch_rows(g, &bl);
  int stage = 0;
  auto run = [&](auto go) {
    launch_parts(all, go);
    ++stage;
    if (ev) cudaEventRecord(ev[stage], st);
  };
  run([&](dim3 gr, int2 o) { k64_strain<<<gr, bl, 0, st>>>(g, o, S, di); });
  run([&](dim3 gr, int2 o) { k64_trial<<<gr, bl, 0, st>>>(g, o, S, sc, di); });
  run([&](dim3 gr, int2 o) {
    if (check) k64_centres<true><<<gr, bl, 0, st>>>(g, o, S, sc, di);
    else k64_centres<false><<<gr, bl, 0, st>>>(g, o, S, sc, di);
  });
  run([&](dim3 gr, int2 o) {
    if (check) k64_edges<true><<<gr, bl, 0, st>>>(g, o, S, di);
    else k64_edges<false><<<gr, bl, 0, st>>>(g, o, S, di);
  });
  run([&](dim3 gr, int2 o) {
    if (check) k64_velocity<true><<<gr, bl, 0, st>>>(g, o, S, sc, di);
    else k64_velocity<false><<<gr, bl, 0, st>>>(g, o, S, sc, di);
  });
}

void launch_rotation_means(const Geo &g, const Stage<double> &S, double *const md[3], double *const ma[3],
                           double *const mb[3], cudaStream_t st) {
  dim3 bl;
  const dim3 all = launch_rows(g, &bl);
  launch_parts(all, [&](dim3 gr, int2 o) {
    k_rotation_means<<<gr, bl, 0, st>>>(g, o, S, md[0], md[1], md[2], ma[0], ma[1], ma[2], mb[0], mb[1], mb[2]);
  });
}

}  // namespace ep
