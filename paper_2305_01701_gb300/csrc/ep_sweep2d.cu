// ep_sweep2d.cu -- the sweep of one 2D grid with a uniform shear modulus, as two
// stage kernels.
//
// The same iteration as ep_stages.cu (Eqs. A41, A5, A23ssP, A2ssP, A6121lambda,
// A22S, A22P).  A vertex's trial needs only its own spin, so the stress kernel
// recomputes the vertices around a centre instead of passing them through memory,
// and the velocity kernel the deviators of the vertices beside a face: two
// launches per iteration where the stages take five.  A warp covers 32 columns
// (31 written, the last one gives its neighbour's values by shuffle) and marches
// `rows` rows, carrying the row's vertices.  The rotation's mean around a vertex
// does not change within an increment and is formed once (k_rotation_mean2d); spins
// and shear rates stay unscaled (w = 2 omega, g = 2 eps).
// Bound: launch and load latency on one grid (a few rows per warp, so that the
// whole chip works on it), the FP64 pipe on large FP64 grids.  Measured, an
// iteration: FP64 64^2 17.2 -> 8.4 us, 511^2 76.5 -> 45.4 us against five stages
// (12.7 and 50.5 us for five stages with the same arithmetic and as many blocks);
// FP32 383 x 191 10.1 -> 9.0 us, 1000 x 700 48.9 -> 22.7 us against one launch of tiles
// in shared memory (warp strips: 35 us).
#include <math.h>

#include <algorithm>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"
#include "ep_measures.cuh"

namespace ep {

namespace {

// row range of this warp
struct Strip {
  int i, j0, j1, lane;
};
__device__ __forceinline__ Strip strip(const Geo &g, int rows) {
  Strip p;
  p.lane = threadIdx.x;
  p.i = blockIdx.x * 31 + threadIdx.x;
  p.j0 = (blockIdx.y * blockDim.y + threadIdx.y) * rows;
  p.j1 = min(p.j0 + rows, g.py);
  return p;
}
template <typename T>
__device__ __forceinline__ T right(T v) { return __shfl_down_sync(0xffffffffu, v, 1); }

template <typename T, bool CHK>
__global__ void __launch_bounds__(128) k_stress2d(Geo g, Stage<T> S, const Scal *sc, DevInfo *di, int rows) {
  if (skip(di)) return;
  const Strip p = strip(g, rows);
  const int i = p.i, nx = g.nx, ny = g.ny;
  const int px = g.px;   // a 2D box has fewer than 2^31 points
  const bool frozen = di != nullptr && di->frozen;
  const SweepScal<T> &Q = sweep_scal<T>(sc);
  const T two_eta = Q.two_eta, eta = Q.eta, bt = Q.bt, ob = Q.ob;
  const T bp = Q.bp, obp = Q.obp, KDt = Q.KDt, Ac = Q.A, rdx = Q.rdx, rdy = Q.rdy;
  const bool x1 = i > 0 && i < nx, own = p.lane < 31 && i <= nx;
  double sig = 0.0, dtau = 0.0, dp = 0.0;   // stopping measures, in FP64
  T u0_m = 0, t_j = 0, p_j = 0;   // x-velocity of the row below; trial and rotation product at row j
  // trial and rotation product of vertex (i, j)
  auto vertex = [&](int j, T u0, T *ts, T *pr) {
    *ts = *pr = 0;
    if (x1 && j > 0 && j < ny) {
      const int e = j * px + i;
      const T x = (u0 - u0_m) * rdy, y = S.u[1][e] - S.u[1][e - 1];
      const T w = fma(y, -rdx, x);
      const T tr = fma(w, S.md[0][e], fma(eta, fma(y, rdx, x), S.tbs[0][e]));
      *ts = fma(bt, S.sos[0][e], ob * tr);
      *pr = S.rq[0][e] * w;
    }
  };
  auto u0_at = [&](int j) { return i <= nx && j >= 0 && j < ny ? S.u[0][j * px + i] : (T)0; };
  if (p.j0 < p.j1) {
    u0_m = u0_at(p.j0 - 1);
    const T u0 = u0_at(p.j0);
    vertex(p.j0, u0, &t_j, &p_j);
    u0_m = u0;
  }
  for (int j = p.j0; j < p.j1; ++j) {
    const int e = j * px + i;
    const T u0 = u0_m, u0_p = u0_at(j + 1);
    T t_p, p_p;
    vertex(j + 1, u0_p, &t_p, &p_p);
    u0_m = u0_p;
    const T pc = p_j + p_p, tc = t_j + t_p;
    const T xy = pc + right(pc), txy = tc + right(tc), u0_r = right(u0);
    if (own) S.Ts[0][e] = t_j;
    if (own && i < nx && j < ny) {
      const T d0 = u0_r - u0, d1 = S.u[1][e + px] - S.u[1][e];
      // the rate e - div / 3 rounded once, then scaled
      const T div = fma(d1, rdy, d0 * rdx), d3 = div * (T)(-1.0 / 3.0);
      const T t0 = fma((T)0.25, xy, fma(two_eta, fma(d0, rdx, d3), S.tbn[0][e]));
      const T t1 = fma((T)-0.25, xy, fma(two_eta, fma(d1, rdy, d3), S.tbn[1][e]));
      const T c0 = fma(bt, S.son[0][e], ob * t0), c1 = fma(bt, S.son[1][e], ob * t1);
      const T pr = fma(bp, S.sop[e], obp * fma(-KDt, div, S.pb[e]));
      T s = 1;
      if (frozen) {
        s = S.s[e];   // frozen plasticity: the held scale (Sec. 3.3)
      } else {
        const T J2 = fma((T)0.0625, txy * txy, (T)0.5 * fma(c1, c1, c0 * c0));
        s = scale_of(J2, fma(Ac, pr, S.yc[e]));
        S.s[e] = s;
      }
      const T n0 = s * c0, n1 = s * c1, s0 = n0 - pr, s1 = n1 - pr;
      S.snn[0][e] = n0;
      S.snn[1][e] = n1;
      S.snp[e] = pr;
      S.sx[0][e] = s0;
      S.sx[1][e] = s1;
      if (CHK) {
        sig = maxn(sig, maxn(fabs((double)s0), fabs((double)s1)));
        dtau = maxn(dtau, maxn(gap(n0, S.cn[0][e]), gap(n1, S.cn[1][e])));
        dp = maxn(dp, gap(pr, S.cp[e]));
        S.cn[0][e] = n0;
        S.cn[1][e] = n1;
        S.cp[e] = pr;
        if (isnan(s) || isnan(pr)) sig = NAN;
      }
    }
    t_j = t_p;
    p_j = p_p;
  }
  if (CHK && di) {
    block_max(sig, &di->red[RED_SIG]);
    block_max(dtau, &di->red[RED_DTAU]);
    block_max(dp, &di->red[RED_DP]);
  }
}

template <typename T, bool CHK>
__global__ void __launch_bounds__(128) k_move2d(Geo g, Stage<T> S, const Scal *sc, DevInfo *di, int rows) {
  if (skip(di)) return;
  const Strip p = strip(g, rows);
  const int i = p.i, nx = g.nx, ny = g.ny;
  const int px = g.px;   // a 2D box has fewer than 2^31 points
  const SweepScal<T> &Q = sweep_scal<T>(sc);
  const T vs = Q.vstep, rdx = Q.rdx, rdy = Q.rdy;
  const bool x1 = i > 0 && i < nx, own = p.lane < 31 && i <= nx;
  double sig = 0.0, dtau = 0.0, rmax = 0.0, du = 0.0, vm = 0.0;   // stopping measures, in FP64
  // scales of the two centres beside column i in row j
  auto pair = [&](int j) { return x1 && j >= 0 && j < ny ? S.s[j * px + i - 1] + S.s[j * px + i] : (T)0; };
  // new deviator of vertex (i, j) from its rows of scales
  auto vertex = [&](int j, T below, T at) {
    return x1 && j > 0 && j < ny ? (below + at) * ((T)0.25 * S.Ts[0][j * px + i]) : (T)0;
  };
  T h_m = pair(p.j0 - 1), h = pair(p.j0), v = vertex(p.j0, h_m, h);
  for (int j = p.j0; j < p.j1; ++j) {
    const int e = j * px + i;
    const T h_p = pair(j + 1), v_p = vertex(j + 1, h, h_p), v_r = right(v);
    if (own) {
      S.sns[0][e] = v;
      if (CHK) {
        sig = maxn(sig, fabs((double)v));
        dtau = maxn(dtau, gap(v, S.cs[0][e]));
        S.cs[0][e] = v;
      }
      // face d: in = inside its extent, in1 = off the walls
      const auto face = [&](int d, bool in, bool in1, T R) {
        const T u = S.u[d][e];
        T un = u;
        if (in1) {
          if (S.f[d]) R += S.f[d][e];
          un = fma(vs, R, u);
          if (CHK) rmax = maxn(rmax, fabs((double)R));
        }
        S.uo[d][e] = un;
        if (CHK && in) {
          du = maxn(du, gap(un, S.uchk[d][e]));
          vm = maxn(vm, fabs(S.v0[d][e] + (double)u));
          S.uchk[d][e] = un;
        }
      };
      const bool ix = j < ny, iy = i < nx;
      T R = 0;
      if (ix && x1) R = fma(v_p - v, rdy, (S.sx[0][e] - S.sx[0][e - 1]) * rdx);
      face(0, ix, ix && x1, R);
      const bool y1 = iy && j > 0 && j < ny;
      if (y1) R = fma(v_r - v, rdx, (S.sx[1][e] - S.sx[1][e - px]) * rdy);
      face(1, iy, y1, R);
    }
    h = h_p;
    v = v_p;
  }
  if (CHK && di) {
    block_max(sig, &di->red[RED_SIG]);
    block_max(dtau, &di->red[RED_DTAU]);
    block_max(rmax, &di->red[RED_R]);
    block_max(du, &di->red[RED_DU]);
    block_max(vm, &di->red[RED_V]);
  }
}

// mean of c2 dt (tyy - txx) over the centres around a vertex, times 1/2: the weight
// of the vertex's w
template <typename T>
__global__ void __launch_bounds__(256) k_rotation_mean2d(Geo g, const T *rd, T *md) {
  const int i = blockIdx.x * 32 + threadIdx.x, px = g.px;
  if (i < 1 || i >= g.nx) return;
  for (int j = blockIdx.y * 8 + threadIdx.y; j < g.ny; j += gridDim.y * 8) {
    if (j < 1) continue;
    const int e = j * px + i;
    md[e] = (T)0.125 * (rd[e - px - 1] + rd[e - px] + rd[e - 1] + rd[e]);
  }
}

// rows per warp (a strip recomputes one row of vertices), doubled up to 8 while
// every SM still has eight warps (152 SMs)
int strip_rows(const Geo &g, dim3 *grid, dim3 *block) {
  const int bx = (g.nx + 31) / 31;   // points 0 .. nx, 31 per warp
  int rows = 1;
  while (rows < 8 && (long long)bx * ((g.py + 2 * rows - 1) / (2 * rows)) >= 1216) rows *= 2;
  while (((g.py + rows - 1) / rows + 3) / 4 > 65535) rows *= 2;   // the longest launch
  const int strips = (g.py + rows - 1) / rows;
  int w = 4;
  while (w > 1 && (long long)bx * ((strips + w - 1) / w) < 304) w /= 2;
  *block = dim3(32, w);
  *grid = dim3(bx, (strips + w - 1) / w);
  return rows;
}

}  // namespace

template <typename T>
void launch_sweep2d(const Geo &g, const Stage<T> &S, const Scal *sc, DevInfo *di, bool check, cudaStream_t st,
                    const cudaEvent_t *ev) {
  dim3 gr, bl;
  const int rows = strip_rows(g, &gr, &bl);
  if (check) k_stress2d<T, true><<<gr, bl, 0, st>>>(g, S, sc, di, rows);
  else k_stress2d<T, false><<<gr, bl, 0, st>>>(g, S, sc, di, rows);
  if (ev) cudaEventRecord(ev[1], st);
  if (check) k_move2d<T, true><<<gr, bl, 0, st>>>(g, S, sc, di, rows);
  else k_move2d<T, false><<<gr, bl, 0, st>>>(g, S, sc, di, rows);
  if (ev) cudaEventRecord(ev[2], st);
}

template <typename T>
void launch_rotation_mean2d(const Geo &g, const T *rd, T *md, cudaStream_t st) {
  k_rotation_mean2d<T><<<dim3((g.nx + 32) / 32, std::min((g.py + 7) / 8, 65535)), dim3(32, 8), 0, st>>>(g, rd, md);
}

template void launch_sweep2d<float>(const Geo &, const Stage<float> &, const Scal *, DevInfo *, bool, cudaStream_t,
                                    const cudaEvent_t *);
template void launch_sweep2d<double>(const Geo &, const Stage<double> &, const Scal *, DevInfo *, bool, cudaStream_t,
                                     const cudaEvent_t *);
template void launch_rotation_mean2d<float>(const Geo &, const float *, float *, cudaStream_t);
template void launch_rotation_mean2d<double>(const Geo &, const double *, double *, cudaStream_t);

}  // namespace ep
