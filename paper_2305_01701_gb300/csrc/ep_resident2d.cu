// ep_resident2d.cu -- the unchecked iterations of a chunk on one small 2D grid, in one
// cooperative launch that keeps the state on the chip.
//
// The same iteration as ep_sweep2d.cu, operation by operation (equal results, bit
// for bit).  Two launches an iteration cost 8 us however small the grid is, most of it
// launch and load latency.  Here a thread owns one point of a lattice for the whole
// chunk and keeps its coefficients and stresses in registers; a block's lattice of
// WX x WY points overlaps its neighbours by two points on each side, where the
// stresses are computed twice, so that the blocks exchange only once an iteration: the
// velocities of the two outer rows and columns that a block owns, and the shear stress
// there.  Points of a block meet in shared memory.
//
// Exchange: ep_words.cuh.  Two buffers alternate: a block
// overwrites a word only after it has read from every neighbour what that one sent
// after reading the word.  All blocks are resident at once (cooperative launch,
// checked against the occupancy); a wait gives up after the grid's bound or when another
// one has: done = 4, every block returns.  Numbers only grow, by the same amount in
// every block of a launch; the buffers start a solve at zero.
//
// Bound: latency of the exchange and of four block barriers; FP64 grids the FP64 pipe
// as well, which takes a warp's instruction in 64 cycles.
// Measured, an iteration against two launches (a box near yield, checks every 1000): FP64
// 64^2 9.1 -> 4.3 us, 128^2 10.3 -> 6.8; FP32 64^2 8.0 -> 1.1, 128^2 8.3 -> 1.3, 383 x 191
// 12.1 -> 1.7, 300^2 12.5 -> 1.7 (a counter per block behind a fence, when the words were
// not yet 16 bytes wide: 64^2 FP64 7.5 us, 383 x 191 FP32 5.8).  FP64 64^2: 6 % of the issue
// slots, warps wait on the FP64 pipe (7.0 a warp instruction), barriers (2.9) and the words.
#include <math.h>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"
#include "ep_words.cuh"

namespace ep {

namespace {

template <typename T, int WX, int WY>
__global__ void __launch_bounds__(WX *WY) k_resident2d(Geo g, Stage<T> S, const Scal *sc, DevInfo *di, int iters,
                                                       unsigned *count, Word *words) {
  __shared__ T su0[WY][WX], su1[WY][WX], sp[WY][WX], st[WY][WX], ss[WY][WX], sx0[WY][WX], sx1[WY][WX], sn[WY][WX];
  const int tid = threadIdx.x, tx = tid % WX, ty = tid / WX;
  // one thread's view of `done` for the block
  if (__syncthreads_or(tid == 0 && *(volatile const int *)&di->done != 0)) return;
  const bool frozen = di->frozen != 0;
  const int nx = g.nx, ny = g.ny, px = g.px;   // a 2D box has fewer than 2^31 points
  const int gi = blockIdx.x * (WX - 4) - 2 + tx, gj = blockIdx.y * (WY - 4) - 2 + ty, e = gj * px + gi;
  const SweepScal<T> &Q = sweep_scal<T>(sc);
  const T two_eta = Q.two_eta, eta = Q.eta, bt = Q.bt, ob = Q.ob;
  const T bp = Q.bp, obp = Q.obp, KDt = Q.KDt, Ac = Q.A, rdx = Q.rdx, rdy = Q.rdy, vs = Q.vstep;

  const bool box = gi >= 0 && gi <= nx && gj >= 0 && gj <= ny;
  const bool owned = box && tx >= 2 && tx < WX - 2 && ty >= 2 && ty < WY - 2;
  const bool ring = owned && (tx < 4 || tx >= WX - 4 || ty < 4 || ty >= WY - 4);
  // interior vertices, and those of them whose deviator is formed here (the others
  // around a centre come from the block that owns them)
  const bool vin = gi > 0 && gi < nx && gj > 0 && gj < ny && tx >= 1 && ty >= 1;
  const bool vown = vin && tx >= 2 && tx < WX - 1 && ty >= 2 && ty < WY - 1;
  const bool cin = gi >= 0 && gi < nx && gj >= 0 && gj < ny && tx >= 1 && tx < WX - 1 && ty >= 1 && ty < WY - 1;
  const bool x1 = gi > 0 && gi < nx;
  const bool fx = owned && gj < ny && x1, fy = owned && gi < nx && gj > 0 && gj < ny;

  T u0 = 0, u1 = 0, md = 0, tbs = 0, rq = 0, tsh = 0;
  T tb0 = 0, tb1 = 0, n0 = 0, n1 = 0, pr = 0, pb = 0, yc = 0, s = 1, f0 = 0, f1 = 0;
  if (box) { u0 = S.u[0][e]; u1 = S.u[1][e]; }
  if (vin) { md = S.md[0][e]; tbs = S.tbs[0][e]; rq = S.rq[0][e]; tsh = S.sos[0][e]; }
  if (cin) {
    tb0 = S.tbn[0][e]; tb1 = S.tbn[1][e]; n0 = S.son[0][e]; n1 = S.son[1][e];
    pr = S.sop[e]; pb = S.pb[e]; yc = S.yc[e];
    if (frozen) s = S.s[e];   // frozen plasticity: the held scale (Sec. 3.3)
  }
  if (fx && S.f[0]) f0 = S.f[0][e];
  if (fy && S.f[1]) f1 = S.f[1][e];
  su0[ty][tx] = u0;
  su1[ty][tx] = u1;

  // iterations before this launch; a point's words: x and y velocity, shear stress
  unsigned *const mine = count + blockIdx.y * gridDim.x + blockIdx.x;
  const unsigned base = *mine;
  __syncthreads();
  if (tid == 0) *mine = base + iters;

  const long long limit = wait_limit(sc);
  for (int q = 0; q < iters; ++q) {
    // ---- vertex: relaxed trial, rotation product ----
    T ts = 0, p = 0;
    if (vin) {
      const T x = (u0 - su0[ty - 1][tx]) * rdy, y = u1 - su1[ty][tx - 1];
      const T w = fma(y, -rdx, x);
      const T tr = fma(w, md, fma(eta, fma(y, rdx, x), tbs));
      ts = fma(bt, tsh, ob * tr);
      p = rq * w;
    }
    sp[ty][tx] = p;
    st[ty][tx] = ts;
    __syncthreads();
    // ---- centre: relaxed trial, pressure, return ----
    T s0 = 0, s1 = 0;
    if (cin) {
      const T xy = (p + sp[ty + 1][tx]) + (sp[ty][tx + 1] + sp[ty + 1][tx + 1]);
      const T txy = (ts + st[ty + 1][tx]) + (st[ty][tx + 1] + st[ty + 1][tx + 1]);
      const T d0 = su0[ty][tx + 1] - u0, d1 = su1[ty + 1][tx] - u1;
      const T div = fma(d1, rdy, d0 * rdx), d3 = div * (T)(-1.0 / 3.0);
      const T t0 = fma((T)0.25, xy, fma(two_eta, fma(d0, rdx, d3), tb0));
      const T t1 = fma((T)-0.25, xy, fma(two_eta, fma(d1, rdy, d3), tb1));
      const T c0 = fma(bt, n0, ob * t0), c1 = fma(bt, n1, ob * t1);
      pr = fma(bp, pr, obp * fma(-KDt, div, pb));
      if (!frozen) {
        const T J2 = fma((T)0.0625, txy * txy, (T)0.5 * fma(c1, c1, c0 * c0));
        s = scale_of(J2, fma(Ac, pr, yc));
      }
      n0 = s * c0;
      n1 = s * c1;
      s0 = n0 - pr;
      s1 = n1 - pr;
    }
    ss[ty][tx] = s;
    sx0[ty][tx] = s0;
    sx1[ty][tx] = s1;
    __syncthreads();
    // ---- vertex: deviator from the mean of its centre scales ----
    T v = 0;
    if (vown) {
      v = ((ss[ty - 1][tx - 1] + ss[ty - 1][tx]) + (ss[ty][tx - 1] + s)) * ((T)0.25 * ts);
      tsh = v;
    }
    sn[ty][tx] = v;
    // the stresses that the last iteration starts from stay where the launch found its own:
    // a commit before the solve is decided takes them.  Every neighbour has read that state:
    // it sent the words of iteration 0 since.
    if (q == iters - 2 && owned) {
      const_cast<T *>(S.sos[0])[e] = vin ? tsh : (T)0;
      if (cin) {
        const_cast<T *>(S.son[0])[e] = n0;
        const_cast<T *>(S.son[1])[e] = n1;
        const_cast<T *>(S.sop)[e] = pr;
      }
    }
    __syncthreads();
    // ---- faces: residual and velocity update ----
    if (fx) {
      T R0 = fma(sn[ty + 1][tx] - v, rdy, (s0 - sx0[ty][tx - 1]) * rdx);
      if (S.f[0]) R0 += f0;
      u0 = fma(vs, R0, u0);
      su0[ty][tx] = u0;
    }
    if (fy) {
      T R1 = fma(sn[ty][tx + 1] - v, rdx, (s1 - sx1[ty - 1][tx]) * rdy);
      if (S.f[1]) R1 += f1;
      u1 = fma(vs, R1, u1);
      su1[ty][tx] = u1;
    }
    if (q == iters - 1) break;

    // ---- exchange with the neighbours ----
    const unsigned tag = base + q + 1;
    Word *const word = words + (q & 1) * g.box * words_of<T>() + e;
    bool lost = false;
    if (ring) {
      send(word, g.box, u0, u1, v, tag);
    } else if (box && !owned) {
      const bool shear = vin && !vown;
      for (Wait w = wait_begin();;) {
        T a, b, c = tsh;
        if (receive(word, g.box, tag, &a, &b, &c, shear)) {
          u0 = a;
          u1 = b;
          tsh = c;
          break;
        }
        if (wait_over(w, limit, di)) {
          lost = true;
          break;
        }
      }
      su0[ty][tx] = u0;
      su1[ty][tx] = u1;
    }
    if (__syncthreads_or(lost)) return;
  }
  if (owned) {
    S.uo[0][e] = u0;
    S.uo[1][e] = u1;
    S.sns[0][e] = vin ? tsh : (T)0;
    if (cin) {
      S.snn[0][e] = n0;
      S.snn[1][e] = n1;
      S.snp[e] = pr;
      if (!frozen) S.s[e] = s;
    }
  }
}

struct Config {
  int wx, wy;
};
// Lattices; a grid takes the one with the fewest points per SM, of equals the first (128^2
// FP32: 16 x 8 1.8 us, 32 x 16 2.05, 32 x 32 2.4; 96^2 FP64: 16 x 8 5.6, 16 x 16 6.5).
template <typename T>
Config config(int c) {
  return c == 0 ? Config{16, 8} : c == 1 ? Config{32, 16} : sizeof(T) == 8 ? Config{16, 16} : Config{32, 32};
}
constexpr int CONFIGS = 3;
template <typename T>
long long blocks_of(int c, const Geo &g) {
  const int ox = config<T>(c).wx - 4, oy = config<T>(c).wy - 4;
  return (long long)((g.nx + ox) / ox) * ((g.ny + oy) / oy);
}

template <typename T>
const void *kernel_of(int c) {
  if (c == 0) return (const void *)k_resident2d<T, 16, 8>;
  if (c == 1) return (const void *)k_resident2d<T, 32, 16>;
  if constexpr (sizeof(T) == 8) return (const void *)k_resident2d<T, 16, 16>;
  else return (const void *)k_resident2d<T, 32, 32>;
}

}  // namespace

bool resident_device_sms(int *sms) {
  int dev = 0, coop = 0;
  return cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop;
}

template <typename T>
int resident2d_config(const Geo &g) {
  int best = -1;
  // Points per SM that it pays up to.  FP32: what the registers hold (1024; 383 x 191
  // takes that).  FP64: the points computed twice go through the FP64 pipe, which several
  // grids solved at once on their own streams share: 128^2 (256 points) 9.1 -> 6.6 us
  // alone, 10.9 -> 9.8 with two grids, 15.0 -> 19.6 with four; 200^2 (512) 12.5 -> 9.9
  // alone but 17.4 -> 19.1 with two, so the two launches stay there.
  long long cost = (sizeof(T) == 4 ? 1024 : 256) + 1;
  for (int c = 0; c < CONFIGS; ++c) {
    const int wx = config<T>(c).wx, wy = config<T>(c).wy;
    const long long rounds = (blocks_of<T>(c, g) + RESIDENT_SMS - 1) / RESIDENT_SMS;
    if (blocks_of<T>(c, g) > RESIDENT_BLOCKS || rounds * wx * wy >= cost) continue;
    cost = rounds * wx * wy;
    best = c;
  }
  return best;
}

template <typename T>
bool resident2d_runs(int c, const Geo &g) {
  int sms = 0, per = 0;
  return c >= 0 && resident_device_sms(&sms) &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of<T>(c), config<T>(c).wx * config<T>(c).wy, 0) ==
             cudaSuccess &&
         blocks_of<T>(c, g) <= (long long)per * sms;
}

template <typename T>
cudaError_t launch_resident2d(int c, const Geo &g, const Stage<T> &S, const Scal *sc, DevInfo *di, int iters,
                              unsigned *count, Word *words, cudaStream_t st) {
  const int wx = config<T>(c).wx, wy = config<T>(c).wy;
  Geo gg = g;
  Stage<T> SS = S;
  void *args[] = {&gg, &SS, &sc, &di, &iters, &count, &words};
  return cudaLaunchCooperativeKernel(kernel_of<T>(c), dim3((g.nx + wx - 4) / (wx - 4), (g.ny + wy - 4) / (wy - 4)),
                                     dim3(wx * wy), args, 0, st);
}

template int resident2d_config<float>(const Geo &);
template int resident2d_config<double>(const Geo &);
template bool resident2d_runs<float>(int, const Geo &);
template bool resident2d_runs<double>(int, const Geo &);
template cudaError_t launch_resident2d<float>(int, const Geo &, const Stage<float> &, const Scal *, DevInfo *, int,
                                              unsigned *, Word *, cudaStream_t);
template cudaError_t launch_resident2d<double>(int, const Geo &, const Stage<double> &, const Scal *, DevInfo *, int,
                                               unsigned *, Word *, cudaStream_t);

}  // namespace ep
