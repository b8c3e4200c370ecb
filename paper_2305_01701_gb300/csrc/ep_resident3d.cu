// ep_resident3d.cu -- the unchecked iterations of a chunk on one small 3D FP32 grid, in
// one cooperative launch that keeps the grid on the chip.
//
// The iteration of ep_sweep64.cu (the same sums and factors) in FP32.  A launch per
// iteration leaves a small grid with too few planes to march: its time is launch and
// load latency.  Here a block owns a box of tx x ty x tz points for the whole chunk:
// velocities, spins, trials and shear stresses sit in shared memory with a halo, normal
// stresses and coefficients in registers.  An iteration has five phases:
//   1. spins w on the points 1 around the edges        (velocity halo of 2)
//   2. trials and rotation products on the block's edges and those that bound it above
//   3. trials, pressure and return at the block's centres; scales and normal stresses
//      go to the neighbours
//   4. shear stresses of the edges of phase 2          (scale halo of 1)
//   5. velocities of the block's faces, which go to the neighbours
// so that only spins and edges are computed twice, and two exchanges carry the rest
// (ep_words.cuh).  One buffer serves both: a block overwrites its velocities after it
// has read every neighbour's scales, which that one sent after reading the velocities, and
// the other way round; every point of the halo is read, also where it holds no centre, so
// that each neighbour is waited for.  All blocks are resident at once (cooperative launch,
// one per SM); a wait gives up after the grid's bound or when another one has: done = 4, every
// block returns.
//
// Bound: shared memory and instruction issue of one block per SM, and the latency of two
// exchanges and five barriers.
// Measured, an iteration against the register sweep's launch (a box near yield, checks every
// 1000): 16^3 9.2 -> 3.5 us, 32^3 11.4 -> 6.2, 44^3 13.1 -> 6.2, 90 x 40 x 24 13.3 -> 7.6 (of
// 14,900 cycles there phases 1 - 5 take 1,500, 2,800, 2,300, 750 and 1,300 and the exchanges
// 6,200; 54 % of L1's rate, stalls on barriers 5.4, words 3.6 and shared memory 4.5 a warp
// instruction); two grids solved at once 20.1 -> 15.4 ms for 1000 iterations each, four
// 39.9 -> 31.0.  A spilled register costs an L2 trip here, since shared memory leaves L1 no
// room (30 spilled loads a warp and iteration: 9.3 us): what a thread keeps of its edges sits
// in shared memory.
#include <math.h>

#include "ep_internal.cuh"
#include "ep_lanes.cuh"
#include "ep_words.cuh"

namespace ep {

namespace {

constexpr int NT_MAX = 704;        // threads, one per owned point: 22 warps of 80 registers
constexpr int SPIN_TRIPS = 4, EDGE_TRIPS = 2, HALO_TRIPS = 4, SHELL_TRIPS = 2;
constexpr size_t SMEM_MAX = 227 * 1024 - 256;
constexpr int PITCH = 2240;        // floats of an array of the block's lattice
constexpr int ARRAYS = 16;         // u, w (then the normal stresses), p, ts, sns (3 each), s
constexpr int OWN = 12 * EDGE_TRIPS;   // coefficients of a thread's edges
constexpr int VALUES = PITCH * ARRAYS + NT_MAX * OWN;

struct Tile3 {
  int t[3];   // owned points along x, y, z
  __host__ __device__ int lat(int d) const { return t[d] + 4; }
  __host__ __device__ int lattice() const { return lat(0) * lat(1) * lat(2); }
  __host__ __device__ int owned() const { return t[0] * t[1] * t[2]; }
  __host__ __device__ int spins() const { return (t[0] + 3) * (t[1] + 3) * (t[2] + 3); }
  __host__ __device__ int edges() const { return (t[0] + 1) * (t[1] + 1) * (t[2] + 1); }
  __host__ __device__ int halo() const { return lattice() - owned(); }
  __host__ int threads() const { const int n = (edges() + 31) / 32 * 32; return n < NT_MAX ? n : NT_MAX; }
  __host__ __device__ int shell() const { return (t[0] + 2) * (t[1] + 2) * (t[2] + 2) - owned(); }
  // values, two counters, the two halo lists (lattice index and bits, point)
  __host__ size_t smem() const { return (size_t)VALUES * 4 + 16 + (size_t)(halo() + shell()) * sizeof(int2); }
};

// which edges of a point are interior: bit c for orientation c (xy, xz, yz)
__device__ __forceinline__ int interior(const Geo &g, int i, int j, int k) {
  const bool x1 = i > 0 && i < g.nx, y1 = j > 0 && j < g.ny, z1 = k > 0 && k < g.nz;
  const bool x0 = i >= 0 && i < g.nx, y0 = j >= 0 && j < g.ny, z0 = k >= 0 && k < g.nz;
  return (x1 && y1 && z0 ? 1 : 0) | (x1 && z1 && y0 ? 2 : 0) | (y1 && z1 && x0 ? 4 : 0);
}

__global__ void __launch_bounds__(NT_MAX, 1) k_resident3d(Geo g, Stage<float> S, const Scal *sc, DevInfo *di, Tile3 T,
                                                         int iters, unsigned *count, Word *words) {
  extern __shared__ float sm[];
  const int tid = threadIdx.x, nt = blockDim.x;
  // one thread's view of `done` for the block
  if (__syncthreads_or(tid == 0 && *(volatile const int *)&di->done != 0)) return;
  const bool frozen = di->frozen != 0;
  const int px = g.px, pl = (int)g.plane;   // the box is small: 32-bit indices
  const int ly = T.lat(0), lz = T.lat(0) * T.lat(1), n = T.lattice();   // lattice strides
  constexpr int N = PITCH;
  float *const u0 = sm, *const u1 = sm + N, *const u2 = sm + 2 * N, *const w0 = sm + 3 * N, *const w1 = sm + 4 * N,
               *const w2 = sm + 5 * N, *const p0 = sm + 6 * N, *const p1 = sm + 7 * N, *const p2 = sm + 8 * N,
               *const t0 = sm + 9 * N, *const t1 = sm + 10 * N, *const t2 = sm + 11 * N, *const n0 = sm + 12 * N,
               *const n1 = sm + 13 * N, *const n2 = sm + 14 * N, *const s = sm + 15 * N;
  // phase 3 writes the normal stresses where phase 1 writes the spins; products and
  // trials of points that are no interior edge stay zero
  float *const x0 = w0, *const x1 = w1, *const x2 = w2;
  float *const own = sm + ARRAYS * N + tid;   // of the thread's edges: tbs, rq, md, ma
  int *const counter = (int *)(sm + VALUES);
  int2 *const hu = (int2 *)(counter + 4), *const hs = hu + T.halo();
  const int bi = blockIdx.x * T.t[0] - 2, bj = blockIdx.y * T.t[1] - 2, bk = blockIdx.z * T.t[2] - 2;
  __shared__ SweepScal<float> Q;
  __shared__ long long limit;
  if (tid == 0) {
    Q = sweep_scal<float>(sc);
    limit = wait_limit(sc);
  }
  __syncthreads();
  const float rdx = Q.rdx, rdy = Q.rdy, rdz = Q.rdz, eta = Q.eta, bt = Q.bt, ob = Q.ob;
  auto in_box = [&](int i, int j, int k) {
    return i >= 0 && i <= g.nx && j >= 0 && j <= g.ny && k >= 0 && k <= g.nz;
  };

  if (tid < 2) counter[tid] = 0;
  for (int t = tid; t < VALUES; t += nt) sm[t] = 0.f;
  __syncthreads();
  // velocities, shear stresses and scales of the lattice; the halo lists
  for (int t = tid; t < n; t += nt) {
    const int a = t % ly, r = t / ly, b = r % T.lat(1), c = r / T.lat(1);
    const int i = bi + a, j = bj + b, k = bk + c;
    if (!in_box(i, j, k)) continue;
    const int e = k * pl + j * px + i;
    u0[t] = S.u[0][e]; u1[t] = S.u[1][e]; u2[t] = S.u[2][e];
    n0[t] = S.sos[0][e]; n1[t] = S.sos[1][e]; n2[t] = S.sos[2][e];
    const bool oa = a >= 2 && a < T.t[0] + 2, obb = b >= 2 && b < T.t[1] + 2, oc = c >= 2 && c < T.t[2] + 2;
    if (oa && obb && oc) continue;
    hu[atomicAdd(&counter[0], 1)] = make_int2(t, e);
    if (a >= 1 && a < T.t[0] + 3 && b >= 1 && b < T.t[1] + 3 && c >= 1 && c < T.t[2] + 3) {
      // normal stresses are needed below the block only
      const int bits = (a == 1 && obb && oc ? 1 : 0) | (b == 1 && oa && oc ? 2 : 0) | (c == 1 && oa && obb ? 4 : 0);
      hs[atomicAdd(&counter[1], 1)] = make_int2(t | bits << 16, e);
    }
  }

  // phases 1 and 2/4: a thread's points as lattice index and interior bits
  int sp[SPIN_TRIPS], eg[EDGE_TRIPS];
#pragma unroll
  for (int r = 0; r < SPIN_TRIPS; ++r) {
    const int t = tid + r * nt, a = t % (T.t[0] + 3) + 1, q = t / (T.t[0] + 3), b = q % (T.t[1] + 3) + 1,
              c = q / (T.t[1] + 3) + 1;
    sp[r] = t < T.spins() ? (c * lz + b * ly + a) | interior(g, bi + a, bj + b, bk + c) << 16 | 1 << 20 : 0;
  }
  float mb[EDGE_TRIPS][3];
#pragma unroll
  for (int r = 0; r < EDGE_TRIPS; ++r) {
    const int t = tid + r * nt, a = t % (T.t[0] + 1) + 2, q = t / (T.t[0] + 1), b = q % (T.t[1] + 1) + 2,
              c = q / (T.t[1] + 1) + 2;
    eg[r] = t < T.edges() ? (c * lz + b * ly + a) | interior(g, bi + a, bj + b, bk + c) << 16 : 0;
    const int e = (bk + c) * pl + (bj + b) * px + bi + a;
#pragma unroll
    for (int o = 0; o < 3; ++o)
      if (eg[r] >> 16 & (1 << o)) {
        own[(12 * r + o) * NT_MAX] = S.tbs[o][e];
        own[(12 * r + 3 + o) * NT_MAX] = S.rq[o][e];
      }
#pragma unroll
    for (int o = 0; o < 3; ++o) mb[r][o] = 0.f;
    // the rotation's coefficients (of the edge's own w; of the sums of four w)
    const float *q0 = S.rq[0], *q1 = S.rq[1], *q2 = S.rq[2], *r0 = S.rd[0], *r1 = S.rd[1];
    if (eg[r] >> 16 & 1) {
      own[(12 * r + 6) * NT_MAX] = 0.125f * (r0[e - px - 1] + r0[e - px] + r0[e - 1] + r0[e]);
      own[(12 * r + 9) * NT_MAX] = 0.03125f * (q2[e - 1] + q2[e] + q2[e - 1 + pl] + q2[e + pl]);
      mb[r][0] = 0.03125f * (q1[e - px] + q1[e] + q1[e - px + pl] + q1[e + pl]);
    }
    if (eg[r] >> 16 & 2) {
      own[(12 * r + 7) * NT_MAX] = 0.125f * (r1[e - pl - 1] + r1[e - pl] + r1[e - 1] + r1[e]);
      own[(12 * r + 10) * NT_MAX] = 0.03125f * (q2[e - 1] + q2[e] + q2[e - 1 + px] + q2[e + px]);
      mb[r][1] = -0.03125f * (q0[e - pl] + q0[e - pl + px] + q0[e] + q0[e + px]);
    }
    if (eg[r] >> 16 & 4) {
      own[(12 * r + 8) * NT_MAX] = 0.125f * ((r1[e - pl - px] - r0[e - pl - px]) + (r1[e - pl] - r0[e - pl]) +
                           (r1[e - px] - r0[e - px]) + (r1[e] - r0[e]));
      own[(12 * r + 11) * NT_MAX] = -0.03125f * (q0[e - pl] + q0[e - pl + 1] + q0[e] + q0[e + 1]);
      mb[r][2] = -0.03125f * (q1[e - px] + q1[e - px + 1] + q1[e] + q1[e + 1]);
    }
  }
  // phases 3 and 5: the thread's own point
  const int oa = tid % T.t[0], orow = tid / T.t[0], ob_ = orow % T.t[1], oc = orow / T.t[1];
  const int i = bi + 2 + oa, j = bj + 2 + ob_, k = bk + 2 + oc;
  const bool owned = tid < T.owned() && in_box(i, j, k);
  const int l = (oc + 2) * lz + (ob_ + 2) * ly + oa + 2, e = k * pl + j * px + i;
  const bool cin = owned && i < g.nx && j < g.ny && k < g.nz;
  const bool fx = owned && i > 0 && i < g.nx && j < g.ny && k < g.nz;
  const bool fy = owned && j > 0 && j < g.ny && i < g.nx && k < g.nz;
  const bool fz = owned && k > 0 && k < g.nz && i < g.nx && j < g.ny;
  float tb0 = 0.f, tb1 = 0.f, tb2 = 0.f, c0 = 0.f, c1 = 0.f, c2 = 0.f, pr = 0.f, pb = 0.f, yc = 0.f, sv = 1.f;
  if (cin) {
    tb0 = S.tbn[0][e]; tb1 = S.tbn[1][e]; tb2 = S.tbn[2][e];
    c0 = S.son[0][e]; c1 = S.son[1][e]; c2 = S.son[2][e];
    pr = S.sop[e]; pb = S.pb[e]; yc = S.yc[e];
    if (frozen) sv = S.s[e];   // frozen plasticity: the held scale (Sec. 3.3)
  }
  unsigned *const mine = count + (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  const unsigned base = *mine;
  const long long field = g.box;   // words: velocities; scale and two normal stresses; the third
  __syncthreads();
  if (tid == 0) *mine = base + iters;

  for (int q = 0; q < iters; ++q) {
    const unsigned tag = base + q + 1;
    // ---- 1: spins (w = 2 omega) ----
#pragma unroll
    for (int r = 0; r < SPIN_TRIPS; ++r) {
      const int m = sp[r] & 0xffff, in = sp[r] >> 16;
      if (!in) continue;
      const float a0 = u0[m], a1 = u1[m], a2 = u2[m], b1 = u1[m - 1], b2 = u2[m - 1], d0 = u0[m - ly],
                  d2 = u2[m - ly], f0 = u0[m - lz], f1 = u1[m - lz];
      w0[m] = in & 1 ? fmaf(a1 - b1, -rdx, (a0 - d0) * rdy) : 0.f;
      w1[m] = in & 2 ? fmaf(a2 - b2, -rdx, (a0 - f0) * rdz) : 0.f;
      w2[m] = in & 4 ? fmaf(a2 - d2, -rdy, (a1 - f1) * rdz) : 0.f;
    }
    __syncthreads();
    // ---- 2: relaxed trials and rotation products at edges ----
    float ts[EDGE_TRIPS][3];
#pragma unroll
    for (int r = 0; r < EDGE_TRIPS; ++r) {
      const int m = eg[r] & 0xffff, in = eg[r] >> 16;
      ts[r][0] = ts[r][1] = ts[r][2] = 0.f;
      if (!in) continue;
      // every load before the first store: a chain of three edges would wait for each
      const float a0 = u0[m], a1 = u1[m], a2 = u2[m], b1 = u1[m - 1], b2 = u2[m - 1], d0 = u0[m - ly],
                  d2 = u2[m - ly], f0 = u0[m - lz], f1 = u1[m - lz];
      const float v0 = w0[m], v1 = w1[m], v2 = w2[m];
      // sums of the spins of the other two orientations
      const float g0 = (w1[m - ly] + v1) + (w1[m - ly + lz] + w1[m + lz]);
      const float h0 = (w2[m - 1] + v2) + (w2[m - 1 + lz] + w2[m + lz]);
      const float g1 = (w0[m - lz] + w0[m - lz + ly]) + (v0 + w0[m + ly]);
      const float h1 = (w2[m - 1] + v2) + (w2[m - 1 + ly] + w2[m + ly]);
      const float g2 = (w1[m - ly] + w1[m - ly + 1]) + (v1 + w1[m + 1]);
      const float h2 = (w0[m - lz] + w0[m - lz + 1]) + (v0 + w0[m + 1]);
      const float o0 = n0[m], o1 = n1[m], o2 = n2[m];
      constexpr int W = NT_MAX;
      const float *c = own + 12 * r * W;
      const float tb[3] = {c[0], c[W], c[2 * W]}, rq[3] = {c[3 * W], c[4 * W], c[5 * W]},
                  md[3] = {c[6 * W], c[7 * W], c[8 * W]}, ma[3] = {c[9 * W], c[10 * W], c[11 * W]};
      auto edge = [&](int o, float gs, float w, float wa, float wb, float old) {
        const float tr = fmaf(w, md[o], fmaf(wa, ma[o], fmaf(wb, mb[r][o], fmaf(eta, gs, tb[o]))));
        ts[r][o] = fmaf(bt, old, ob * tr);
      };
      edge(0, fmaf(a1 - b1, rdx, (a0 - d0) * rdy), v0, g0, h0, o0);
      edge(1, fmaf(a2 - b2, rdx, (a0 - f0) * rdz), v1, g1, h1, o1);
      edge(2, fmaf(a2 - d2, rdy, (a1 - f1) * rdz), v2, g2, h2, o2);
      if (in & 1) { t0[m] = ts[r][0]; p0[m] = rq[0] * v0; }
      if (in & 2) { t1[m] = ts[r][1]; p1[m] = rq[1] * v1; }
      if (in & 4) { t2[m] = ts[r][2]; p2[m] = rq[2] * v2; }
    }
    __syncthreads();
    // ---- 3: relaxed trial, pressure and return at the own centre ----
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    if (cin) {
      const float d0 = u0[l + 1] - u0[l], d1 = u1[l + ly] - u1[l], d2 = u2[l + lz] - u2[l];
      const float div = fmaf(d2, rdz, fmaf(d1, rdy, d0 * rdx)), d3 = div * (-1.f / 3.f);
      const float xy = (p0[l] + p0[l + 1]) + (p0[l + ly] + p0[l + ly + 1]);
      const float xz = (p1[l] + p1[l + 1]) + (p1[l + lz] + p1[l + lz + 1]);
      const float yz = (p2[l] + p2[l + ly]) + (p2[l + lz] + p2[l + lz + ly]);
      c0 = fmaf(bt, c0, ob * fmaf(0.25f, xy + xz, fmaf(Q.two_eta, fmaf(d0, rdx, d3), tb0)));
      c1 = fmaf(bt, c1, ob * fmaf(0.25f, yz - xy, fmaf(Q.two_eta, fmaf(d1, rdy, d3), tb1)));
      c2 = fmaf(bt, c2, ob * fmaf(-0.25f, xz + yz, fmaf(Q.two_eta, fmaf(d2, rdz, d3), tb2)));
      pr = fmaf(Q.bp, pr, Q.obp * fmaf(-Q.KDt, div, pb));
      if (!frozen) {
        const float txy = (t0[l] + t0[l + 1]) + (t0[l + ly] + t0[l + ly + 1]);
        const float txz = (t1[l] + t1[l + 1]) + (t1[l + lz] + t1[l + lz + 1]);
        const float tyz = (t2[l] + t2[l + ly]) + (t2[l + lz] + t2[l + lz + ly]);
        const float J2 = fmaf(0.0625f, fmaf(tyz, tyz, fmaf(txz, txz, txy * txy)),
                              0.5f * fmaf(c2, c2, fmaf(c1, c1, c0 * c0)));
        sv = scale_of(J2, fmaf(Q.A, pr, yc));
      }
      c0 *= sv; c1 *= sv; c2 *= sv;
      s0 = c0 - pr; s1 = c1 - pr; s2 = c2 - pr;
    }
    if (owned) {
      send(words + field + e, 0, sv, s0, s1, tag);
      send(words + 2 * field + e, 0, s2, 0.f, 0.f, tag);
      s[l] = sv;
      x0[l] = s0; x1[l] = s1; x2[l] = s2;
    }
    bool lost = false;
    {
      Wait w = wait_begin();
      bool need[SHELL_TRIPS];
#pragma unroll
      for (int r = 0; r < SHELL_TRIPS; ++r) need[r] = tid + r * nt < counter[1];
      for (;;) {
        bool again = false;
#pragma unroll
        for (int r = 0; r < SHELL_TRIPS; ++r) {
          if (!need[r]) continue;
          const int2 h = hs[tid + r * nt];
          const int m = h.x & 0xffff, bits = h.x >> 16;
          float a, b0, b1, b2 = 0.f, none;
          bool ok = receive(words + field + h.y, 0, tag, &a, &b0, &b1, true);
          if (bits & 4) ok = receive(words + 2 * field + h.y, 0, tag, &b2, &none, &none, false) && ok;
          if (ok) {
            s[m] = a;
            if (bits & 1) x0[m] = b0;
            if (bits & 2) x1[m] = b1;
            if (bits & 4) x2[m] = b2;
            need[r] = false;
          }
          again |= need[r];
        }
        if (!again) break;
        if (wait_over(w, limit, di)) { lost = true; break; }
      }
    }
    if (__syncthreads_or(lost)) return;
    // ---- 4: shear stresses from the mean of the scales around ----
#pragma unroll
    for (int r = 0; r < EDGE_TRIPS; ++r) {
      const int m = eg[r] & 0xffff, in = eg[r] >> 16;
      if (!in) continue;
      const float a = s[m], b = s[m - 1], c = s[m - ly], d = s[m - lz];
      const float v0 = ((s[m - ly - 1] + c) + (b + a)) * (0.25f * ts[r][0]);
      const float v1 = ((s[m - lz - 1] + d) + (b + a)) * (0.25f * ts[r][1]);
      const float v2 = ((s[m - lz - ly] + d) + (c + a)) * (0.25f * ts[r][2]);
      if (in & 1) n0[m] = v0;
      if (in & 2) n1[m] = v1;
      if (in & 4) n2[m] = v2;
    }
    __syncthreads();
    // the stresses that the last iteration starts from stay where the launch found its own:
    // a commit before the solve is decided takes them.  Every neighbour has read that state:
    // it sent the words of iteration 0 since.
    if (q == iters - 2 && owned) {
      const_cast<float *>(S.sos[0])[e] = n0[l];
      const_cast<float *>(S.sos[1])[e] = n1[l];
      const_cast<float *>(S.sos[2])[e] = n2[l];
      if (cin) {
        const_cast<float *>(S.son[0])[e] = c0;
        const_cast<float *>(S.son[1])[e] = c1;
        const_cast<float *>(S.son[2])[e] = c2;
        const_cast<float *>(S.sop)[e] = pr;
      }
    }
    // ---- 5: residual and velocity of the own faces ----
    float un0 = 0.f, un1 = 0.f, un2 = 0.f;
    if (owned) {
      const float a0 = n0[l], a1 = n1[l], a2 = n2[l], b0 = n0[l + 1], b1 = n1[l + 1], d0 = n0[l + ly], d2 = n2[l + ly],
                  h1 = n1[l + lz], h2 = n2[l + lz], y0 = x0[l - 1], y1 = x1[l - ly], y2 = x2[l - lz];
      un0 = u0[l]; un1 = u1[l]; un2 = u2[l];
      if (fx) un0 = fmaf(Q.vstep, fmaf(h1 - a1, rdz, fmaf(d0 - a0, rdy, (s0 - y0) * rdx)), un0);
      if (fy) un1 = fmaf(Q.vstep, fmaf(h2 - a2, rdz, fmaf(b0 - a0, rdx, (s1 - y1) * rdy)), un1);
      if (fz) un2 = fmaf(Q.vstep, fmaf(d2 - a2, rdy, fmaf(b1 - a1, rdx, (s2 - y2) * rdz)), un2);
      if (q < iters - 1) send(words + e, 0, un0, un1, un2, tag);
      u0[l] = un0; u1[l] = un1; u2[l] = un2;
    }
    if (q == iters - 1) break;
    {
      Wait w = wait_begin();
      bool need[HALO_TRIPS];
#pragma unroll
      for (int r = 0; r < HALO_TRIPS; ++r) need[r] = tid + r * nt < counter[0];
      for (;;) {
        float a[HALO_TRIPS][3];
        bool ok[HALO_TRIPS], again = false;
#pragma unroll
        for (int r = 0; r < HALO_TRIPS; ++r) {
          ok[r] = false;
          if (!need[r]) continue;
          const int x = hu[tid + r * nt].y;
          ok[r] = receive(words + x, 0, tag, &a[r][0], &a[r][1], &a[r][2], true);
        }
#pragma unroll
        for (int r = 0; r < HALO_TRIPS; ++r) {
          if (ok[r]) {
            const int m = hu[tid + r * nt].x;
            u0[m] = a[r][0]; u1[m] = a[r][1]; u2[m] = a[r][2];
            need[r] = false;
          }
          again |= need[r];
        }
        if (!again) break;
        if (wait_over(w, limit, di)) { lost = true; break; }
      }
    }
    if (__syncthreads_or(lost)) return;
  }
  if (owned) {
    S.uo[0][e] = u0[l]; S.uo[1][e] = u1[l]; S.uo[2][e] = u2[l];
    S.sns[0][e] = n0[l]; S.sns[1][e] = n1[l]; S.sns[2][e] = n2[l];
    if (cin) {
      S.snn[0][e] = c0; S.snn[1][e] = c1; S.snn[2][e] = c2;
      S.snp[e] = pr;
      if (!frozen) S.s[e] = sv;
    }
  }
}

dim3 blocks_of(const Tile3 &T, const Geo &g) {
  return dim3((g.nx + T.t[0]) / T.t[0], (g.ny + T.t[1]) / T.t[1], (g.nz + T.t[2]) / T.t[2]);
}

// The box that each block owns: of those whose blocks are at most one per SM, the one
// with the least work (points of the phases, weighted by their instructions).  A grid of
// more points than the blocks hold (152 x 704) takes the register sweep.
bool tile_of(const Geo &g, int sms, Tile3 *best) {
  long long cost = 0;
  const int n[3] = {g.nx + 1, g.ny + 1, g.nz + 1};
  for (int tx = 4; tx <= 32; ++tx)
    for (int ty = 2; ty <= 32; ++ty)
      for (int tz = 2; tz <= 32 && tx * ty * tz <= NT_MAX; ++tz) {
        const Tile3 T{{tx, ty, tz}};
        const int nt = T.threads();
        const long long blocks = (long long)((n[0] + tx - 1) / tx) * ((n[1] + ty - 1) / ty) * ((n[2] + tz - 1) / tz);
        if (T.owned() > nt || blocks > sms || T.smem() > SMEM_MAX || T.lattice() > PITCH ||
            T.spins() > SPIN_TRIPS * nt || T.edges() > EDGE_TRIPS * nt || T.halo() > HALO_TRIPS * nt ||
            T.shell() > SHELL_TRIPS * nt)
          continue;
        const long long c = T.spins() + 4LL * T.edges() + 4LL * T.owned() + 2LL * T.halo();
        if (!cost || c < cost) {
          cost = c;
          *best = T;
        }
      }
  return cost != 0;
}

}  // namespace

bool resident3d_tile(const Geo &g, int tile[3]) {
  Tile3 T;
  if (g.ndim != 3 || (g.nx + 1LL) * (g.ny + 1) * (g.nz + 1) > (long long)RESIDENT_SMS * NT_MAX ||
      !tile_of(g, RESIDENT_SMS, &T))
    return false;
  for (int d = 0; d < 3; ++d) tile[d] = T.t[d];
  return true;
}

bool resident3d_runs(const Geo &g, const int tile[3]) {
  const Tile3 T{{tile[0], tile[1], tile[2]}};
  const dim3 b = blocks_of(T, g);
  int sms = 0, per = 0;
  return resident_device_sms(&sms) &&
         cudaFuncSetAttribute(k_resident3d, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) == cudaSuccess &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_resident3d, T.threads(), T.smem()) == cudaSuccess &&
         (long long)b.x * b.y * b.z <= (long long)per * sms;
}

cudaError_t launch_resident3d(const int tile[3], const Geo &g, const Stage<float> &S, const Scal *sc, DevInfo *di,
                              int iters, unsigned *count, Word *words, cudaStream_t st) {
  Tile3 T{{tile[0], tile[1], tile[2]}};
  Geo gg = g;
  Stage<float> SS = S;
  void *args[] = {&gg, &SS, &sc, &di, &T, &iters, &count, &words};
  return cudaLaunchCooperativeKernel((const void *)k_resident3d, blocks_of(T, g), dim3(T.threads()), args, T.smem(), st);
}

}  // namespace ep
