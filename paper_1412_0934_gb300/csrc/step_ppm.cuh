// The step with piecewise-parabolic reconstruction (PPM; the paper lists it among its hydro
// methods, Sec. 2) on a periodic box.  Per axis and primitive variable (Colella & Woodward 1984):
//   dq_i    = MC-limited slope (the PLM MC limiter of q_i - q_{i-1} and q_{i+1} - q_i);
//   q_{i+h} = q_i + (q_{i+1} - q_i)/2 - (dq_{i+1} - dq_i)/6      (h = 1/2);
//   edges qL = q_{i-h}, qR = q_{i+h}, then: both set to q_i at a local extremum
//   ((qR - q)(q - qL) <= 0); else with D = qR - qL, Q6 = 6 (q - (qL + qR)/2): qL = 3q - 2qR if
//   D Q6 > D^2, qR = 3q - 2qL if -D^2 > D Q6.
// In double and double-float only the distances l = q - qL and r = qR - q are formed, from differences alone:
//   l = (q_i - q_{i-1})/2 + (dq_i - dq_{i-1})/6,   r = (q_{i+1} - q_i)/2 - (dq_{i+1} - dq_i)/6,
// both 0 where l r <= 0; there D = l + r and Q6 = 3 (l - r), so the two steepness tests are |l| > 2|r|
// (then l = 2r) and |r| > 2|l| (then r = 2l).  Half the operations of the edge form, none of its
// cancellation against q: the double-float step of a 191x203x187 box went from 8.2 to 7.7 ms.
// The rest is the PLM step with the parabola's centre slope D in the Hancock predictor and face
// states q_h + (qR - q), q_h + (qL - q) in place of q_h +- dq/2.  The stencil radius is 3.
//
// Kernel layout in float arithmetic: one thread per column of a TX x TY tile marching up z (as the PLM
// kernel), on a periodic box (indices wrapped) or on a patch carrying three ghost layers filled by the
// caller; 8-byte arithmetic splits each plane's work over 512 threads (PpmWideShared, below).
// Shared memory holds a ring of five recovered planes (p-2 .. p+2) over the tile and three halo
// cells each side, the x- and y-face states of plane p (the tile's cells and one ring cell beyond
// each edge) and the x and y fluxes of plane p.  The z reconstruction of a column reads its own
// five ring entries; the z-face state of the plane below, the z flux below and the x/y flux
// difference of the plane below stay in registers until the plane is updated one plane later.
#pragma once

#include <algorithm>

#include "adjoint.cuh"
#include "hydro_device.cuh"
#include "internal.h"
#include "step_tile.cuh"

namespace hydro {

constexpr int kPpmHalo = 3;

template <class R, int TX, int TY>
struct PpmShared {
  static constexpr int QX = TX + 2 * kPpmHalo, QY = TY + 2 * kPpmHalo;
  Plane5<R, QY, QX> q[5];       // ring of recovered planes: [slot] at (y + 3, x + 3)
  Plane5<R, TY, TX + 2> wx[2];  // x-face states at n+1/2: [0: low face, 1: high face] at (y, x + 1)
  Plane5<R, TY + 2, TX> wy[2];  // y-face states: [low/high] at (y + 1, x)
  Plane5<R, TY, TX + 1> fx;     // flux through the low x face of cell x, x = 0 .. TX
  Plane5<R, TY + 1, TX> fy;     // flux through the low y face of cell y, y = 0 .. TY
  int sx[QX], sy[QY];      // stored index of each tile column / row (wrapped, or clamped to the ghosts)
  R red[TX * TY / 32];     // per-warp maxima of the CFL speed
  int tile;                // batched kernel: the tile taken from the work-list
};

__device__ __forceinline__ int wrap_index(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// Distances (l, r) of the middle cell's edges from its four neighbour differences.
template <class R>
__device__ __forceinline__ void ppm_limit(R& l, R& r) {
  if (prod_nonpos(r, l)) {
    l = r = R(0);
    return;
  }
  const R l2 = twice_(l), r2 = twice_(r);
  if (abs_lt(r2, l)) l = r2;
  else if (abs_lt(l2, r)) r = l2;
}
__device__ __forceinline__ void ppm_limit(df& l, df& r) {  // selected, not branched
  const df l2 = twice_(l), r2 = twice_(r);
  const bool zero = prod_nonpos(r, l), pos = l.h > 0.f;
  const bool big_l = pos ? r2 < l : l < r2, big_r = pos ? l2 < r : r < l2;
  l = df(zero ? 0.f : (big_l ? r2.h : l.h), zero ? 0.f : (big_l ? r2.l : l.l));
  r = df(zero ? 0.f : (big_r ? l2.h : r.h), zero ? 0.f : (big_r ? l2.l : r.l));
}
template <class R>
__device__ __forceinline__ void ppm_edge(R ba, R cb, R dc, R ed, R sixth, R& l, R& r) {
  const R sb = mc_slope(ba, cb), sc = mc_slope(cb, dc), sd = mc_slope(dc, ed);
  l = half_(cb) + (sc - sb) * sixth;
  r = half_(dc) - (sd - sc) * sixth;
  ppm_limit(l, r);
}
__device__ __forceinline__ void ppm_edge(const df& ba, const df& cb, const df& dc, const df& ed, const df& sixth, df& l,
                                         df& r) {
  const df sb = mc_slope(ba, cb), sc = mc_slope(cb, dc), sd = mc_slope(dc, ed);
  l = half_(cb) + prod_(sum_(sc, -sb), sixth);
  r = half_(dc) + prod_(sum_(sc, -sd), sixth);
  ppm_limit(l, r);
}
__device__ __forceinline__ void ppm_edge(const df2& ba, const df2& cb, const df2& dc, const df2& ed, const df& sixth,
                                         df l[2], df r[2]) {
  const df2 sb = mc_slope(ba, cb), sc = mc_slope(cb, dc), sd = mc_slope(dc, ed), s6 = both_(sixth);
  const df2 x = half_(cb) + prod_(sum_(sc, neg_(sb)), s6), y = half_(dc) + prod_(sum_(sc, neg_(sd)), s6);
  l[0] = first_(x);
  r[0] = first_(y);
  l[1] = second_(x);
  r[1] = second_(y);
  ppm_limit(l[0], r[0]);
  ppm_limit(l[1], r[1]);
}

// The same for the five values of consecutive cells a, b, c, d, e, and the centre slopes D = l + r
// (double-float: values 0, 1 and 2, 3 in packed FP32).
template <class R>
__device__ __forceinline__ void ppm_edges5(const R a[5], const R b[5], const R c[5], const R d[5], const R e[5],
                                           R sixth, R l[5], R r[5], R D[5]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) ppm_edge(b[v] - a[v], c[v] - b[v], d[v] - c[v], e[v] - d[v], sixth, l[v], r[v]);
  add5(l, r, D);
}
// Float forms the edges themselves (Colella & Woodward's constraints as printed): mixed precision keeps
// the roundings of its float arithmetic in a double state, so they are part of its results.
__device__ __forceinline__ void ppm_edges5(const float a[5], const float b[5], const float c[5], const float d[5],
                                           const float e[5], float sixth, float l[5], float r[5], float D[5]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const float sb = mc_slope(b[v] - a[v], c[v] - b[v]), sc = mc_slope(c[v] - b[v], d[v] - c[v]),
                sd = mc_slope(d[v] - c[v], e[v] - d[v]);
    float qL = (b[v] + half_(c[v] - b[v])) - (sc - sb) * sixth;
    float qR = (c[v] + half_(d[v] - c[v])) - (sd - sc) * sixth;
    if (prod_nonpos(qR - c[v], c[v] - qL)) {
      qL = qR = c[v];
    } else {
      const float S = qR - qL, Q6 = mulf_(c[v] - half_(qL + qR), 6.f);
      const float SQ = S * Q6, SS = S * S;
      if (SQ > SS)
        qL = mulf_(c[v], 3.f) - twice_(qR);
      else if (-SS > SQ)
        qR = mulf_(c[v], 3.f) - twice_(qL);
    }
    D[v] = qR - qL;
    l[v] = c[v] - qL;
    r[v] = qR - c[v];
  }
}
__device__ __forceinline__ void ppm_edges5(const df a[5], const df b[5], const df c[5], const df d[5], const df e[5],
                                           df sixth, df l[5], df r[5], df D[5]) {
#pragma unroll
  for (int v = 0; v < 4; v += 2) {
    const df2 A = pair_(a[v], a[v + 1]), B = pair_(b[v], b[v + 1]), C = pair_(c[v], c[v + 1]),
              G = pair_(d[v], d[v + 1]), E = pair_(e[v], e[v + 1]);
    ppm_edge(B - A, C - B, G - C, E - G, sixth, l + v, r + v);
  }
  ppm_edge(b[4] - a[4], c[4] - b[4], d[4] - c[4], e[4] - d[4], sixth, l[4], r[4]);
  add5(l, r, D);
}

// Edge distances of tile cell (i, j) of the middle plane along axis d (0 x, 1 y, 2 z); q: the cell's
// own values.  sl: ring slots of planes p-2 .. p+2.
template <class R, class Sh>
__device__ __forceinline__ void ppm_axis(const Sh& sm, const int sl[5], int i, int j, int d,
                                         const R q[5], R sixth, R l[5], R r[5], R D[5]) {
  const int X = i + kPpmHalo, Y = j + kPpmHalo, dx = d == 0, dy = d == 1;
  R a[5], b[5], e[5], f[5];
  sm.q[d == 2 ? sl[0] : sl[2]].ld(Y - 2 * dy, X - 2 * dx, a);
  sm.q[d == 2 ? sl[1] : sl[2]].ld(Y - dy, X - dx, b);
  sm.q[d == 2 ? sl[3] : sl[2]].ld(Y + dy, X + dx, e);
  sm.q[d == 2 ? sl[4] : sl[2]].ld(Y + 2 * dy, X + 2 * dx, f);
  ppm_edges5(a, b, q, e, f, sixth, l, r, D);
}

// Edge distances of tile cell (i, j) along x, y and z, and the Hancock-predicted state qh.
template <class R, int TX, int TY>
__device__ __forceinline__ void ppm_cell(const PpmShared<R, TX, TY>& sm, const int sl[5], int i, int j, R gamma,
                                         R hdt, R sixth, R l[3][5], R r[3][5], R qh[5]) {
  R q[5], D[3][5];
  sm.q[sl[2]].ld(j + kPpmHalo, i + kPpmHalo, q);
#pragma unroll
  for (int d = 0; d < 3; ++d) ppm_axis(sm, sl, i, j, d, q, sixth, l[d], r[d], D[d]);
  hancock(q, D[0], D[1], D[2], gamma, hdt, qh);
}

// Resident blocks per SM: the 8-byte ring and face arrays take ~165 KB of shared memory.
template <class Pol>
constexpr int ppm_min_blocks() { return sizeof(typename Pol::R) >= 8 ? 1 : 2; }

// Block-wide maximum of v (all threads call); the result is valid in thread 0.
template <class R, class Sh>
__device__ __forceinline__ R ppm_block_max(Sh& sm, R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    R w = shfl_xor_(v, o);
    v = w > v ? w : v;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < (int)(blockDim.x / 32); ++w) v = sm.red[w] > v ? sm.red[w] : v;
  return v;
}

// Columns [x0, x0+TX) x rows [y0, y0+TY) x planes [z0, z1) of patch P (P.gin == 0: a periodic box;
// P.gin == 3: ghost layers filled by the caller) stepped by dt; with want_cfl the largest CFL speed
// of the updated cells of this thread is folded into smax.
template <class Pol, int TX, int TY>
__device__ __forceinline__ void ppm_tile(PpmShared<typename Pol::R, TX, TY>& sm, const PatchIO<typename Pol::S>& P,
                                         int x0, int y0, int z0, int z1, const Params& prm, double dtv, bool want_cfl,
                                         unsigned& flags, typename Pol::R& smax) {
  using S = typename Pol::S;
  using R = typename Pol::R;
  constexpr int QX = TX + 2 * kPpmHalo, QY = TY + 2 * kPpmHalo, NT = TX * TY;
  const int tid = threadIdx.x;
  const bool periodic = P.gin == 0;
  __syncthreads();  // the previous tile's last reads of the index tables are done
  for (int k = tid; k < QX; k += NT)
    sm.sx[k] = periodic ? wrap_index(x0 + k - kPpmHalo, P.nx) : min(x0 + k - kPpmHalo + P.gin, P.nx + 2 * P.gin - 1);
  for (int k = tid; k < QY; k += NT)
    sm.sy[k] = periodic ? wrap_index(y0 + k - kPpmHalo, P.ny) : min(y0 + k - kPpmHalo + P.gin, P.ny + 2 * P.gin - 1);
  __syncthreads();
  const R gamma = kc<R>(prm, K_GAMMA), igm1 = kc<R>(prm, K_IGM1), sixth = kc<R>(prm, K_SIXTH);
  const R rf = kc<R>(prm, K_RHOF), pf = kc<R>(prm, K_PF);
  const R hdt = (R)(0.5 * dtv / P.dx);
  const R dtdx = (R)(dtv / P.dx);

  // plane z of the patch (wrapped, or within the ghost layers), recovered into ring slot s over
  // the tile and its halo
  auto load_plane = [&](int z, int s, int first, int stride) {
    const long long zo = (long long)(periodic ? wrap_index(z, P.nz) : z + P.gin) * P.isz;
    for (int c = first; c < QX * QY; c += stride) {
      const int y = c / QX, x = c - y * QX;
      const long long a = zo + (long long)sm.sy[y] * P.isy + sm.sx[x];
      S U[5];
      R q[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = __ldg(P.in[v] + a);
      Pol::recover(U, prm, q, flags);
      sm.q[s].st(y, x, q);
    }
  };
  // slot of plane z: (z - z0 + 3) mod 5
  for (int k = 0; k < 5; ++k) load_plane(z0 - kPpmHalo + k, k, tid, NT);
  __syncthreads();

  const int i = tid % TX, j = tid / TX;
  const bool own = x0 + i < P.nx && y0 + j < P.ny;
  // ring cell of this thread: x-low (i = -1), x-high (i = TX), y-low (j = -1), y-high (j = TY)
  int rk = -1, ri = 0, rj = 0;
  if (tid < TY) { rk = 0; ri = -1; rj = tid; }
  else if (tid < 2 * TY) { rk = 1; ri = TX; rj = tid - TY; }
  else if (tid < 2 * TY + TX) { rk = 2; ri = tid - 2 * TY; rj = -1; }
  else if (tid < 2 * TY + 2 * TX) { rk = 3; ri = tid - 2 * TY - TX; rj = TY; }

  R zhi[5], fzb[5], dxy[5];  // z-high face state, z flux below, x/y flux difference: plane p-1
#pragma unroll
  for (int v = 0; v < 5; ++v) zhi[v] = fzb[v] = dxy[v] = R(0);
  auto xy_div = [&]() {
    R xp[5], xm[5], yp[5], ym[5];
    sm.fx.ld(j, i + 1, xp);
    sm.fx.ld(j, i, xm);
    sm.fy.ld(j + 1, i, yp);
    sm.fy.ld(j, i, ym);
    div_xy(xp, xm, yp, ym, dxy);
  };
  for (int p = z0 - 1; p <= z1; ++p) {
    const int base = p - z0 + 1;
    int sl[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) sl[k] = (base + k) % 5;
    const bool xy = p >= z0 && p < z1;  // plane p is updated: its x and y faces are needed
    R zlo[5], znew[5];
    // z face p - 1/2, then the update of plane p - 1 (its faces p - 3/2 and p - 1/2 are known)
    auto zface_update = [&]() {
      if (p > z0 - 1) {
        R ql[5], qr[5], F[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          ql[v] = zhi[v];
          qr[v] = zlo[v];
        }
        floor_max(ql, rf, pf);
        floor_max(qr, rf, pf);
        hllc<2>(ql, qr, gamma, igm1, F);
        if (p > z0 && own) {
          const int z = p - 1;
          const long long ai = (long long)(z + P.gin) * P.isz + (long long)(y0 + j + P.gin) * P.isy + (x0 + i + P.gin);
          const long long ao = (long long)(z + P.gout) * P.osz + (long long)(y0 + j + P.gout) * P.osy + (x0 + i + P.gout);
          S Uo[5], Un[5];
          R dz[5];
          sub5(F, fzb, dz);
          add5(dxy, dz, dxy);
#pragma unroll
          for (int v = 0; v < 5; ++v) Uo[v] = __ldg(P.in[v] + ai);
          Pol::update5(Uo, dtdx, dxy, Un);
#pragma unroll
          for (int v = 0; v < 5; ++v) P.out[v][ao] = Un[v];
          if (want_cfl) {
            const R sp = Pol::speed(Un, prm, flags);
            smax = sp > smax ? sp : smax;
          }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) fzb[v] = F[v];
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) zhi[v] = znew[v];
    };
    {
      R l[3][5], r[3][5], qh[5];
      ppm_cell(sm, sl, i, j, gamma, hdt, sixth, l, r, qh);
      sub5(qh, l[2], zlo);
      add5(qh, r[2], znew);
      if (xy) {
        sub5(qh, l[0], l[0]);
        add5(qh, r[0], r[0]);
        sub5(qh, l[1], l[1]);
        add5(qh, r[1], r[1]);
        sm.wx[0].st(j, i + 1, l[0]);
        sm.wx[1].st(j, i + 1, r[0]);
        sm.wy[0].st(j + 1, i, l[1]);
        sm.wy[1].st(j + 1, i, r[1]);
      }
    }
    if (xy && rk >= 0) {
      R l[3][5], r[3][5], qh[5], w[5];
      ppm_cell(sm, sl, ri, rj, gamma, hdt, sixth, l, r, qh);
#pragma unroll
      for (int v = 0; v < 5; ++v)
        w[v] = rk == 0 ? qh[v] + r[0][v] : (rk == 1 ? qh[v] - l[0][v] : (rk == 2 ? qh[v] + r[1][v] : qh[v] - l[1][v]));
      if (rk == 0) sm.wx[1].st(rj, 0, w);
      else if (rk == 1) sm.wx[0].st(rj, TX + 1, w);
      else if (rk == 2) sm.wy[1].st(0, ri, w);
      else sm.wy[0].st(TY + 1, ri, w);
    }
    zface_update();
    __syncthreads();  // face states written; ring slot of plane p-2 free
    if (xy) {
      for (int f = tid; f < (TX + 1) * TY; f += NT) {
        const int fy = f / (TX + 1), fx = f - fy * (TX + 1);
        R ql[5], qr[5], F[5];
        sm.wx[1].ld(fy, fx, ql);
        sm.wx[0].ld(fy, fx + 1, qr);
        floor_max(ql, rf, pf);
        floor_max(qr, rf, pf);
        hllc<0>(ql, qr, gamma, igm1, F);
        sm.fx.st(fy, fx, F);
      }
      for (int f = tid; f < TX * (TY + 1); f += NT) {
        const int fy = f / TX, fx = f - fy * TX;
        R ql[5], qr[5], F[5];
        sm.wy[1].ld(fy, fx, ql);
        sm.wy[0].ld(fy + 1, fx, qr);
        floor_max(ql, rf, pf);
        floor_max(qr, rf, pf);
        hllc<1>(ql, qr, gamma, igm1, F);
        sm.fy.st(fy, fx, F);
      }
    }
    if (p < z1) load_plane(p + kPpmHalo, sl[0], tid, NT);
    __syncthreads();  // fluxes and plane p+3 in place
    if (xy) xy_div();
  }
}

// ------------------------------------------------------------------ 8-byte tile
// Double-float and double run the same tile with 512 threads.  One thread per column left 8 warps per SM
// (the five-plane ring fills the SM's shared memory) with ~11000 dependent instructions each per plane:
// the double-float kernel waited on latencies at 36% of its issue slots.  Here a plane takes three phases between block
// barriers, and the first two split a cell's work:
//   A  the edge reconstructions, one (cell, axis) per thread: 768 of the tile's cells and, where plane
//      p's x and y faces are needed, 192 of the ring's; edge distances to shared memory
//   B  the first 256 threads: predictor, face states, z face p - 1/2 and the update of plane p - 1;
//      the others: the ring cells' predictor and face states, and the load of plane p + 3 into the
//      slot of plane p - 2
//   C  the 544 x and y faces
// 191x203x187 double-float step: 7.7 -> 4.0 ms (2.8 with branch-free comparisons); 96^3 double (FP64
// pipe): 2.83 -> 2.46 ms.
template <class R, int TX, int TY>
struct PpmWideShared {
  static constexpr int QX = TX + 2 * kPpmHalo, QY = TY + 2 * kPpmHalo;
  Plane5<R, QY, QX> q[5];       // ring of recovered planes
  Plane5<R, TY, TX + 2> wx[2];  // x faces: [low/high] edge distances, then states, at (y, x + 1)
  Plane5<R, TY + 2, TX> wy[2];  // y faces, at (y + 1, x)
  Plane5<R, TY, TX> wz[2];      // z edge distances of the tile's cells
  Plane5<R, 3, 2 * (TX + TY)> slope;  // the ring cells' centre slopes, [axis][ring cell]
  Plane5<R, TY, TX + 1> fx;
  Plane5<R, TY + 1, TX> fy;
  int sx[QX], sy[QY];
  R red[2 * TX * TY / 32];
  int tile;
};

template <class Pol, int TX, int TY>
__device__ __forceinline__ void ppm_tile(PpmWideShared<typename Pol::R, TX, TY>& sm, const PatchIO<double>& P, int x0,
                                         int y0, int z0, int z1, const Params& prm, double dtv, bool want_cfl,
                                         unsigned& flags, typename Pol::R& smax) {
  using R = typename Pol::R;
  constexpr int QX = TX + 2 * kPpmHalo, QY = TY + 2 * kPpmHalo, NC = TX * TY, NT = 2 * NC, NR = 2 * (TX + TY);
  static_assert(NC % 32 == 0 && NR % 32 == 0 && NR <= NC, "whole warps per axis and per role");
  const int tid = threadIdx.x;
  const bool periodic = P.gin == 0;
  __syncthreads();  // the previous tile's last reads of the index tables are done
  for (int k = tid; k < QX; k += NT)
    sm.sx[k] = periodic ? wrap_index(x0 + k - kPpmHalo, P.nx) : min(x0 + k - kPpmHalo + P.gin, P.nx + 2 * P.gin - 1);
  for (int k = tid; k < QY; k += NT)
    sm.sy[k] = periodic ? wrap_index(y0 + k - kPpmHalo, P.ny) : min(y0 + k - kPpmHalo + P.gin, P.ny + 2 * P.gin - 1);
  __syncthreads();
  const R gamma = kc<R>(prm, K_GAMMA), igm1 = kc<R>(prm, K_IGM1), sixth = kc<R>(prm, K_SIXTH);
  const R rf = kc<R>(prm, K_RHOF), pf = kc<R>(prm, K_PF);
  const R hdt = (R)(0.5 * dtv / P.dx);
  const R dtdx = (R)(dtv / P.dx);
  auto load_plane = [&](int z, int s, int first, int stride) {
    const long long zo = (long long)(periodic ? wrap_index(z, P.nz) : z + P.gin) * P.isz;
    for (int c = first; c < QX * QY; c += stride) {
      const int y = c / QX, x = c - y * QX;
      const long long a = zo + (long long)sm.sy[y] * P.isy + sm.sx[x];
      double U[5];
      R q[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = __ldg(P.in[v] + a);
      Pol::recover(U, prm, q, flags);
      sm.q[s].st(y, x, q);
    }
  };
  // ring cell r: x-low, x-high, y-low, y-high sides in turn
  auto ring_cell = [&](int r, int& side, int& i, int& j) {
    if (r < TY) { side = 0; i = -1; j = r; }
    else if (r < 2 * TY) { side = 1; i = TX; j = r - TY; }
    else if (r < 2 * TY + TX) { side = 2; i = r - 2 * TY; j = -1; }
    else { side = 3; i = r - 2 * TY - TX; j = TY; }
  };
  for (int k = 0; k < 5; ++k) load_plane(z0 - kPpmHalo + k, k, tid, NT);  // slot of plane z: (z - z0 + 3) mod 5
  __syncthreads();

  const int i = tid % TX, j = (tid % NC) / TX;  // column of the first NC threads
  const bool column = tid < NC, own = column && x0 + i < P.nx && y0 + j < P.ny;
  R zhi[5], fzb[5];  // z-high face state of plane p-1 and z flux below it
#pragma unroll
  for (int v = 0; v < 5; ++v) zhi[v] = fzb[v] = R(0);
  for (int p = z0 - 1; p <= z1; ++p) {
    const int base = p - z0 + 1;
    int sl[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) sl[k] = (base + k) % 5;
    const bool xy = p >= z0 && p < z1;  // plane p is updated: its x and y faces are needed
    // ---- A
    for (int t = tid; t < 3 * (xy ? NC + NR : NC); t += NT) {
      const bool ring = t >= 3 * NC;
      const int d = ring ? (t - 3 * NC) / NR : t / NC, c = ring ? (t - 3 * NC) % NR : t % NC;
      int ci = c % TX, cj = c / TX, side = 0;
      if (ring) ring_cell(c, side, ci, cj);
      R q[5], l[5], r[5], D[5];
      sm.q[sl[2]].ld(cj + kPpmHalo, ci + kPpmHalo, q);
      ppm_axis(sm, sl, ci, cj, d, q, sixth, l, r, D);
      if (ring) {
        sm.slope.st(d, c, D);
        if (d == (side >> 1)) {
          if (side == 0) sm.wx[1].st(cj, 0, r);
          else if (side == 1) sm.wx[0].st(cj, TX + 1, l);
          else if (side == 2) sm.wy[1].st(0, ci, r);
          else sm.wy[0].st(TY + 1, ci, l);
        }
      } else if (d == 0) {
        sm.wx[0].st(cj, ci + 1, l);
        sm.wx[1].st(cj, ci + 1, r);
      } else if (d == 1) {
        sm.wy[0].st(cj + 1, ci, l);
        sm.wy[1].st(cj + 1, ci, r);
      } else {
        sm.wz[0].st(cj, ci, l);
        sm.wz[1].st(cj, ci, r);
      }
    }
    __syncthreads();
    // ---- B
    auto low = [&](const R qh[5], auto& w, int y, int x) {  // edge distance -> face state
      R t[5];
      w.ld(y, x, t);
      sub5(qh, t, t);
      w.st(y, x, t);
    };
    auto high = [&](const R qh[5], auto& w, int y, int x) {
      R t[5];
      w.ld(y, x, t);
      add5(qh, t, t);
      w.st(y, x, t);
    };
    if (column) {
      R q[5], D[3][5], l[5], qh[5];
      sm.q[sl[2]].ld(j + kPpmHalo, i + kPpmHalo, q);
      sm.wx[0].ld(j, i + 1, l);
      sm.wx[1].ld(j, i + 1, D[0]);
      add5(l, D[0], D[0]);
      sm.wy[0].ld(j + 1, i, l);
      sm.wy[1].ld(j + 1, i, D[1]);
      add5(l, D[1], D[1]);
      sm.wz[0].ld(j, i, l);
      sm.wz[1].ld(j, i, D[2]);
      add5(l, D[2], D[2]);
      hancock(q, D[0], D[1], D[2], gamma, hdt, qh);
      if (xy) {
        low(qh, sm.wx[0], j, i + 1);
        high(qh, sm.wx[1], j, i + 1);
        low(qh, sm.wy[0], j + 1, i);
        high(qh, sm.wy[1], j + 1, i);
      }
      R zlo[5], znew[5];
      sm.wz[0].ld(j, i, zlo);
      sm.wz[1].ld(j, i, znew);
      sub5(qh, zlo, zlo);
      add5(qh, znew, znew);
      if (p > z0 - 1) {
        R F[5];
        floor_max(zhi, rf, pf);
        floor_max(zlo, rf, pf);
        hllc<2>(zhi, zlo, gamma, igm1, F);
        if (p > z0) {
          R xp[5], xm[5], yp[5], ym[5], div[5];  // plane p-1's x and y fluxes
          sm.fx.ld(j, i + 1, xp);
          sm.fx.ld(j, i, xm);
          sm.fy.ld(j + 1, i, yp);
          sm.fy.ld(j, i, ym);
          div_xy(xp, xm, yp, ym, div);
          sub5(F, fzb, xp);
          add5(div, xp, div);
          if (own) {
            const int z = p - 1;
            const long long ai = (long long)(z + P.gin) * P.isz + (long long)(y0 + j + P.gin) * P.isy + (x0 + i + P.gin);
            const long long ao = (long long)(z + P.gout) * P.osz + (long long)(y0 + j + P.gout) * P.osy + (x0 + i + P.gout);
            double Uo[5], Un[5];
#pragma unroll
            for (int v = 0; v < 5; ++v) Uo[v] = __ldg(P.in[v] + ai);
            Pol::update5(Uo, dtdx, div, Un);
#pragma unroll
            for (int v = 0; v < 5; ++v) P.out[v][ao] = Un[v];
            if (want_cfl) {
              const R sp = Pol::speed(Un, prm, flags);
              smax = sp > smax ? sp : smax;
            }
          }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) fzb[v] = F[v];
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) zhi[v] = znew[v];
    } else {
      const int u = tid - NC;
      if (xy && u < NR) {
        int side, ci, cj;
        ring_cell(u, side, ci, cj);
        R q[5], D[3][5], qh[5];
        sm.q[sl[2]].ld(cj + kPpmHalo, ci + kPpmHalo, q);
#pragma unroll
        for (int d = 0; d < 3; ++d) sm.slope.ld(d, u, D[d]);
        hancock(q, D[0], D[1], D[2], gamma, hdt, qh);
        if (side == 0) high(qh, sm.wx[1], cj, 0);
        else if (side == 1) low(qh, sm.wx[0], cj, TX + 1);
        else if (side == 2) high(qh, sm.wy[1], 0, ci);
        else low(qh, sm.wy[0], TY + 1, ci);
      }
      // the threads without a ring cell come first, where some take a cell more
      if (p < z1) load_plane(p + kPpmHalo, sl[0], NC - 1 - u, NC);
    }
    __syncthreads();
    // ---- C
    if (xy) {
      constexpr int NXF = (TX + 1) * TY;
      for (int f = tid; f < NXF + TX * (TY + 1); f += NT) {
        const int d = f < NXF ? 0 : 1, g = d == 0 ? f : f - NXF, w = d == 0 ? TX + 1 : TX;
        const int fy = g / w, fx = g - fy * w;
        R ql[5], qr[5], F[5];
        if (d == 0) {
          sm.wx[1].ld(fy, fx, ql);
          sm.wx[0].ld(fy, fx + 1, qr);
        } else {
          sm.wy[1].ld(fy, fx, ql);
          sm.wy[0].ld(fy + 1, fx, qr);
        }
        floor_max(ql, rf, pf);
        floor_max(qr, rf, pf);
        hllc_dyn(d, ql, qr, gamma, igm1, F);
        if (d == 0) sm.fx.st(fy, fx, F);
        else sm.fy.st(fy, fx, F);
      }
    }
    __syncthreads();
  }
}

// The tile's shared memory and block size by policy.
template <class Pol, int TX, int TY>
using PpmTileShared = typename std::conditional<sizeof(typename Pol::R) >= 8, PpmWideShared<typename Pol::R, TX, TY>,
                                                PpmShared<typename Pol::R, TX, TY>>::type;
template <class Pol, int TX, int TY>
constexpr int ppm_threads() { return sizeof(typename Pol::R) >= 8 ? 2 * TX * TY : TX * TY; }

// Periodic box: one tile per block, tiles from the block index.
template <class Pol, int TX, int TY>
__global__ void __launch_bounds__((ppm_threads<Pol, TX, TY>()), ppm_min_blocks<Pol>())
    k_step_ppm(PatchIO<typename Pol::S> P, Params prm, const double* dt_dev, double* dt_next, int zchunk,
               unsigned* err) {
  using R = typename Pol::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<PpmTileShared<Pol, TX, TY>*>(smem_raw);
  const double dt = dt_dev[0];
  if (!(dt > 0.0 && dt <= 1e300)) {
    if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) atomicOr(err, HYDRO_EBIT_BAD_DT);
    return;
  }
  unsigned flags = 0;
  R smax = 0;
  const int z0 = blockIdx.z * zchunk;
  ppm_tile<Pol, TX, TY>(sm, P, blockIdx.x * TX, blockIdx.y * TY, z0, min(z0 + zchunk, P.nz), prm, dt,
                        dt_next != nullptr, flags, smax);
  if (dt_next) {
    const R m = ppm_block_max(sm, smax);
    if (threadIdx.x == 0) publish_dt(prm.cfl, P.dx, (double)m, dt_next);
  }
  flush_flags(flags, err);
}

// Patches with three ghost layers: a persistent grid taking tiles from the device work-list by an
// atomic counter (as the PLM batched kernel); per-patch dt, dx and dt_next.
template <class Pol, int TX, int TY>
__global__ void __launch_bounds__((ppm_threads<Pol, TX, TY>()), ppm_min_blocks<Pol>())
    k_step_ppm_batched(const PatchIO<typename Pol::S>* patches, const TileRec* tiles, int ntiles, int* counter,
                       Params prm, const double* dt_dev, double* dt_next, int zchunk, unsigned* err) {
  using R = typename Pol::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<PpmTileShared<Pol, TX, TY>*>(smem_raw);
  unsigned flags = 0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) sm.tile = atomicAdd(counter, 1);
    __syncthreads();
    const int t = sm.tile;
    if (t >= ntiles) break;
    const TileRec r = tiles[t];
    const PatchIO<typename Pol::S> P = patches[r.patch];
    if (r.x0 < 0 || r.y0 < 0 || r.z0 < 0 || r.x0 >= P.nx || r.y0 >= P.ny || r.z0 >= P.nz || P.gin != kPpmHalo) {
      flags |= HYDRO_EBIT_BAD_TILE;
      continue;
    }
    const double dt = dt_dev[r.patch];
    if (!(dt > 0.0 && dt <= 1e300)) {
      flags |= HYDRO_EBIT_BAD_DT;
      continue;
    }
    R smax = 0;
    ppm_tile<Pol, TX, TY>(sm, P, r.x0, r.y0, r.z0, min(r.z0 + zchunk, P.nz), prm, dt, dt_next != nullptr, flags,
                          smax);
    if (dt_next) {
      const R m = ppm_block_max(sm, smax);
      if (threadIdx.x == 0) publish_dt(prm.cfl, P.dx, (double)m, dt_next + r.patch);
    }
  }
  flush_flags(flags, err);
}

constexpr int kPpmTX = 16, kPpmTY = 16;
static_assert(kTileX[0] == kPpmTX && kTileY[0] == kPpmTY, "the PPM work-list is built with tile shape 0");

template <class Pol>
cudaError_t ppm_attr(const void* fn) {
  const size_t smem = sizeof(PpmTileShared<Pol, kPpmTX, kPpmTY>);
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <class Pol>
cudaError_t launch_ppm(const HostPatchIO& P, const Params& prm, const double* dt, double* dt_next, int zchunk,
                       unsigned* err, cudaStream_t s) {
  static PerDeviceOnce attr;
  cudaError_t ea = attr.call([&] { return ppm_attr<Pol>(reinterpret_cast<const void*>(k_step_ppm<Pol, kPpmTX, kPpmTY>)); });
  if (ea != cudaSuccess) return ea;
  const size_t smem = sizeof(PpmTileShared<Pol, kPpmTX, kPpmTY>);
  dim3 grid((P.nx + kPpmTX - 1) / kPpmTX, (P.ny + kPpmTY - 1) / kPpmTY, (P.nz + zchunk - 1) / zchunk);
  k_step_ppm<Pol, kPpmTX, kPpmTY><<<grid, ppm_threads<Pol, kPpmTX, kPpmTY>(), smem, s>>>(to_dev<Pol>(P), prm, dt, dt_next, zchunk, err);
  return cudaGetLastError();
}

template <class Pol>
cudaError_t launch_ppm_batched(const HostPatchIO* d_patches, const HostTileRec* d_tiles, int ntiles, int* d_counter,
                               const Params& prm, const double* dt, double* dt_next, int zchunk, unsigned* err,
                               int sm_count, cudaStream_t s) {
  using K = decltype(&k_step_ppm_batched<Pol, kPpmTX, kPpmTY>);
  const K fn = &k_step_ppm_batched<Pol, kPpmTX, kPpmTY>;
  static PerDeviceOnce attr;
  cudaError_t ea = attr.call([&] { return ppm_attr<Pol>(reinterpret_cast<const void*>(fn)); });
  if (ea != cudaSuccess) return ea;
  const size_t smem = sizeof(PpmTileShared<Pol, kPpmTX, kPpmTY>);
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, ppm_threads<Pol, kPpmTX, kPpmTY>(), smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  const int grid = std::max(1, std::min(ntiles, sm_count * per_sm));
  fn<<<grid, ppm_threads<Pol, kPpmTX, kPpmTY>(), smem, s>>>(reinterpret_cast<const PatchIO<typename Pol::S>*>(d_patches),
                                         reinterpret_cast<const TileRec*>(d_tiles), ntiles, d_counter, prm, dt,
                                         dt_next, zchunk, err);
  return cudaGetLastError();
}

}  // namespace hydro
