// Kernels and launchers of one precision policy POL (included once per policy by kernels_*.cu):
// the step kernels of step_tile.cuh for every compiled tile shape, the PPM step of step_ppm.cuh,
// the standalone CFL dt
// reduction, the oct-group step, the primitive->conservative map and its adjoint, and the
// adjoint step (adjoint.cuh).
#pragma once
#include "adjoint.cuh"
#include "internal.h"
#include "oct_cube.cuh"
#include "step_ppm.cuh"
#include "step_tile.cuh"

namespace hydro {

// ------------------------------------------------------------------ step launchers
// The step kernels are compiled once per PLM limiter (LIM: HYDRO_MINMOD, HYDRO_MC, HYDRO_NOLIMIT).

template <class Pol, int TX, int TY, int MINB, int LIM>
cudaError_t launch_uniform_t(const HostPatchIO& P, const Params& prm, const double* dt, double* dt_next, int zchunk,
                             unsigned* err, cudaStream_t s) {
  const size_t smem = sizeof(TileShared<Pol, TX, TY>);
  static PerDeviceOnce attr;
  cudaError_t e = attr.call([&] {
    return cudaFuncSetAttribute(k_step_uniform<Pol, TX, TY, MINB, LIM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem);
  });
  if (e != cudaSuccess) return e;
  dim3 grid((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY, (P.nz + zchunk - 1) / zchunk);
  k_step_uniform<Pol, TX, TY, MINB, LIM><<<grid, TX * TY, smem, s>>>(to_dev<Pol>(P), prm, dt, dt_next, zchunk, err);
  return cudaGetLastError();
}

template <class Pol, int TX, int TY, int MINB, int LIM>
cudaError_t launch_batched_t(const HostPatchIO* d_patches, const HostTileRec* d_tiles, int ntiles, int* d_counter,
                             const Params& prm, const double* dt, double* dt_next, int zchunk, unsigned* err, int grid,
                             cudaStream_t s) {
  const size_t smem = sizeof(TileShared<Pol, TX, TY>);
  static PerDeviceOnce attr;
  cudaError_t e = attr.call([&] {
    return cudaFuncSetAttribute(k_step_batched<Pol, TX, TY, MINB, LIM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem);
  });
  if (e != cudaSuccess) return e;
  k_step_batched<Pol, TX, TY, MINB, LIM><<<grid, TX * TY, smem, s>>>(
      reinterpret_cast<const PatchIO<typename Pol::S>*>(d_patches), reinterpret_cast<const TileRec*>(d_tiles), ntiles,
      d_counter, prm, dt, dt_next, zchunk, err);
  return cudaGetLastError();
}

template <class Pol, int TX, int TY, int MINB, int LIM>
int blocks_per_sm_t() {
  const size_t smem = sizeof(TileShared<Pol, TX, TY>);
  cudaFuncSetAttribute(k_step_batched<Pol, TX, TY, MINB, LIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_step_batched<Pol, TX, TY, MINB, LIM>, TX * TY, smem) !=
      cudaSuccess)
    return 1;
  return n > 0 ? n : 1;
}

// Tile id -> compiled shape, and the limiter -> compiled variant.
#define HYDRO_LIM_SWITCH(T, lim, CALL)                     \
  (lim == HYDRO_MINMOD ? CALL(T, HYDRO_MINMOD)             \
                       : lim == HYDRO_MC ? CALL(T, HYDRO_MC) : CALL(T, HYDRO_NOLIMIT))
#define HYDRO_TILE_SWITCH(tile, lim, CALL)                    \
  switch (tile) {                                             \
    case 0: return HYDRO_LIM_SWITCH(0, lim, CALL);           \
    case 1: return HYDRO_LIM_SWITCH(1, lim, CALL);           \
    case 2: return HYDRO_LIM_SWITCH(2, lim, CALL);           \
    case 3: return HYDRO_LIM_SWITCH(3, lim, CALL);           \
    case 4: return HYDRO_LIM_SWITCH(4, lim, CALL);           \
  }

template <class Pol>
cudaError_t launch_uniform(int tile, const HostPatchIO& P, const Params& prm, const double* dt, double* dt_next,
                           int zchunk, unsigned* err, cudaStream_t s) {
#define HYDRO_CALL(T, L) launch_uniform_t<Pol, kTileX[T], kTileY[T], kTileMinBlocks[T], L>(P, prm, dt, dt_next, zchunk, err, s)
  HYDRO_TILE_SWITCH(tile, prm.limiter, HYDRO_CALL)
#undef HYDRO_CALL
  return cudaErrorInvalidValue;
}

template <class Pol>
cudaError_t launch_batched(int tile, const HostPatchIO* d_patches, const HostTileRec* d_tiles, int ntiles,
                           int* d_counter, const Params& prm, const double* dt, double* dt_next, int zchunk,
                           unsigned* err, int grid, cudaStream_t s) {
#define HYDRO_CALL(T, L)                                                                                          \
  launch_batched_t<Pol, kTileX[T], kTileY[T], kTileMinBlocks[T], L>(d_patches, d_tiles, ntiles, d_counter, prm, dt, \
                                                                    dt_next, zchunk, err, grid, s)
  HYDRO_TILE_SWITCH(tile, prm.limiter, HYDRO_CALL)
#undef HYDRO_CALL
  return cudaErrorInvalidValue;
}

template <class Pol>
int batched_blocks_per_sm(int tile, int limiter) {
#define HYDRO_CALL(T, L) blocks_per_sm_t<Pol, kTileX[T], kTileY[T], kTileMinBlocks[T], L>()
  HYDRO_TILE_SWITCH(tile, limiter, HYDRO_CALL)
#undef HYDRO_CALL
  return 1;
}
#undef HYDRO_TILE_SWITCH
#undef HYDRO_LIM_SWITCH

// ------------------------------------------------------------------ CFL dt (standalone)
// blockIdx.y walks the patches, blockIdx.x the interior cells of one patch.  The per-block
// largest speed is reduced by warp shuffles and shared memory and folded into the patch's dt
// slot exactly as the step's fused epilogue does, so both give the same bits.
template <class Pol>
__global__ void __launch_bounds__(256) k_cfl(const PatchIO<typename Pol::S>* patches, PatchIO<typename Pol::S> single,
                                             int npatch, Params prm, double* dt_out, unsigned* err) {
  using S = typename Pol::S;
  using R = typename Pol::R;
  __shared__ R red[8];
  unsigned flags = 0;
  for (int pi = blockIdx.y; pi < npatch; pi += gridDim.y) {
    const PatchIO<S> P = patches ? patches[pi] : single;
    // cells by (row, x): rows = (z, y) pairs, one 32-bit division per row (64-bit integer division
    // is a long sequence that runs partly on the FP64 pipe)
    const int rows = P.ny * P.nz;
    R smax = 0;
    const int nxb = (P.nx + 31) / 32;  // 32-wide segments per row
    for (long long s = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); s < (long long)rows * nxb;
         s += (long long)gridDim.x * 8) {
      const int row = (int)(s / nxb), i = (int)(s - (long long)row * nxb) * 32 + (threadIdx.x & 31);
      if (i >= P.nx) continue;
      const int k = row / P.ny, j = row - k * P.ny;
      const long long a = (long long)(k + P.gin) * P.isz + (long long)(j + P.gin) * P.isy + (i + P.gin);
      S U[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = __ldg(P.in[v] + a);
      const R sp = Pol::speed(U, prm, flags);
      smax = sp > smax ? sp : smax;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      R w = shfl_xor_(smax, o);
      smax = w > smax ? w : smax;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = smax;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) smax = red[w] > smax ? red[w] : smax;
      publish_dt(prm.cfl, P.dx, (double)smax, dt_out + pi);
    }
  }
  flush_flags(flags, err);
}

template <class Pol>
cudaError_t launch_cfl(const HostPatchIO* d_patches, const HostPatchIO& single, int npatch, const Params& prm,
                       double* dt_out, unsigned* err, cudaStream_t s) {
  long long maxcells = (long long)single.nx * single.ny * single.nz;
  int gx;
  if (d_patches) {
    gx = 64;  // patches up to a few 10^5 cells
  } else {
    long long b = (maxcells + 256 * 4 - 1) / (256 * 4);
    gx = (int)(b < 1 ? 1 : (b > 152 * 16 ? 152 * 16 : b));
  }
  dim3 grid(gx, npatch < 65535 ? npatch : 65535);
  k_cfl<Pol><<<grid, 256, 0, s>>>(reinterpret_cast<const PatchIO<typename Pol::S>*>(d_patches), to_dev<Pol>(single),
                                  npatch, prm, dt_out, err);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ oct groups
// One warp per batch of groups.  Per group, the 80 cells of the 6^3 stencil that the step reads are
// recovered into shared memory; the 32 cells next to the oct's faces (the oct and the 24 outside
// neighbours across its faces) are predicted; 32 of the oct's 36 faces get their HLLC fluxes, one per
// lane.  The other four (the upper z faces) and the oct's 8 updates would leave most lanes idle, so
// they wait in shared memory for the batch's end: four groups' 16 left faces share one round and their 32
// updates fill one, where a group of its own took a second face round and an update round for itself (eight
// groups would fill the left faces' round too, but their scratch leaves too few warps per SM: 262144 groups,
// mixed, 558 us against 392).  Local coordinates run from -2 to 3 (stored at +2).
__device__ __forceinline__ bool oct_needed(int x, int y, int z) {
  const int ox = (x < 0 || x > 1), oy = (y < 0 || y > 1), oz = (z < 0 || z > 1);
  const int nout = ox + oy + oz;
  const bool far = (x == -2 || x == 3 || y == -2 || y == 3 || z == -2 || z == 3);
  return nout <= 1 || (nout == 2 && !far);
}
// Coordinates of predicted cell e (0..31): 0..7 the oct, 8..31 the face neighbours.
__device__ __forceinline__ void oct_ecell(int e, int& x, int& y, int& z) {
  if (e < 8) { x = e & 1; y = (e >> 1) & 1; z = (e >> 2) & 1; return; }
  const int r = e - 8, f = r >> 2, a = r & 1, b = (r >> 1) & 1;
  const int out = (f & 1) ? 2 : -1;
  const int d = f >> 1;
  x = d == 0 ? out : a;
  y = d == 1 ? out : (d == 0 ? a : b);
  z = d == 2 ? out : b;
}
__device__ __forceinline__ int oct_eindex(int x, int y, int z) {
  const bool ix = (x == 0 || x == 1), iy = (y == 0 || y == 1), iz = (z == 0 || z == 1);
  if (ix && iy && iz) return x + 2 * y + 4 * z;
  int d, c, a, b;
  if (!ix) { d = 0; c = x; a = y; b = z; }
  else if (!iy) { d = 1; c = y; a = x; b = z; }
  else { d = 2; c = z; a = x; b = y; }
  const int f = 2 * d + (c == 2 ? 1 : 0);
  return 8 + 4 * f + a + 2 * b;
}

constexpr int kOctWarps = 4;
constexpr int kOctBatch = 4;

template <class Pol>
struct OctSmem {
  using R = typename Pol::R;
  R q[kOctWarps][5][80];      // needed cells in the order of need[]
  R qh[kOctWarps][5][32];
  R sl[kOctWarps][3][5][32];  // kept slopes
  R f[kOctWarps][kOctBatch][5][36];
  R left[kOctWarps][kOctBatch][10][4];  // lower and upper states of the upper z faces
  short need[80], at[216];    // needed cell -> stencil cell, and back
};

// Where a group's 6^3 stencil comes from and where its 8 cells go.  OctGathered: the caller's
// gathered buffer, group g's cell c (z, y, x from -2) at g*216 + c.  OctLevel: a periodic level
// grid and the groups' origins (the oct's lowest cell, x, y, z), wrapped on the fly -- no gathered
// copy of the stencils.  Both write group g's cells at g*8 .. g*8+7.  OctTable: octs stored
// oct-major (cell (i, j, k) of oct o at o*8 + (k*2 + j)*2 + i) with their neighbour table; group g
// steps oct list[g] and writes it in place of that oct.
template <class S>
struct OctGathered {
  static constexpr bool kGathered = true;
  const S* f[5];
  __device__ __forceinline__ bool begin(long long, unsigned&) const { return true; }
  __device__ __forceinline__ long long cell(long long g, int c) const { return g * 216 + c; }
  // input and output index of cell e of group g's oct (any lane's own group, already found valid)
  __device__ __forceinline__ void own(long long g, int e, long long& in, long long& out) const {
    in = g * 216 + ((e >> 2) + 2) * 36 + (((e >> 1) & 1) + 2) * 6 + (e & 1) + 2;
    out = g * 8 + e;
  }
};
template <class S>
struct OctLevel {
  static constexpr bool kGathered = false;
  const S* f[5];
  int nx, ny, nz;
  long long sy, sz;
  const int* origins;  // [ngroups][3]
  int ox, oy, oz;      // origin of the current group
  // Loads group g's origin; an origin outside the grid flags HYDRO_EBIT_BAD_TILE and the group
  // is skipped (nothing is read or written for it).
  __device__ __forceinline__ bool begin(long long g, unsigned& flags) {
    ox = __ldg(origins + 3 * g);
    oy = __ldg(origins + 3 * g + 1);
    oz = __ldg(origins + 3 * g + 2);
    if (ox < 0 || oy < 0 || oz < 0 || ox >= nx || oy >= ny || oz >= nz) {
      flags |= HYDRO_EBIT_BAD_TILE;
      return false;
    }
    return true;
  }
  __device__ __forceinline__ long long cell(long long, int c) const {
    int x = ox + c % 6 - 2, y = oy + (c / 6) % 6 - 2, z = oz + c / 36 - 2;
    x += x < 0 ? nx : (x >= nx ? -nx : 0);
    y += y < 0 ? ny : (y >= ny ? -ny : 0);
    z += z < 0 ? nz : (z >= nz ? -nz : 0);
    return z * sz + y * sy + x;
  }
  __device__ __forceinline__ void own(long long g, int e, long long& in, long long& out) const {
    int x = __ldg(origins + 3 * g) + (e & 1), y = __ldg(origins + 3 * g + 1) + ((e >> 1) & 1),
        z = __ldg(origins + 3 * g + 2) + (e >> 2);
    x -= x >= nx ? nx : 0;
    y -= y >= ny ? ny : 0;
    z -= z >= nz ? nz : 0;
    in = z * sz + y * sy + x;
    out = g * 8 + e;
  }
};
template <class S>
struct OctTable {
  static constexpr bool kGathered = false;
  const S* f[5];
  const int* nbr;   // [noct][27]: oct at offset (dx, dy, dz) in entry ((dz+1)*3 + dy+1)*3 + dx+1
  const int* list;  // [ngroups]: the octs to step
  int noct;
  int oct;          // the current group's oct
  // Loads group g's oct and checks it and its 27 neighbour entries (one per lane, warp-wide):
  // an index outside [0, noct) flags HYDRO_EBIT_BAD_TILE and the group is skipped.
  __device__ __forceinline__ bool begin(long long g, unsigned& flags) {
    oct = __ldg(list + g);
    bool bad = (unsigned)oct >= (unsigned)noct;
    const int lane = threadIdx.x & 31;
    if (!bad && lane < 27) bad = (unsigned)__ldg(nbr + 27LL * oct + lane) >= (unsigned)noct;
    if (__any_sync(0xffffffffu, bad)) {
      flags |= HYDRO_EBIT_BAD_TILE;
      return false;
    }
    return true;
  }
  // Stencil cell (x, y, z), each 0..5, is cell (x%2, y%2, z%2) of neighbour (x/2, y/2, z/2).
  __device__ __forceinline__ long long cell(long long, int c) const {
    const int x = c % 6, y = (c / 6) % 6, z = c / 36;
    const int n = __ldg(nbr + 27LL * oct + ((z >> 1) * 3 + (y >> 1)) * 3 + (x >> 1));
    return 8LL * n + ((z & 1) * 2 + (y & 1)) * 2 + (x & 1);
  }
  __device__ __forceinline__ void own(long long g, int e, long long& in, long long& out) const {
    in = out = 8LL * __ldg(list + g) + e;
  }
};

// Resident blocks per SM: as many as the batch's scratch leaves room for, in float arithmetic six (80
// registers), five for the gathered buffer, whose prefetch spills at 80 (262144 groups, mixed: 392 us
// against 403, and 514 for a group at a time; the whole level through its table: 3.34 ms at six, 3.47 at five).
template <class Pol, class Src>
constexpr int oct_min_blocks() { return sizeof(typename Pol::R) >= 8 ? 3 : (Src::kGathered ? 5 : 6); }

template <class Pol, class Src>
__global__ void __launch_bounds__(32 * kOctWarps, (oct_min_blocks<Pol, Src>())) k_octs(Src src, typename Pol::S* o0, typename Pol::S* o1,
                                                         typename Pol::S* o2, typename Pol::S* o3,
                                                         typename Pol::S* o4, long long ngroups, const int* count, int batch, double dx,
                                                         Params prm,
                                                         const double* dt_dev, unsigned* err) {
  using S = typename Pol::S;
  using R = typename Pol::R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<OctSmem<Pol>*>(smem_raw);
  S* gout[5] = {o0, o1, o2, o3, o4};
  if (count) {  // groups left by the cube kernel: often none, and then only block 0 stays, to check dt
    ngroups = *count;
    if (blockIdx.x > 0 && (long long)blockIdx.x * kOctWarps * batch >= ngroups) return;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // needed cells numbered in stencil order: a ballot per 32 cells, the first warp's lanes together
  if (threadIdx.x < 32) {
    int n = 0;
    for (int c = lane; c < 224; c += 32) {
      const bool needed = c < 216 && oct_needed(c % 6 - 2, (c / 6) % 6 - 2, c / 36 - 2);
      const unsigned who = __ballot_sync(0xffffffffu, needed);
      const int k = n + __popc(who & ((1u << lane) - 1u));
      if (c < 216) sm.at[c] = (short)k;
      if (needed) sm.need[k] = (short)c;
      n += __popc(who);
    }
  }
  __syncthreads();
  const double dt = dt_dev[0];
  if (!(dt > 0.0 && dt <= 1e300)) {
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(err, HYDRO_EBIT_BAD_DT);
    return;
  }
  const R hdt = (R)(0.5 * dt / dx);
  const R dtdx = (R)(dt / dx);
  const R gamma = kc<R>(prm, K_GAMMA), igm1 = kc<R>(prm, K_IGM1);
  const R rf = kc<R>(prm, K_RHOF), pf = kc<R>(prm, K_PF);
  unsigned flags = 0;
  // This lane's predicted cell and its six neighbours among the needed cells, and its face.
  int pc, pn[3][2];
  {
    int x, y, z;
    oct_ecell(lane, x, y, z);
    const int c = (z + 2) * 36 + (y + 2) * 6 + (x + 2);
    pc = sm.at[c];
    pn[0][0] = sm.at[c - 1]; pn[0][1] = sm.at[c + 1];
    pn[1][0] = sm.at[c - 6]; pn[1][1] = sm.at[c + 6];
    pn[2][0] = sm.at[c - 36]; pn[2][1] = sm.at[c + 36];
  }
  // The upper z faces' normal, 2, kept from the compiler: the flux of a run-time normal rounds as the
  // other faces' (a fixed one contracts its kinetic sum differently).
  int dz = 2;
  asm("" : "+r"(dz));
  // face between cells at coordinate s-1 and s along d; (a, b) the transverse coordinates
  const int fd = lane / 12;
  int eL, eR;
  {
    const int m = lane % 12, s = m >> 2, a = m & 1, b = (m >> 1) & 1;
    const int lx = fd == 0 ? s - 1 : a, ly = fd == 1 ? s - 1 : (fd == 0 ? a : b), lz = fd == 2 ? s - 1 : b;
    eL = oct_eindex(lx, ly, lz);
    eR = oct_eindex(lx + (fd == 0), ly + (fd == 1), lz + (fd == 2));
  }
  // The needed cells of the next group are loaded into registers while this group is computed.
  const long long bstride = (long long)gridDim.x * kOctWarps * batch;
  S pre[3][5];
  Src nxt = src;  // source state of the prefetched group
  bool nxt_ok = false;
  auto fetch = [&](long long g) {
    nxt_ok = nxt.begin(g, flags);
    if (!nxt_ok) return;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int k = lane + 32 * t;
      if (k < 80) {
        const long long a = nxt.cell(g, sm.need[k]);
#pragma unroll
        for (int v = 0; v < 5; ++v) pre[t][v] = __ldg(nxt.f[v] + a);
      }
    }
  };
  long long g0 = ((long long)blockIdx.x * kOctWarps + w) * batch;
  if (g0 < ngroups) fetch(g0);
  for (; g0 < ngroups; g0 += bstride) {
    const int nb = (int)(ngroups - g0 < batch ? ngroups - g0 : batch);
    unsigned valid = 0;  // groups of the batch to update (warp-uniform)
    for (int b = 0; b < nb; ++b) {
      const bool ok = nxt_ok;
      if (ok) {
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const int k = lane + 32 * t;
          if (k < 80) {
            R q[5];
            Pol::recover(pre[t], prm, q, flags);
#pragma unroll
            for (int v = 0; v < 5; ++v) sm.q[w][v][k] = q[v];
          }
        }
      }
      const long long gn = b + 1 < nb ? g0 + b + 1 : g0 + bstride;
      if (gn < ngroups) fetch(gn);
      if (!ok) continue;
      valid |= 1u << b;
      __syncwarp();
      {
        R q0[5], dq[3][5], qh[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) q0[v] = sm.q[w][v][pc];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          R m[5], p[5];
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            m[v] = sm.q[w][v][pn[d][0]];
            p[v] = sm.q[w][v][pn[d][1]];
          }
          sub5(q0, m, m);
          sub5(p, q0, p);
#pragma unroll
          for (int v = 0; v < 5; ++v) dq[d][v] = limited_sel(m[v], p[v], prm.limiter);
        }
        hancock(q0, dq[0], dq[1], dq[2], gamma, hdt, qh);
#pragma unroll
        for (int v = 0; v < 5; ++v) sm.qh[w][v][lane] = qh[v];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          keep5(dq[d], dq[d]);
#pragma unroll
          for (int v = 0; v < 5; ++v) sm.sl[w][d][v][lane] = dq[d][v];
        }
        // the states of the upper z faces: cells 4-7 below them, 28-31 above
        if (lane >= 4 && lane < 8) {
          side5<1>(qh, dq[2], qh);
#pragma unroll
          for (int v = 0; v < 5; ++v) sm.left[w][b][v][lane - 4] = qh[v];
        } else if (lane >= 28) {
          side5<-1>(qh, dq[2], qh);
#pragma unroll
          for (int v = 0; v < 5; ++v) sm.left[w][b][5 + v][lane - 28] = qh[v];
        }
      }
      __syncwarp();
      R qL[5], qR[5], F[5], sL[5], sR[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        qL[v] = sm.qh[w][v][eL];
        qR[v] = sm.qh[w][v][eR];
        sL[v] = sm.sl[w][fd][v][eL];
        sR[v] = sm.sl[w][fd][v][eR];
      }
      side5<1>(qL, sL, qL);
      side5<-1>(qR, sR, qR);
      floor_max(qL, rf, pf);
      floor_max(qR, rf, pf);
      hllc_dyn(fd, qL, qR, gamma, igm1, F);
#pragma unroll
      for (int v = 0; v < 5; ++v) sm.f[w][b][v][lane] = F[v];
      __syncwarp();
    }
    // the upper z faces of the batch, four per group
    if (lane < 4 * nb && (valid >> (lane >> 2) & 1)) {
      const int b = lane >> 2, m = lane & 3;
      R qL[5], qR[5], F[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        qL[v] = sm.left[w][b][v][m];
        qR[v] = sm.left[w][b][5 + v][m];
      }
      floor_max(qL, rf, pf);
      floor_max(qR, rf, pf);
      hllc_dyn(dz, qL, qR, gamma, igm1, F);
#pragma unroll
      for (int v = 0; v < 5; ++v) sm.f[w][b][v][32 + m] = F[v];
    }
    __syncwarp();
    // updates, one cell per lane
    for (int u = lane; u < 8 * nb; u += 32) {
      const int b = u >> 3, e = u & 7;
      if (!(valid >> b & 1)) continue;
      const int x = e & 1, y = (e >> 1) & 1, z = e >> 2;
      const int fx = x * 4 + y + 2 * z, fy = 12 + y * 4 + x + 2 * z, fz = 24 + z * 4 + x + 2 * y;
      R a[6][5], div[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const R* F = sm.f[w][b][v];
        a[0][v] = F[fx + 4];
        a[1][v] = F[fx];
        a[2][v] = F[fy + 4];
        a[3][v] = F[fy];
        a[4][v] = F[fz + 4];
        a[5][v] = F[fz];
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) div[v] = ((a[0][v] - a[1][v]) + (a[2][v] - a[3][v])) + (a[4][v] - a[5][v]);
      long long in, out;
      src.own(g0 + b, e, in, out);
      S Uo[5], Un[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) Uo[v] = __ldg(src.f[v] + in);
      Pol::update5(Uo, dtdx, div, Un);
#pragma unroll
      for (int v = 0; v < 5; ++v) gout[v][out] = Un[v];
    }
    __syncwarp();
  }
  flush_flags(flags, err);
}

// ------------------------------------------------------------------ cubes of octs
// A run of 64 list entries that are the octs of a 4^3 cube in Morton order (found by find_oct_cubes) is
// stepped as one box of 8^3 cells by one block: a listed oct on its own recovers 80 cells, predicts 32
// and solves 36 faces for its 8 cells; the cube recovers 1376, predicts 896 and solves 1728 for its 512,
// a third of the work per cell.  Every cell and face takes the operations of k_octs, so the same bits.
// Four phases over shared memory: recover, predict (each cell's states at its faces), fluxes (in the
// place of the recovered cells), updates.  512 threads; two blocks per SM in float arithmetic, one in
// 8-byte, whose scratch fills the SM (2097152 octs, mixed, order and table built too: 1.96 ms, 2.09 with
// 256 threads, 2.04 with 384).
constexpr int kCubeThreads = 512;
constexpr int kCubeQ = 12;  // cells per axis with the two beyond each side

template <class R>
struct CubeSmem {
  R q[5][kCubeQ * kCubeQ * kCubeQ];  // recovered cells (stored at +2); then the fluxes, [axis][9][64]
  R st[6][5][512];                   // states at the cells' low and high faces, 2 axis + high
  R shell[6][5][64];                 // states toward the cube of the cells beyond its six sides
  int ids[216];                      // octs of the 6^3 neighbourhood
  static_assert(3 * 9 * 64 <= kCubeQ * kCubeQ * kCubeQ, "the fluxes fit in the place of the cells");
};

template <class Pol>
__global__ void __launch_bounds__(kCubeThreads, sizeof(typename Pol::R) >= 8 ? 1 : 2)
    k_oct_cubes(OctTable<typename Pol::S> src, typename Pol::S* o0, typename Pol::S* o1, typename Pol::S* o2,
                typename Pol::S* o3, typename Pol::S* o4, OctCubes cubes, double dx, Params prm, const double* dt_dev,
                unsigned* err) {
  using S = typename Pol::S;
  using R = typename Pol::R;
  constexpr int NT = kCubeThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<CubeSmem<R>*>(smem_raw);
  S* gout[5] = {o0, o1, o2, o3, o4};
  const double dt = dt_dev[0];
  if (!(dt > 0.0 && dt <= 1e300)) return;  // k_octs, launched after this kernel, raises the flag
  const R hdt = (R)(0.5 * dt / dx);
  const R dtdx = (R)(dt / dx);
  const R gamma = kc<R>(prm, K_GAMMA), igm1 = kc<R>(prm, K_IGM1);
  const R rf = kc<R>(prm, K_RHOF), pf = kc<R>(prm, K_PF);
  const int tid = threadIdx.x, n = min(cubes.counts[0], cubes.max_cubes);
  unsigned flags = 0;
  for (int b = blockIdx.x; b < n; b += gridDim.x) {
    const int* member = src.list + cubes.start[b];
    __syncthreads();  // the previous cube's updates are done with the neighbourhood
    for (int t = tid; t < 216; t += NT) sm.ids[t] = cube_oct(member, src.nbr, t);
    __syncthreads();
    // ---- recover: eight consecutive threads read an oct's eight cells
    for (int t = tid; t < 1728; t += NT) {
      const int o = t >> 3, e = t & 7;
      const int x = 2 * (o % 6) + (e & 1) - 2, y = 2 * (o / 6 % 6) + ((e >> 1) & 1) - 2, z = 2 * (o / 36) + (e >> 2) - 2;
      const int nout = (x < 0 || x > 7) + (y < 0 || y > 7) + (z < 0 || z > 7);
      const bool far = x == -2 || x == 9 || y == -2 || y == 9 || z == -2 || z == 9;
      if (nout > 2 || (nout == 2 && far)) continue;
      const long long a = 8LL * sm.ids[o] + e;
      S U[5];
      R q[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = __ldg(src.f[v] + a);
      Pol::recover(U, prm, q, flags);
      const int c = ((z + 2) * kCubeQ + y + 2) * kCubeQ + x + 2;
#pragma unroll
      for (int v = 0; v < 5; ++v) sm.q[v][c] = q[v];
    }
    __syncthreads();
    // ---- predict: the 512 cells and the 384 beyond the six sides
    for (int t = tid; t < 896; t += NT) {
      const int f = (t - 512) >> 6, m = t & 63;  // side (t >= 512)
      int x = t & 7, y = (t >> 3) & 7, z = t >> 6;
      if (t >= 512) {
        const int w = f & 1 ? 8 : -1, lo = m & 7, hi = m >> 3;
        x = f < 2 ? w : lo;
        y = f < 2 ? lo : (f < 4 ? w : hi);
        z = f < 4 ? hi : w;
      }
      const int c = ((z + 2) * kCubeQ + y + 2) * kCubeQ + x + 2;
      R q0[5], dq[3][5], qh[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) q0[v] = sm.q[v][c];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int o = d == 0 ? 1 : (d == 1 ? kCubeQ : kCubeQ * kCubeQ);
        R l[5], h[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          l[v] = sm.q[v][c - o];
          h[v] = sm.q[v][c + o];
        }
        sub5(q0, l, l);
        sub5(h, q0, h);
#pragma unroll
        for (int v = 0; v < 5; ++v) dq[d][v] = limited_sel(l[v], h[v], prm.limiter);
      }
      hancock(q0, dq[0], dq[1], dq[2], gamma, hdt, qh);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        R lo[5], hi[5];
        keep5(dq[d], dq[d]);
        side5<-1>(qh, dq[d], lo);
        side5<1>(qh, dq[d], hi);
        if (t < 512) {
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            sm.st[2 * d][v][t] = lo[v];
            sm.st[2 * d + 1][v][t] = hi[v];
          }
        } else if (d == (f >> 1)) {
#pragma unroll
          for (int v = 0; v < 5; ++v) sm.shell[f][v][m] = f & 1 ? lo[v] : hi[v];
        }
      }
    }
    __syncthreads();
    // ---- fluxes: face s (0 .. 8) of column m along axis d, between cells s - 1 and s
    for (int t = tid; t < 1728; t += NT) {
      const int d = t / 576, s = t / 64 % 9, m = t & 63, lo = m & 7, hi = m >> 3;
      const int step = d == 0 ? 1 : (d == 1 ? 8 : 64);
      const int c = s * step + (d == 0 ? 8 * lo + 64 * hi : (d == 1 ? lo + 64 * hi : m));  // cell s of the column
      R qL[5], qR[5], F[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        qL[v] = s > 0 ? sm.st[2 * d + 1][v][c - step] : sm.shell[2 * d][v][m];
        qR[v] = s < 8 ? sm.st[2 * d][v][c] : sm.shell[2 * d + 1][v][m];
      }
      floor_max(qL, rf, pf);
      floor_max(qR, rf, pf);
      hllc_dyn(d, qL, qR, gamma, igm1, F);
#pragma unroll
      for (int v = 0; v < 5; ++v) sm.q[v][t] = F[v];
    }
    __syncthreads();
    // ---- updates, eight consecutive threads to an oct
    for (int t = tid; t < 512; t += NT) {
      const int o = t >> 3, e = t & 7;
      const int x = 2 * (o & 3) + (e & 1), y = 2 * ((o >> 2) & 3) + ((e >> 1) & 1), z = 2 * (o >> 4) + (e >> 2);
      const int fx = x * 64 + y + 8 * z, fy = 576 + y * 64 + x + 8 * z, fz = 1152 + z * 64 + x + 8 * y;
      const long long a = 8LL * sm.ids[((o >> 4) + 1) * 36 + (((o >> 2) & 3) + 1) * 6 + (o & 3) + 1] + e;
      R div[5];
      S Uo[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const R* F = sm.q[v];
        div[v] = ((F[fx + 64] - F[fx]) + (F[fy + 64] - F[fy])) + (F[fz + 64] - F[fz]);
        Uo[v] = __ldg(src.f[v] + a);
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) gout[v][a] = Pol::update(Uo[v], dtdx, div[v]);
    }
  }
  flush_flags(flags, err);
}

template <class Pol, class Src>
cudaError_t launch_octs_src(const Src& src, void* const out[5], long long ngroups, double dx, const Params& prm,
                            const double* dt, unsigned* err, cudaStream_t s, const int* count = nullptr) {
  using S = typename Pol::S;
  const size_t smem = sizeof(OctSmem<Pol>);
  static PerDeviceOnce attr;
  cudaError_t e = attr.call(
      [&] { return cudaFuncSetAttribute(k_octs<Pol, Src>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
  if (e != cudaSuccess) return e;
  // groups per batch: full batches once every resident warp has one, fewer on a small list
  const long long warps = 152LL * oct_min_blocks<Pol, Src>() * kOctWarps;
  const int batch = (int)std::min<long long>(kOctBatch, std::max<long long>(1, ngroups / warps));
  const long long per_block = (long long)kOctWarps * batch;
  const long long blocks = std::min((ngroups + per_block - 1) / per_block, 152LL * 64);
  k_octs<Pol, Src><<<(unsigned)blocks, 32 * kOctWarps, smem, s>>>(src, (S*)out[0], (S*)out[1], (S*)out[2], (S*)out[3],
                                                                   (S*)out[4], ngroups, count, batch, dx, prm, dt, err);
  return cudaGetLastError();
}

template <class Pol>
cudaError_t launch_octs(void* const gathered[5], void* const out[5], long long ngroups, double dx, const Params& prm,
                        const double* dt, unsigned* err, cudaStream_t s) {
  using S = typename Pol::S;
  OctGathered<S> src;
  for (int v = 0; v < 5; ++v) src.f[v] = static_cast<const S*>(gathered[v]);
  return launch_octs_src<Pol>(src, out, ngroups, dx, prm, dt, err, s);
}

template <class Pol>
cudaError_t launch_octs_level(const HostPatchIO& level, const int* origins, void* const out[5], long long ngroups,
                              const Params& prm, const double* dt, unsigned* err, cudaStream_t s) {
  using S = typename Pol::S;
  OctLevel<S> src;
  for (int v = 0; v < 5; ++v) src.f[v] = static_cast<const S*>(level.in[v]);
  src.nx = level.nx; src.ny = level.ny; src.nz = level.nz;
  src.sy = level.isy; src.sz = level.isz;
  src.origins = origins;
  src.ox = src.oy = src.oz = 0;
  return launch_octs_src<Pol>(src, out, ngroups, level.dx, prm, dt, err, s);
}

template <class Pol>
cudaError_t launch_octs_table(void* const in[5], const int* nbr, int noct, const int* list, void* const out[5],
                              long long ngroups, double dx, const Params& prm, const double* dt, unsigned* err,
                              const OctCubes* cubes, cudaStream_t s) {
  using S = typename Pol::S;
  OctTable<S> src;
  for (int v = 0; v < 5; ++v) src.f[v] = static_cast<const S*>(in[v]);
  src.nbr = nbr;
  src.list = list;
  src.noct = noct;
  src.oct = 0;
  if (!cubes) return launch_octs_src<Pol>(src, out, ngroups, dx, prm, dt, err, s);
  const size_t smem = sizeof(CubeSmem<typename Pol::R>);
  static PerDeviceOnce attr;
  cudaError_t e = attr.call([&] {
    return cudaFuncSetAttribute(k_oct_cubes<Pol>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  const int blocks = (int)std::min<long long>(152 * (sizeof(typename Pol::R) >= 8 ? 1 : 2), ngroups / 64);
  k_oct_cubes<Pol><<<blocks, kCubeThreads, smem, s>>>(
      src, (S*)out[0], (S*)out[1], (S*)out[2], (S*)out[3], (S*)out[4], *cubes, dx, prm, dt, err);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  src.list = cubes->left;  // the octs outside the cubes
  return launch_octs_src<Pol>(src, out, ngroups, dx, prm, dt, err, s, cubes->counts + 1);
}

// ------------------------------------------------------------------ primitive <-> conservative
// Interior cell c -> (i, j, k), in 32-bit arithmetic when the patch has fewer than 2^31 cells (a
// 64-bit integer division is a long sequence that runs partly on the FP64 pipe).
template <class S>
__device__ __forceinline__ void cell_ijk(const PatchIO<S>& P, long long c, int& i, int& j, int& k) {
  const long long nxy = (long long)P.nx * P.ny;
  if (nxy * P.nz <= 0x7fffffffLL) {
    const int cc = (int)c, nxy32 = (int)nxy;
    k = cc / nxy32;
    const int r = cc - k * nxy32;
    j = r / P.nx;
    i = r - j * P.nx;
  } else {
    k = (int)(c / nxy);
    const long long r = c - (long long)k * nxy;
    j = (int)(r / P.nx);
    i = (int)(r - (long long)j * P.nx);
  }
}
template <class S>
__device__ __forceinline__ long long cell_offset(const PatchIO<S>& P, int i, int j, int k, bool out_side) {
  const int g = out_side ? P.gout : P.gin;
  const long long sy = out_side ? P.osy : P.isy, sz = out_side ? P.osz : P.isz;
  return (long long)(k + g) * sz + (long long)(j + g) * sy + (i + g);
}

// U = (rho, rho u, rho v, rho w, p/(gamma-1) + rho |u|^2 / 2), in the storage type.
template <class S>
__global__ void k_p2c(PatchIO<S> P, double gamma) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  const S igm1 = (S)(1.0 / (gamma - 1.0));
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(P, c, i, j, k);
    const long long a = cell_offset(P, i, j, k, false), b = cell_offset(P, i, j, k, true);
    const S r = P.in[0][a], u = P.in[1][a], v = P.in[2][a], w = P.in[3][a], p = P.in[4][a];
    P.out[0][b] = r;
    P.out[1][b] = r * u;
    P.out[2][b] = r * v;
    P.out[3][b] = r * w;
    P.out[4][b] = p * igm1 + S(0.5) * r * ((u * u + v * v) + w * w);
  }
}

// lamW = (dU/dW)^T lamU.  W and lamU share one layout (P.in / L.in); lamW uses P.out's layout.
template <class S>
__global__ void k_p2c_adjoint(PatchIO<S> P, PatchIO<S> L, double gamma) {
  const long long n = (long long)P.nx * P.ny * P.nz;
  const S igm1 = (S)(1.0 / (gamma - 1.0));
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    int i, j, k;
    cell_ijk(P, c, i, j, k);
    const long long a = cell_offset(P, i, j, k, false), la = cell_offset(L, i, j, k, false),
                    b = cell_offset(P, i, j, k, true);
    const S r = P.in[0][a], u = P.in[1][a], v = P.in[2][a], w = P.in[3][a];
    const S l0 = L.in[0][la], l1 = L.in[1][la], l2 = L.in[2][la], l3 = L.in[3][la], l4 = L.in[4][la];
    P.out[0][b] = l0 + u * l1 + v * l2 + w * l3 + S(0.5) * ((u * u + v * v) + w * w) * l4;
    P.out[1][b] = r * l1 + r * u * l4;
    P.out[2][b] = r * l2 + r * v * l4;
    P.out[3][b] = r * l3 + r * w * l4;
    P.out[4][b] = igm1 * l4;
  }
}

template <class Pol>
cudaError_t launch_p2c(const HostPatchIO& W, void* const U[5], const Params& prm, cudaStream_t s) {
  HostPatchIO h = W;
  for (int v = 0; v < 5; ++v) h.out[v] = U[v];
  k_p2c<typename Pol::S><<<152 * 8, 256, 0, s>>>(to_dev<Pol>(h), prm.gamma);
  return cudaGetLastError();
}

template <class Pol>
cudaError_t launch_p2c_adjoint(const HostPatchIO& W, const HostPatchIO& lamU, void* const lamW[5], const Params& prm,
                               cudaStream_t s) {
  HostPatchIO h = W;
  for (int v = 0; v < 5; ++v) h.out[v] = lamW[v];
  k_p2c_adjoint<typename Pol::S><<<152 * 8, 256, 0, s>>>(to_dev<Pol>(h), to_dev<Pol>(lamU), prm.gamma);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ flux registers
// Fluxes through the six boundary faces of boxes (AMR refluxing, Berger & Colella 1989: the
// coarse level's fluxes at a fine patch's boundary are replaced by the fine ones): one thread per
// face; both adjacent cells predicted from their own 3^3-minus-corners stencil exactly as the step
// does (recovery, limited slopes, Hancock predictor), face states floored, HLLC.  A box is either
// a ghosted patch's interior or a box of a periodic level.  The register (storage type, layout
// x-low [nz][ny], x-high, y-low [nz][nx], y-high, z-low [ny][nx], z-high per field) receives
// dt * F, added to its contents when accumulating (the time integral over a patch's substeps).
// Face f of a box's register (32-bit arithmetic: a box has fewer than 2^31 boundary faces).
__device__ __forceinline__ void box_face(const HostBoxFluxes& B, int f, int& d, int& i, int& j, int& k) {
  const int nx = B.n[0], ny = B.n[1], nz = B.n[2];
  const int X = ny * nz, Y = nx * nz;
  if (f < 2 * X) {
    d = 0;
    const int side = f >= X, r = f - side * X;
    k = r / ny;
    j = r - k * ny;
    i = side ? nx - 1 : -1;
  } else if (f < 2 * X + 2 * Y) {
    d = 1;
    const int g = f - 2 * X, side = g >= Y, r = g - side * Y;
    k = r / nx;
    i = r - k * nx;
    j = side ? ny - 1 : -1;
  } else {
    d = 2;
    const int g = f - 2 * X - 2 * Y, Z = nx * ny, side = g >= Z, r = g - side * Z;
    j = r / nx;
    i = r - j * nx;
    k = side ? nz - 1 : -1;
  }
}

template <class Pol>
__global__ void __launch_bounds__(256) k_box_fluxes(const HostBoxFluxes* boxes, const int2* blocks, Params prm,
                                                    const double* dt_dev, int accumulate) {
  using S = typename Pol::S;
  using R = typename Pol::R;
  const int2 b = blocks[blockIdx.x];
  const HostBoxFluxes B = boxes[b.x];
  const int nface = 2 * (B.n[1] * B.n[2] + B.n[0] * B.n[2] + B.n[0] * B.n[1]);
  const int f = b.y * 256 + threadIdx.x;
  if (f >= nface) return;
  int d, i, j, k;
  box_face(B, f, d, i, j, k);  // the face between cell (i, j, k) and its +d neighbour
  const double dt = dt_dev[B.dt_index];
  unsigned flags = 0;
  // address of cell (x, y, z) in box coordinates (interior from 0; the stencil reaches -2 .. n+1)
  auto addr = [&](int x, int y, int z) -> long long {
    if (B.periodic) {  // origin in [0, N), box no larger than N: o + x in [-2, 2N + 2)
      auto wrap = [](int v, int n) {
        v += v < 0 ? n : 0;
        v -= v >= n ? n : 0;
        return v >= n ? v - n : v;
      };
      x = wrap(x + B.o[0], B.N[0]);
      y = wrap(y + B.o[1], B.N[1]);
      z = wrap(z + B.o[2], B.N[2]);
      return (long long)z * B.sz + (long long)y * B.sy + x;
    }
    return (long long)(z + 2) * B.sz + (long long)(y + 2) * B.sy + (x + 2);
  };
  auto q_at = [&](int x, int y, int z, R q[5]) {
    const long long a = addr(x, y, z);
    S U[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) U[v] = __ldg(static_cast<const S*>(B.U[v]) + a);
    Pol::recover(U, prm, q, flags);
  };
  const R hdt = (R)(0.5 * dt / B.dx);
  R st[2][5];  // face states: left then right
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int x = i + (side && d == 0), y = j + (side && d == 1), z = k + (side && d == 2);
    R c[5], m[5], p[5], dq[3][5], qh[5];
    q_at(x, y, z, c);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      q_at(x - (e == 0), y - (e == 1), z - (e == 2), m);
      q_at(x + (e == 0), y + (e == 1), z + (e == 2), p);
#pragma unroll
      for (int v = 0; v < 5; ++v) dq[e][v] = limited_sel(c[v] - m[v], p[v] - c[v], prm.limiter);
    }
    hancock(c, dq[0], dq[1], dq[2], kc<R>(prm, K_GAMMA), hdt, qh);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const R sd = d == 0 ? dq[0][v] : (d == 1 ? dq[1][v] : dq[2][v]);
      st[side][v] = side ? qh[v] - half_(sd) : qh[v] + half_(sd);
    }
  }
  floor_state(st[0], kc<R>(prm, K_RHOF), kc<R>(prm, K_PF));
  floor_state(st[1], kc<R>(prm, K_RHOF), kc<R>(prm, K_PF));
  R F[5];
  hllc_dyn(d, st[0], st[1], kc<R>(prm, K_GAMMA), kc<R>(prm, K_IGM1), F);
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    S* reg = static_cast<S*>(B.reg) + (long long)v * nface + f;
    const S add = (S)(dt * (double)F[v]);
    *reg = accumulate ? *reg + add : add;
  }
}

template <class Pol>
cudaError_t launch_box_fluxes(const HostBoxFluxes* d_boxes, const int2* d_blocks, int nblocks, const Params& prm,
                              const double* dt, int accumulate, cudaStream_t s) {
  k_box_fluxes<Pol><<<nblocks, 256, 0, s>>>(d_boxes, d_blocks, prm, dt, accumulate);
  return cudaGetLastError();
}

template <class Pol>
const KernelOps& make_ops() {
  static const KernelOps ops = {
      &launch_uniform<Pol>,      &launch_batched<Pol>,      &batched_blocks_per_sm<Pol>,
      &launch_cfl<Pol>,          &launch_octs<Pol>,         &launch_octs_level<Pol>,   &launch_octs_table<Pol>,
      &launch_adjoint<Pol>,
      &adjoint_scratch_bytes<Pol>, &launch_p2c<Pol>,        &launch_p2c_adjoint<Pol>,
      &launch_box_fluxes<Pol>,   &launch_ppm<Pol>,          &launch_ppm_batched<Pol>,
      (int)sizeof(typename Pol::S), 1};
  return ops;
}

}  // namespace hydro
