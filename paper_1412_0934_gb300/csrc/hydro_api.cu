// C ABI of the hydro library (include/hydro.h): argument validation, the context and its
// library-owned scratch, patch-set caching and work-list rebuilds, launch selection, the
// CUDA-graph multi-step runner and the autotuner.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "hydro.h"
#include "hydro_device.cuh"
#include "internal.h"

using hydro::HostPatchIO;
using hydro::HostTileRec;

// How many graphs hold an address: captured calls add to it, and the graph's and its executables' end
// takes it back (graph_holds, below), from a thread of the driver's and perhaps after the context's end.
using GraphRefs = std::shared_ptr<std::atomic<int>>;
bool held(const GraphRefs& refs) { return refs && refs->load() > 0; }

// What a call derives from its descriptors (field pointers, shapes, origins, boxes) and keeps on the
// device: descriptor copies, block tables, copy tasks, work-lists.  The last kKept sets of each kind of
// call stay, the least recently used making room: a level's patches step from one buffer set to another
// and back, so consecutive calls alternate between sets (with one kept set, each substep of a subcycled
// level rebuilt its tables and drained the stream for it).  A set that a graph was captured with stays
// beside them until that graph is gone.
struct SetCache {
  static constexpr int kKept = 4;
  struct Entry {
    std::vector<char> key;
    bool valid = false;
    unsigned long long used = 0;
    char* d = nullptr;
    size_t cap = 0;
    size_t off[4] = {};  // offsets of the parts in d
    int n[10] = {};      // counts and settings of the set
    GraphRefs graphs;
  };
  std::vector<std::unique_ptr<Entry>> entry;
  unsigned long long clock = 0;
  Entry* find(const std::vector<char>& key) {
    for (auto& e : entry)
      if (e->valid && e->key == key) {
        e->used = ++clock;
        return e.get();
      }
    return nullptr;
  }
  // The entry to fill for a new key, with room for n bytes (nullptr: no memory); valid once the
  // caller has enqueued its contents and calls done().
  Entry* replace(size_t n) {
    Entry* o = nullptr;
    for (;;) {  // the least recently used of kKept sets that no graph holds; sets beyond those are freed
      size_t oldest = 0;
      int free_sets = 0;
      for (size_t i = 0; i < entry.size(); ++i)
        if (!held(entry[i]->graphs)) {
          if (free_sets++ == 0 || entry[i]->used < entry[oldest]->used) oldest = i;
        }
      if (free_sets < kKept) {
        entry.emplace_back(new Entry);
        o = entry.back().get();
        break;
      }
      if (free_sets == kKept) {
        o = entry[oldest].get();
        break;
      }
      cudaFree(entry[oldest]->d);
      entry.erase(entry.begin() + oldest);
    }
    o->valid = false;
    if (o->cap < n) {
      cudaFree(o->d);
      o->d = nullptr;
      o->cap = 0;
      if (cudaMalloc(&o->d, n + n / 4) != cudaSuccess) return nullptr;
      o->cap = n + n / 4;
    }
    return o;
  }
  void done(Entry* e, std::vector<char>&& key) {
    e->key = std::move(key);
    e->used = ++clock;
    e->valid = true;
  }
  void free_all() {
    for (auto& e : entry) cudaFree(e->d);
  }
};

// Device scratch that grows with the largest call; what a graph holds is set aside, not freed, when a
// larger block takes its place.
struct Scratch {
  char* d = nullptr;
  size_t cap = 0;
  GraphRefs graphs;
};

struct hydro_ctx {
  hydro_config cfg;
  hydro::Params prm;
  cudaStream_t stream = nullptr;
  cudaStream_t capture = nullptr;  // private stream used to capture graphs
  const hydro::KernelOps* ops = nullptr;
  int device = 0, sm_count = 0;
  unsigned* d_err = nullptr;
  // page-locked staging of uploads: two buffers in turn, each reused once its last copy has run
  char* h_stage[2] = {nullptr, nullptr};
  size_t h_stage_cap[2] = {0, 0};
  cudaEvent_t ev_stage[2] = {nullptr, nullptr};
  int stage_turn = 0;
  // batched step: descriptors and work-list of the last patch sets
  SetCache batch;
  int* d_counter = nullptr;  // 1 + HYDRO_NUM_PATCH_CLASSES tile counters
  // tile shape per patch-shape class (-1: the context's tile_id / zchunk)
  int cls_tile[HYDRO_NUM_PATCH_CLASSES] = {-1, -1, -1}, cls_zc[HYDRO_NUM_PATCH_CLASSES] = {0, 0, 0};
  double* d_cls_dt = nullptr;  // the autotuner's per-class time steps
  size_t cls_dt_cap = 0;
  SetCache cfl_sets;  // CFL of many patches: descriptors
  // tuning; until a caller sets it (hydro_set_tuning, hydro_autotune), hydro_step and hydro_run take each
  // box's and patch set's tile shape and z chunk from the rule of default_tuning (a batch with a tile shape
  // per class, hydro_set_class_tuning, takes those, and 16x16 tiles of 32 planes for the other classes)
  int tile_id = 0, zchunk = 32;
  bool tuned = false;
  int rule_n[3] = {0, 0, 0}, rule_tile = 0, rule_zc = 0;  // the rule's choice for the last box size
  // graph cache of hydro_run
  cudaGraphExec_t graph = nullptr;
  hydro_patch g_a = {}, g_b = {};
  int g_n = -1;
  double* g_dt = nullptr;
  int g_tile = -1, g_zc = -1;
  bool g_tuned = false;
  // adjoint scratch
  Scratch adj;
  std::vector<Scratch> aside;  // outgrown blocks that graphs held
  // host-buffer step: device staging of one box (in and out), its descriptor and slab tile list,
  // per-slab tile counters, the two copy streams and the events that chain the pipeline
  char* d_stage = nullptr;
  size_t stage_cap = 0;
  HostPatchIO* d_stage_io = nullptr;
  HostTileRec* d_stage_tiles = nullptr;
  size_t stage_tiles_cap = 0;
  int* d_stage_counters = nullptr;
  size_t stage_counters_cap = 0;
  long long stage_key[7] = {-1, -1, -1, -1, -1, -1, -1};  // nx ny nz sy sz tile zc of the uploaded list
  double stage_dx = 0.0;
  cudaStream_t s_h2d = nullptr, s_d2h = nullptr;
  cudaStream_t s_cmp2 = nullptr;  // second compute stream: consecutive slabs' kernels overlap
  cudaEvent_t ev_ready = nullptr;
  std::vector<cudaEvent_t> ev_copied, ev_stepped, ev_halo;
  cudaEvent_t ev_begin = nullptr, ev_end = nullptr;
  // coarse-to-fine ghost fill: descriptors and block table; same-level exchange: descriptors and tasks
  SetCache ghost_sets, xchg_sets;
  // flux registers (patch boxes, level boxes), refluxing, average-down, MHD step and CFL on patches:
  // descriptors and block tables
  static constexpr int kAux = 6;  // 0, 1 box fluxes; 2 reflux; 3 average-down; 4 MHD step; 5 MHD CFL
  SetCache aux[kAux];
  // oct builder scratch: key bitmap, word prefix sums, block prefix sums; and, for eager calls only (a
  // graph never holds the address of what a longer list makes the context replace), octs by key
  Scratch octs;
  int* d_octs_slots = nullptr;
  size_t octs_slots_cap = 0;
  // oct step through the table: the list's cubes (OctCubes), for eager calls only too
  char* d_cubes = nullptr;
  size_t cubes_cap = 0;
  // MHD step scratch: constants, face states, fluxes
  Scratch mhd;
  long long launches = 0;
};

namespace hydro {
const KernelOps* ops_for(int precision) {
  switch (precision) {
    case HYDRO_FP64: return &ops_f64();
    case HYDRO_FP32: return &ops_f32();
    case HYDRO_MIXED: return &ops_mixed();
    case HYDRO_FP64_DF: return &ops_df();
  }
  return nullptr;
}
}  // namespace hydro

namespace {

bool finite_pos(double x) { return std::isfinite(x) && x > 0.0; }

int cuda_status(cudaError_t e) { return e == cudaSuccess ? HYDRO_OK : HYDRO_ERR_CUDA; }

int elem_size(const hydro_ctx* c) { return c->cfg.precision == HYDRO_FP32 ? 4 : 8; }

// PPM (stencil radius 3) steps periodic boxes and patches with three ghost layers; the calls built
// on the radius-2 PLM stencil alone (the host-buffer step, octs, boundary fluxes, the adjoint)
// reject a PPM context.
bool ppm(const hydro_ctx* c) { return c->cfg.limiter == HYDRO_PPM; }

bool valid_patch(const hydro_ctx* c, const hydro_patch& p) {
  if (p.nx < 1 || p.ny < 1 || p.nz < 1) return false;
  if (p.ng != 0 && p.ng != 2 && !(p.ng == 3 && ppm(c))) return false;
  if (!finite_pos(p.dx)) return false;
  const long long gx = p.nx + 2LL * p.ng, gy = p.ny + 2LL * p.ng;
  if (p.sy < gx || p.sz < p.sy * gy) return false;
  const int es = elem_size(c);
  for (int v = 0; v < 5; ++v) {
    if (!p.U[v]) return false;
    if (reinterpret_cast<uintptr_t>(p.U[v]) % es) return false;
  }
  return true;
}

// Byte extent of a field of patch p.
size_t field_bytes(const hydro_ctx* c, const hydro_patch& p) {
  return (size_t)(p.nz + 2 * p.ng) * (size_t)p.sz * elem_size(c);
}

bool overlaps(const hydro_ctx* c, const hydro_patch& a, const hydro_patch& b) {
  const size_t na = field_bytes(c, a), nb = field_bytes(c, b);
  for (int i = 0; i < 5; ++i)
    for (int j = 0; j < 5; ++j) {
      const char* x = static_cast<const char*>(a.U[i]);
      const char* y = static_cast<const char*>(b.U[j]);
      if (x < y + nb && y < x + na) return true;
    }
  return false;
}

bool same_shape(const hydro_patch& a, const hydro_patch& b) {
  return a.nx == b.nx && a.ny == b.ny && a.nz == b.nz && a.dx == b.dx;
}

HostPatchIO make_io(const hydro_patch& in, const hydro_patch& out) {
  HostPatchIO h;
  for (int v = 0; v < 5; ++v) {
    h.in[v] = in.U[v];
    h.out[v] = out.U[v];
  }
  h.nx = in.nx; h.ny = in.ny; h.nz = in.nz;
  h.gin = in.ng; h.gout = out.ng;
  h.isy = in.sy; h.isz = in.sz; h.osy = out.sy; h.osz = out.sz;
  h.dx = in.dx;
  return h;
}

template <class T>
int ensure_device(T** d, size_t* cap, size_t n) {
  if (*cap >= n) return HYDRO_OK;
  if (*d) cudaFree(*d);
  *d = nullptr;
  *cap = 0;
  if (cudaMalloc(reinterpret_cast<void**>(d), n * sizeof(T)) != cudaSuccess) return HYDRO_ERR_NOMEM;
  *cap = n;
  return HYDRO_OK;
}

// Where the context's stream is being captured: the graph takes a reference to `refs`, which it drops when
// it and the executables made of it are destroyed.
int graph_holds(hydro_ctx* c, GraphRefs& refs) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaGraph_t g = nullptr;
  if (cudaStreamIsCapturing(c->stream, &cs) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (cs == cudaStreamCaptureStatusNone) return HYDRO_OK;
  if (cudaStreamGetCaptureInfo(c->stream, &cs, nullptr, &g) != cudaSuccess || cs != cudaStreamCaptureStatusActive)
    return HYDRO_ERR_CUDA;
  if (!refs) refs = std::make_shared<std::atomic<int>>(0);
  GraphRefs* mine = new GraphRefs(refs);
  cudaUserObject_t object;
  auto drop = [](void* p) {
    GraphRefs* r = static_cast<GraphRefs*>(p);
    --**r;
    delete r;
  };
  if (cudaUserObjectCreate(&object, mine, drop, 1, cudaUserObjectNoDestructorSync) != cudaSuccess) {
    delete mine;
    return HYDRO_ERR_CUDA;
  }
  ++*refs;
  if (cudaGraphRetainUserObject(g, object, 1, cudaGraphUserObjectMove) != cudaSuccess) {
    cudaUserObjectRelease(object, 1);  // runs drop
    return HYDRO_ERR_CUDA;
  }
  return HYDRO_OK;
}

// At least n bytes of scratch, held by the graph where the call is captured.
int ensure_scratch(hydro_ctx* c, Scratch& s, size_t n) {
  if (s.cap < n) {
    if (held(s.graphs)) {
      c->aside.push_back(s);
    } else {
      cudaFree(s.d);
    }
    s = Scratch();
    for (size_t i = c->aside.size(); i-- > 0;)
      if (!held(c->aside[i].graphs)) {
        cudaFree(c->aside[i].d);
        c->aside.erase(c->aside.begin() + i);
      }
    if (cudaMalloc(&s.d, n) != cudaSuccess) return HYDRO_ERR_NOMEM;
    s.cap = n;
  }
  return graph_holds(c, s.graphs);
}

// Scratch that a call can do without, for eager calls only; false where it is captured or there is no
// memory (that failure ends here).
template <class T>
bool eager_scratch(hydro_ctx* c, T** d, size_t* cap, size_t n) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(c->stream, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone &&
      ensure_device(d, cap, n) == HYDRO_OK)
    return true;
  cudaGetLastError();
  return false;
}

template <class T>
size_t append(std::vector<char>& bytes, const T* p, size_t n) {
  const size_t off = (bytes.size() + 255) / 256 * 256;
  bytes.resize(off + n * sizeof(T));
  if (n) std::memcpy(bytes.data() + off, p, n * sizeof(T));
  return off;
}

// Enqueue the copy of n host bytes to device memory on the context's stream, through page-locked
// staging: the caller may free p, and the stream's order keeps earlier readers of d safe, so nothing
// is drained.
bool upload(hydro_ctx* c, void* d, const void* p, size_t n) {
  if (n == 0) return true;
  const int t = c->stage_turn ^= 1;
  if (!c->ev_stage[t] && cudaEventCreateWithFlags(&c->ev_stage[t], cudaEventDisableTiming) != cudaSuccess) return false;
  if (c->h_stage[t] && cudaEventSynchronize(c->ev_stage[t]) != cudaSuccess) return false;
  if (c->h_stage_cap[t] < n) {
    cudaFreeHost(c->h_stage[t]);
    c->h_stage[t] = nullptr;
    c->h_stage_cap[t] = 0;
    const size_t cap_n = std::max<size_t>(n + n / 4, 1 << 18);
    if (cudaMallocHost(&c->h_stage[t], cap_n) != cudaSuccess) return false;
    c->h_stage_cap[t] = cap_n;
  }
  std::memcpy(c->h_stage[t], p, n);
  return cudaMemcpyAsync(d, c->h_stage[t], n, cudaMemcpyHostToDevice, c->stream) == cudaSuccess &&
         cudaEventRecord(c->ev_stage[t], c->stream) == cudaSuccess;
}

// An entry of `cache` for a new set of n bytes; *rc says why there is none.  Refused while the stream is
// being captured: a graph must neither allocate nor hold the staging buffer.
SetCache::Entry* new_entry(hydro_ctx* c, SetCache& cache, size_t n, int* rc) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  *rc = HYDRO_ERR_CUDA;
  if (cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return nullptr;
  *rc = HYDRO_ERR_NOMEM;
  return cache.replace(std::max<size_t>(n, 256));
}

// The entry holding `bytes` on the device, uploaded unless one of the last sets has them.
SetCache::Entry* upload_set(hydro_ctx* c, SetCache& cache, std::vector<char>&& bytes) {
  if (SetCache::Entry* e = cache.find(bytes)) return graph_holds(c, e->graphs) ? nullptr : e;
  int rc;
  SetCache::Entry* e = new_entry(c, cache, bytes.size(), &rc);
  if (!e || !upload(c, e->d, bytes.data(), bytes.size())) return nullptr;
  cache.done(e, std::move(bytes));
  return e;
}

// Patch-shape class of a patch for the per-class tile choice (include/hydro.h): 0 an x or y edge
// of 8 cells or fewer, 1 an x or y edge not a multiple of 16, 2 both multiples of 16.
int patch_class(const hydro_patch& p) {
  if (p.nx <= 8 || p.ny <= 8) return 0;
  if (p.nx % 16 || p.ny % 16) return 1;
  return 2;
}

bool per_class(const hydro_ctx* c) {
  if (ppm(c)) return false;
  for (int k = 0; k < HYDRO_NUM_PATCH_CLASSES; ++k)
    if (c->cls_tile[k] >= 0) return true;
  return false;
}
int class_tile(const hydro_ctx* c, int k) { return c->cls_tile[k] >= 0 ? c->cls_tile[k] : c->tile_id; }
int class_zc(const hydro_ctx* c, int k) { return c->cls_tile[k] >= 0 ? c->cls_zc[k] : c->zchunk; }

// ------------------------------------------------------------------ default tuning
// The tile shape and z chunk of a box or patch set whose context has no tuning of the caller's, from a
// cost model of the step kernels: a block marching zc planes alone on an SM takes plane * (zc + start)
// microseconds, and k blocks resident together (at most `resident`) take share[k] times that.  With n =
// ceil(blocks / SMs) blocks per SM the launch takes their rounds, full ones of `resident` blocks and the
// rest.  Short chunks fill the SMs of a small box (32^3 at one 32-plane chunk of 16x16 tiles is 4 blocks)
// and repeat two planes each; long ones serve the large boxes.  The constants are fits to steps of 16^3
// to 512^3 boxes at 2 to 128-plane chunks; the model stays within 5% of those and picks, against the
// fixed 16x16 tiles of 32 planes: FP64 32^3 1367 -> 97 us, double-float 61^3 256 -> 70, FP32 96^3 76 -> 46,
// mixed 64^3 124 -> 33; 512^3 within 1% of the best of the sweep.  (Double-float since its comparisons are
// branch-free: 16x16 tiles with two blocks per SM take the 512^3 step in 20.8 ms, 32x16 tiles in 23.2.)
struct ShapeCost {
  int tile;
  double plane, start;
  int resident;
  double share[4];
};
constexpr ShapeCost kCostF64[] = {{0, 41.0, 1.2, 2, {0.0, 1.0, 1.77}},
                                  {2, 28.4, 1.25, 3, {0.0, 1.0, 1.0, 1.27}},
                                  {3, 73.6, 1.04, 1, {0.0, 1.0}}};
constexpr ShapeCost kCostDF[] = {{0, 7.6, 1.9, 2, {0.0, 1.0, 1.52}}, {3, 12.6, 1.8, 1, {0.0, 1.0}}};
constexpr ShapeCost kCostF32[] = {{0, 1.95, 5.3, 3, {0.0, 1.0, 1.29, 1.76}},
                                  {1, 1.94, 5.3, 3, {0.0, 1.0, 1.29, 1.76}},
                                  {3, 2.5, 4.9, 1, {0.0, 1.0}}};
constexpr ShapeCost kCostMixed[] = {{0, 3.4, 4.0, 3, {0.0, 1.0, 1.27, 1.65}},
                                    {1, 3.38, 4.0, 3, {0.0, 1.0, 1.27, 1.65}},
                                    {3, 4.55, 3.2, 1, {0.0, 1.0}}};
constexpr ShapeCost kCostPpm8[] = {{0, 1.0, 4.0, 1, {0.0, 1.0}}};  // one tile shape: only the chunk is chosen
constexpr ShapeCost kCostPpm4[] = {{0, 1.0, 4.0, 2, {0.0, 1.0, 1.3}}};

double rounds(const ShapeCost& s, long long n) {
  return (double)(n / s.resident) * s.share[s.resident] + s.share[n % s.resident];
}

void default_tuning(const hydro_ctx* c, const hydro_patch* in, int n, int* tile, int* zchunk) {
  const ShapeCost* shapes = kCostF64;
  int ns = 3;
  switch (c->cfg.precision) {
    case HYDRO_FP32: shapes = kCostF32; break;
    case HYDRO_MIXED: shapes = kCostMixed; break;
    case HYDRO_FP64_DF: shapes = kCostDF; ns = 2; break;
  }
  if (ppm(c)) {
    shapes = (c->cfg.precision == HYDRO_FP32 || c->cfg.precision == HYDRO_MIXED) ? kCostPpm4 : kCostPpm8;
    ns = 1;
  }
  int maxnz = 1;
  for (int i = 0; i < n; ++i) maxnz = std::max(maxnz, in[i].nz);
  double best = 1e300;
  *tile = 0;
  *zchunk = 32;
  // the fixed 16x16 tiles of 32 planes first: another choice has to save 3% of their time
  long long blocks0 = -1;  // blocks of those
  auto consider = [&](int zc, int kinds) {
    for (int k = 0; k < kinds; ++k) {
      const ShapeCost& s = shapes[k];
      const int tx = hydro::kTileX[s.tile], ty = hydro::kTileY[s.tile];
      long long blocks = 0;
      double planes = 0.0;  // marched by all blocks, their start planes included
      for (int i = 0; i < n; ++i) {
        const long long cols = (long long)((in[i].nx + tx - 1) / tx) * ((in[i].ny + ty - 1) / ty);
        const long long chunks = (in[i].nz + zc - 1) / zc;
        blocks += cols * chunks;
        planes += (double)cols * (in[i].nz + chunks * s.start);
      }
      if (blocks0 < 0) blocks0 = blocks;
      const long long per_sm = (blocks + c->sm_count - 1) / c->sm_count;
      const double t = s.plane * planes / (double)blocks * rounds(s, per_sm);
      if (t < best) {
        best = best == 1e300 ? 0.97 * t : t;
        *tile = s.tile;
        *zchunk = zc;
      }
    }
  };
  consider(32, 1);
  // Where that fills every SM four times over there is little left to balance, and differences the model
  // does not hold (caches, uneven patches, the last tiles' tail) decide: the batched, FP64 and PPM steps
  // keep it (4096 uneven patches, mixed: 10.8 ms, 11.6 with the model's choice; FP64 256^3 16.4 against
  // 16.9).  Uniform boxes in double-float and float still gain 2-4% from fewer start planes.
  if (blocks0 >= 4LL * shapes[0].resident * c->sm_count && (n > 1 || ppm(c) || c->cfg.precision == HYDRO_FP64)) return;
  if (n == 1) {
    // one box: every chunk count up to 64, and two-plane chunks at the least
    for (int k = 1; k <= 64; ++k) {
      const int zc = (maxnz + k - 1) / k;
      if (zc > 128 && k < 64) continue;
      consider(std::min(zc, 4096), ns);
      if (zc <= 2) break;
    }
  } else {
    for (int zc : {2, 4, 8, 16, 32}) {
      consider(zc, ns);
      if (zc >= maxnz) break;
    }
  }
}

// Counts and settings of a batch entry (SetCache::Entry::n).
enum { B_NTILES, B_TILE, B_ZCHUNK, B_PER_CLASS, B_CLS_OFF, B_CLS_NTILES = B_CLS_OFF + HYDRO_NUM_PATCH_CLASSES };
// Its parts: descriptors, tile records, prefix-sum counts, patch indices by class.
enum { B_PATCHES, B_TILES, B_COUNTS, B_INDEX };

// Upload the descriptors of (in, out) and build the tile work-list for the current tuning,
// unless one of the last sets and its tuning are the same.  With a tile shape per patch-shape class the
// work-list holds one segment per class, each built with its class's tile shape and z chunk.
int prepare_batch(hydro_ctx* c, const hydro_patch* in, const hydro_patch* out, int n, SetCache::Entry** entry) {
  constexpr int NC = HYDRO_NUM_PATCH_CLASSES;
  // the PPM kernel's tiles are 16 x 16 (tile shape 0)
  int tile = ppm(c) ? 0 : c->tile_id, zchunk = c->zchunk;
  const bool pc = per_class(c);
  std::vector<char> key(2 * (size_t)n * sizeof(hydro_patch));
  std::memcpy(key.data(), in, (size_t)n * sizeof(hydro_patch));
  std::memcpy(key.data() + (size_t)n * sizeof(hydro_patch), out, (size_t)n * sizeof(hydro_patch));
  int setting[2 * NC + 2] = {};
  for (int k = 0; k < NC && pc; ++k) {
    setting[2 * k] = 1 + class_tile(c, k);
    setting[2 * k + 1] = class_zc(c, k);
  }
  if (!pc && c->tuned) {
    setting[2 * NC] = 1 + tile;
    setting[2 * NC + 1] = zchunk;
  }
  append(key, setting, 2 * NC + 2);
  if ((*entry = c->batch.find(key))) return graph_holds(c, (*entry)->graphs);
  if (!pc && !c->tuned) default_tuning(c, in, n, &tile, &zchunk);
  // patches by class (all in class 0 without a tile shape per class) and tiles per class: the counts on
  // the host size the buffer, the device builds the list itself
  int t[NC], z[NC], cnt[NC] = {}, first[NC] = {};
  size_t tiles[NC] = {}, total = 0;
  std::vector<int> idx;
  for (int k = 0; k < (pc ? NC : 1); ++k) {
    t[k] = pc ? class_tile(c, k) : tile;
    z[k] = pc ? class_zc(c, k) : zchunk;
    const int kx = hydro::kTileX[t[k]], ky = hydro::kTileY[t[k]];
    first[k] = (int)idx.size();
    for (int i = 0; i < n; ++i) {
      if (pc && patch_class(in[i]) != k) continue;
      if (pc) idx.push_back(i);
      ++cnt[k];
      tiles[k] += (size_t)((in[i].nx + kx - 1) / kx) * ((in[i].ny + ky - 1) / ky) * ((in[i].nz + z[k] - 1) / z[k]);
    }
    total += tiles[k];
  }
  if (total > 0x7fffffff) return HYDRO_ERR_ARG;
  std::vector<HostPatchIO> io((size_t)n);
  for (int i = 0; i < n; ++i) io[i] = make_io(in[i], out[i]);
  std::vector<char> bytes;
  size_t off[4] = {};
  off[B_PATCHES] = append(bytes, io.data(), io.size());
  off[B_INDEX] = append(bytes, idx.data(), idx.size());
  auto align = [](size_t x) { return (x + 255) / 256 * 256; };
  off[B_TILES] = align(bytes.size());
  off[B_COUNTS] = align(off[B_TILES] + total * sizeof(HostTileRec));
  int rc;
  SetCache::Entry* e = new_entry(c, c->batch, off[B_COUNTS] + ((size_t)n + NC) * sizeof(int), &rc);
  if (!e) return rc;
  if (!upload(c, e->d, bytes.data(), bytes.size())) return HYDRO_ERR_CUDA;
  std::memcpy(e->off, off, sizeof(off));
  e->n[B_NTILES] = (int)total;
  e->n[B_TILE] = tile;
  e->n[B_ZCHUNK] = zchunk;
  e->n[B_PER_CLASS] = pc;
  size_t done = 0;
  for (int k = 0; k < (pc ? NC : 1); ++k) {
    e->n[B_CLS_OFF + k] = (int)done;
    e->n[B_CLS_NTILES + k] = (int)tiles[k];
    if (cnt[k]) {
      if (hydro::build_worklist(reinterpret_cast<HostPatchIO*>(e->d + off[B_PATCHES]), cnt[k], hydro::kTileX[t[k]],
                                hydro::kTileY[t[k]], z[k], reinterpret_cast<int*>(e->d + off[B_COUNTS]) + first[k] + k,
                                reinterpret_cast<HostTileRec*>(e->d + off[B_TILES]) + done, c->stream,
                                pc ? reinterpret_cast<int*>(e->d + off[B_INDEX]) + first[k] : nullptr) != cudaSuccess)
        return HYDRO_ERR_CUDA;
      c->launches += 3;
    }
    done += tiles[k];
  }
  c->batch.done(e, std::move(key));
  *entry = e;
  return HYDRO_OK;
}

int reset_slots(hydro_ctx* c, double* p, int n, cudaStream_t s) {
  // 0xFF.. is above the bits of every positive double: the neutral element of the min.
  return cuda_status(cudaMemsetAsync(p, 0xFF, (size_t)n * sizeof(double), s));
}

int step_one_uniform(hydro_ctx* c, const hydro_patch& in, const hydro_patch& out, const double* dt, double* dt_next,
                     cudaStream_t s) {
  if (dt_next) {
    int rc = reset_slots(c, dt_next, 1, s);
    if (rc) return rc;
  }
  int tile = c->tile_id, zc = c->zchunk;
  if (!c->tuned) {
    if (c->rule_n[0] != in.nx || c->rule_n[1] != in.ny || c->rule_n[2] != in.nz) {
      default_tuning(c, &in, 1, &c->rule_tile, &c->rule_zc);
      c->rule_n[0] = in.nx; c->rule_n[1] = in.ny; c->rule_n[2] = in.nz;
    }
    tile = c->rule_tile;
    zc = c->rule_zc;
  }
  zc = std::min(zc, in.nz);
  cudaError_t e = ppm(c) ? c->ops->step_ppm(make_io(in, out), c->prm, dt, dt_next, zc, c->d_err, s)
                         : c->ops->step_uniform(tile, make_io(in, out), c->prm, dt, dt_next, zc, c->d_err, s);
  c->launches += 1;
  return cuda_status(e);
}

int box_fluxes(hydro_ctx* c, int kind, const std::vector<hydro::HostBoxFluxes>& boxes, const double* dt_dev,
               int accumulate) {
  std::vector<int2> blocks;
  for (size_t b = 0; b < boxes.size(); ++b) {
    const long long nx = boxes[b].n[0], ny = boxes[b].n[1], nz = boxes[b].n[2];
    const long long faces = 2 * (ny * nz + nx * nz + nx * ny);
    if (faces > 0x7fffffffLL) return HYDRO_ERR_ARG;
    for (long long k = 0; k * 256 < faces; ++k) blocks.push_back(make_int2((int)b, (int)k));
  }
  if (blocks.size() > 0x7fffffff) return HYDRO_ERR_ARG;
  std::vector<char> bytes;
  const size_t ob = append(bytes, boxes.data(), boxes.size());
  const size_t ok = append(bytes, blocks.data(), blocks.size());
  const SetCache::Entry* e = upload_set(c, c->aux[kind], std::move(bytes));
  if (!e) return HYDRO_ERR_CUDA;
  char* d = e->d;
  c->launches += 1;
  return cuda_status(c->ops->box_fluxes(reinterpret_cast<const hydro::HostBoxFluxes*>(d + ob),
                                        reinterpret_cast<const int2*>(d + ok), (int)blocks.size(), c->prm, dt_dev,
                                        accumulate, c->stream));
}

}  // namespace

extern "C" {

const char* hydro_status_string(int status) {
  switch (status) {
    case HYDRO_OK: return "ok";
    case HYDRO_ERR_ARG: return "invalid argument";
    case HYDRO_ERR_CUDA: return "CUDA error";
    case HYDRO_ERR_UNPHYSICAL: return "unphysical state flagged on the device";
    case HYDRO_ERR_TIMEOUT: return "bounded device wait timed out";
    case HYDRO_ERR_NOMEM: return "device allocation failed";
    case HYDRO_ERR_STATE: return "invalid context state";
  }
  return "unknown status";
}

int hydro_init(hydro_ctx** ctx, const hydro_config* cfg) {
  if (!ctx) return HYDRO_ERR_ARG;
  *ctx = nullptr;
  if (!cfg) return HYDRO_ERR_ARG;
  if (!(cfg->gamma > 1.0 && std::isfinite(cfg->gamma))) return HYDRO_ERR_ARG;
  if (!(cfg->cfl > 0.0 && cfg->cfl <= 1.0)) return HYDRO_ERR_ARG;
  if (!(cfg->rho_floor >= 0.0 && cfg->p_floor >= 0.0)) return HYDRO_ERR_ARG;
  if (cfg->limiter < HYDRO_MINMOD || cfg->limiter > HYDRO_PPM) return HYDRO_ERR_ARG;
  if (!hydro::ops_for(cfg->precision)) return HYDRO_ERR_ARG;
  hydro_ctx* c = new hydro_ctx();
  c->cfg = *cfg;
  c->prm = hydro::make_params(cfg->gamma, cfg->cfl, cfg->rho_floor, cfg->p_floor, cfg->limiter);
  c->stream = static_cast<cudaStream_t>(cfg->cuda_stream);
  c->ops = hydro::ops_for(cfg->precision);
  if (cudaGetDevice(&c->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    delete c;
    return HYDRO_ERR_CUDA;
  }
  if (cudaMalloc(&c->d_err, sizeof(unsigned)) != cudaSuccess || cudaMalloc(&c->d_counter, (1 + HYDRO_NUM_PATCH_CLASSES) * sizeof(int)) != cudaSuccess) {
    hydro_finalize(c);
    return HYDRO_ERR_NOMEM;
  }
  if (cudaMemsetAsync(c->d_err, 0, sizeof(unsigned), c->stream) != cudaSuccess ||
      cudaStreamCreateWithFlags(&c->capture, cudaStreamNonBlocking) != cudaSuccess) {
    hydro_finalize(c);
    return HYDRO_ERR_CUDA;
  }
  // FP64 favours the square tile (fewest recomputed halo cells per update); others the wide one.
  c->tile_id = 0;
  c->zchunk = 32;
  *ctx = c;
  return HYDRO_OK;
}

int hydro_finalize(hydro_ctx* c) {
  if (!c) return HYDRO_OK;
  cudaStreamSynchronize(c->stream);
  if (c->graph) cudaGraphExecDestroy(c->graph);
  if (c->capture) cudaStreamDestroy(c->capture);
  cudaFree(c->d_err);
  cudaFree(c->d_counter);
  cudaFree(c->d_cls_dt);
  cudaFree(c->adj.d);
  if (c->s_h2d) cudaStreamSynchronize(c->s_h2d);
  if (c->s_d2h) cudaStreamSynchronize(c->s_d2h);
  if (c->s_cmp2) cudaStreamSynchronize(c->s_cmp2);
  cudaFree(c->d_stage);
  cudaFree(c->d_stage_io);
  cudaFree(c->d_stage_tiles);
  cudaFree(c->d_stage_counters);
  c->batch.free_all();
  c->cfl_sets.free_all();
  c->ghost_sets.free_all();
  c->xchg_sets.free_all();
  for (SetCache& s : c->aux) s.free_all();
  cudaFree(c->octs.d);
  cudaFree(c->d_octs_slots);
  cudaFree(c->d_cubes);
  cudaFree(c->mhd.d);
  for (Scratch& s : c->aside) cudaFree(s.d);
  for (cudaEvent_t e : c->ev_copied) cudaEventDestroy(e);
  for (cudaEvent_t e : c->ev_stepped) cudaEventDestroy(e);
  for (cudaEvent_t e : c->ev_halo) cudaEventDestroy(e);
  if (c->ev_begin) cudaEventDestroy(c->ev_begin);
  if (c->ev_end) cudaEventDestroy(c->ev_end);
  if (c->s_h2d) cudaStreamDestroy(c->s_h2d);
  if (c->s_d2h) cudaStreamDestroy(c->s_d2h);
  if (c->s_cmp2) cudaStreamDestroy(c->s_cmp2);
  if (c->ev_ready) cudaEventDestroy(c->ev_ready);
  for (int t = 0; t < 2; ++t) {
    cudaFreeHost(c->h_stage[t]);
    if (c->ev_stage[t]) cudaEventDestroy(c->ev_stage[t]);
  }
  delete c;
  return HYDRO_OK;
}

int hydro_cfl_dt(hydro_ctx* c, const hydro_patch* p, int npatch, double* dt_dev) {
  if (!c || !p || npatch < 1 || !dt_dev) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i)
    if (!valid_patch(c, p[i])) return HYDRO_ERR_ARG;
  int rc = reset_slots(c, dt_dev, npatch, c->stream);
  if (rc) return rc;
  if (npatch == 1) {
    c->launches += 1;
    return cuda_status(c->ops->cfl(nullptr, make_io(p[0], p[0]), 1, c->prm, dt_dev, c->d_err, c->stream));
  }
  std::vector<char> key;
  append(key, p, (size_t)npatch);
  SetCache::Entry* e = c->cfl_sets.find(key);
  if (!e) {
    std::vector<HostPatchIO> io((size_t)npatch);
    for (int i = 0; i < npatch; ++i) io[i] = make_io(p[i], p[i]);
    if (!(e = new_entry(c, c->cfl_sets, io.size() * sizeof(io[0]), &rc))) return rc;
    if (!upload(c, e->d, io.data(), io.size() * sizeof(io[0]))) return HYDRO_ERR_CUDA;
    c->cfl_sets.done(e, std::move(key));
  }
  if ((rc = graph_holds(c, e->graphs))) return rc;
  HostPatchIO big = make_io(p[0], p[0]);
  c->launches += 1;
  return cuda_status(c->ops->cfl(reinterpret_cast<const HostPatchIO*>(e->d), big, npatch, c->prm, dt_dev, c->d_err, c->stream));
}

int hydro_step(hydro_ctx* c, const hydro_patch* in, const hydro_patch* out, int npatch, const double* dt_dev,
               double* dt_next_dev) {
  if (!c || !in || !out || npatch < 1 || !dt_dev) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i) {
    if (!valid_patch(c, in[i]) || !valid_patch(c, out[i])) return HYDRO_ERR_ARG;
    if (!same_shape(in[i], out[i])) return HYDRO_ERR_ARG;
    if (overlaps(c, in[i], out[i])) return HYDRO_ERR_ARG;
  }
  if (npatch == 1 && in[0].ng == 0) return step_one_uniform(c, in[0], out[0], dt_dev, dt_next_dev, c->stream);
  for (int i = 0; i < npatch; ++i)  // ghost layers the reconstruction's stencil needs
    if (in[i].ng != (ppm(c) ? 3 : 2)) return HYDRO_ERR_ARG;
  SetCache::Entry* e = nullptr;
  int rc = prepare_batch(c, in, out, npatch, &e);
  if (rc) return rc;
  const HostPatchIO* d_patches = reinterpret_cast<const HostPatchIO*>(e->d + e->off[B_PATCHES]);
  const HostTileRec* d_tiles = reinterpret_cast<const HostTileRec*>(e->d + e->off[B_TILES]);
  const int ntiles = e->n[B_NTILES], tile = e->n[B_TILE], zchunk = e->n[B_ZCHUNK];
  if (cudaMemsetAsync(c->d_counter, 0, (1 + HYDRO_NUM_PATCH_CLASSES) * sizeof(int), c->stream) != cudaSuccess)
    return HYDRO_ERR_CUDA;
  if (dt_next_dev) {
    rc = reset_slots(c, dt_next_dev, npatch, c->stream);
    if (rc) return rc;
  }
  if (e->n[B_PER_CLASS]) {
    // one persistent launch per class, each over its own work-list segment and counter
    for (int k = 0; k < HYDRO_NUM_PATCH_CLASSES; ++k) {
      const int nt = e->n[B_CLS_NTILES + k];
      if (!nt) continue;
      const int t = class_tile(c, k);
      const int per_sm = c->ops->batched_blocks_per_sm(t, c->cfg.limiter);
      const int grid = std::max(1, std::min(nt, c->sm_count * per_sm));
      c->launches += 1;
      cudaError_t err = c->ops->step_batched(t, d_patches, d_tiles + e->n[B_CLS_OFF + k], nt, c->d_counter + 1 + k, c->prm,
                                             dt_dev, dt_next_dev, class_zc(c, k), c->d_err, grid, c->stream);
      if (err != cudaSuccess) return HYDRO_ERR_CUDA;
    }
    return HYDRO_OK;
  }
  c->launches += 1;
  if (ppm(c))
    return cuda_status(c->ops->step_ppm_batched(d_patches, d_tiles, ntiles, c->d_counter, c->prm, dt_dev, dt_next_dev,
                                                zchunk, c->d_err, c->sm_count, c->stream));
  const int per_sm = c->ops->batched_blocks_per_sm(tile, c->cfg.limiter);
  const int grid = std::max(1, std::min(ntiles, c->sm_count * per_sm));
  return cuda_status(c->ops->step_batched(tile, d_patches, d_tiles, ntiles, c->d_counter, c->prm, dt_dev, dt_next_dev,
                                          zchunk, c->d_err, grid, c->stream));
}

// Host-buffer step of one periodic box: the state crosses the host link in z slabs on two copy
// streams while the step kernel runs on the slabs that have arrived (copies of a quarter of the
// GPU hydro time and more are the paper's data-movement cost, Sec. 3 and Table 1; here they
// overlap the compute instead of preceding and following it).
//   H2D:  planes nz-2, nz-1 (slab 0's lower halo), then slabs 0 .. S-1
//   step: slab k once slab k+1 has arrived (slab S-1 wraps onto slab 0, already there)
//   D2H:  slab k once its step has run
int hydro_step_host(hydro_ctx* c, const hydro_patch* in, const hydro_patch* out, const double* dt_dev,
                    double* dt_next_dev) {
  if (!c || !in || !out || !dt_dev || ppm(c)) return HYDRO_ERR_ARG;
  const hydro_patch &I = *in, &O = *out;
  if (!valid_patch(c, I) || !valid_patch(c, O) || !same_shape(I, O) || overlaps(c, I, O)) return HYDRO_ERR_ARG;
  if (I.ng != 0 || O.ng != 0 || I.sy != O.sy || I.sz != O.sz) return HYDRO_ERR_ARG;
  for (int v = 0; v < 5; ++v) {
    for (const void* ptr : {static_cast<const void*>(I.U[v]), static_cast<const void*>(O.U[v])}) {
      cudaPointerAttributes a;
      if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) return HYDRO_ERR_CUDA;
      if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return HYDRO_ERR_ARG;
    }
  }
  const int es = elem_size(c);
  const size_t plane = (size_t)I.sz * es;
  const size_t fb = (size_t)I.nz * plane;
  // slabs: the z chunk shortened until the box has >= 16 slabs (or 2-plane chunks)
  int zc = c->zchunk;
  while (zc > 2 && I.nz / zc < 16) zc /= 2;
  // at least two planes per slab: a slab's upper halo (two planes) then lies in the next slab
  zc = std::max(std::min(2, I.nz), std::min(zc, I.nz));
  // Slab boundaries: zc planes each, but ramped at both ends (zc/4, zc/2, ..., zc/2, zc/4, each at
  // least two planes) where the box is tall enough: the first step waits for the first slab and its
  // halo to arrive, and the last copy-out waits for the last slab's step, so short end slabs cut
  // the pipeline's fill and drain.
  std::vector<int> zs;  // slab k covers planes [zs[k], zs[k+1])
  {
    const int a = std::max(2, zc / 4), b = std::max(2, zc / 2);
    const int ends = 2 * (a + b);
    zs.push_back(0);
    if (zc >= 8 && I.nz >= ends + 2 * zc) {
      for (int h : {a, b}) zs.push_back(zs.back() + h);
      const int mid = I.nz - ends, nm = mid / zc, rem = mid - nm * zc;
      for (int k = 0; k < nm; ++k) zs.push_back(zs.back() + zc);
      if (rem >= 2) zs.push_back(zs.back() + rem);
      else if (rem > 0) zs.back() += rem;  // one plane left over: the last middle slab takes it
      for (int h : {b, a}) zs.push_back(zs.back() + h);
    } else {
      for (int z = zc; z < I.nz; z += zc) zs.push_back(z);
      zs.push_back(I.nz);
    }
  }
  const int S = (int)zs.size() - 1;
  const int tx = hydro::kTileX[c->tile_id], ty = hydro::kTileY[c->tile_id];
  const int ntx = (I.nx + tx - 1) / tx, nty = (I.ny + ty - 1) / ty, tps = ntx * nty;
  // staging, descriptors, tile list, counters, streams, events
  int rc = HYDRO_OK;
  if (c->stage_cap < 10 * fb) {
    if (c->s_h2d) cudaStreamSynchronize(c->s_h2d);
    if (c->s_d2h) cudaStreamSynchronize(c->s_d2h);
    if (c->s_cmp2) cudaStreamSynchronize(c->s_cmp2);
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return HYDRO_ERR_CUDA;
    cudaFree(c->d_stage);
    c->d_stage = nullptr;
    c->stage_cap = 0;
    if (cudaMalloc(&c->d_stage, 10 * fb) != cudaSuccess) return HYDRO_ERR_NOMEM;
    c->stage_cap = 10 * fb;
    c->stage_key[0] = -1;
  }
  if (!c->d_stage_io && cudaMalloc(&c->d_stage_io, sizeof(HostPatchIO)) != cudaSuccess) return HYDRO_ERR_NOMEM;
  rc = ensure_device(&c->d_stage_tiles, &c->stage_tiles_cap, (size_t)S * tps);
  if (rc) return rc;
  rc = ensure_device(&c->d_stage_counters, &c->stage_counters_cap, (size_t)S);
  if (rc) return rc;
  if (!c->s_h2d && cudaStreamCreateWithFlags(&c->s_h2d, cudaStreamNonBlocking) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (!c->s_d2h && cudaStreamCreateWithFlags(&c->s_d2h, cudaStreamNonBlocking) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (!c->s_cmp2 && cudaStreamCreateWithFlags(&c->s_cmp2, cudaStreamNonBlocking) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (!c->ev_ready && cudaEventCreateWithFlags(&c->ev_ready, cudaEventDisableTiming) != cudaSuccess)
    return HYDRO_ERR_CUDA;
  if (!c->ev_begin && (cudaEventCreateWithFlags(&c->ev_begin, cudaEventDisableTiming) != cudaSuccess ||
                       cudaEventCreateWithFlags(&c->ev_end, cudaEventDisableTiming) != cudaSuccess))
    return HYDRO_ERR_CUDA;
  while ((int)c->ev_copied.size() < S) {
    cudaEvent_t e[3];
    for (int k = 0; k < 3; ++k)
      if (cudaEventCreateWithFlags(&e[k], cudaEventDisableTiming) != cudaSuccess) {
        for (int m = 0; m < k; ++m) cudaEventDestroy(e[m]);
        return HYDRO_ERR_CUDA;
      }
    c->ev_copied.push_back(e[0]);
    c->ev_stepped.push_back(e[1]);
    c->ev_halo.push_back(e[2]);
  }
  char* din[5];
  char* dout[5];
  for (int v = 0; v < 5; ++v) {
    din[v] = c->d_stage + v * fb;
    dout[v] = c->d_stage + (5 + v) * fb;
  }
  const long long key[7] = {I.nx, I.ny, I.nz, I.sy, I.sz, c->tile_id, zc};
  if (std::memcmp(key, c->stage_key, sizeof(key)) != 0 || c->stage_dx != I.dx) {
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return HYDRO_ERR_CUDA;
    HostPatchIO h;
    for (int v = 0; v < 5; ++v) {
      h.in[v] = din[v];
      h.out[v] = dout[v];
    }
    h.nx = I.nx; h.ny = I.ny; h.nz = I.nz; h.gin = 0; h.gout = 0;
    h.isy = h.osy = I.sy; h.isz = h.osz = I.sz; h.dx = I.dx;
    std::vector<HostTileRec> t((size_t)S * tps);
    for (int k = 0; k < S; ++k)
      for (int j = 0; j < nty; ++j)
        for (int i = 0; i < ntx; ++i) t[(size_t)k * tps + j * ntx + i] = HostTileRec{0, i * tx, j * ty, zs[k]};
    if (cudaMemcpy(c->d_stage_io, &h, sizeof(h), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(c->d_stage_tiles, t.data(), t.size() * sizeof(HostTileRec), cudaMemcpyHostToDevice) != cudaSuccess)
      return HYDRO_ERR_CUDA;
    std::memcpy(c->stage_key, key, sizeof(key));
    c->stage_dx = I.dx;
  }
  // planes [za, zb) of the five fields, one copy per field (a z range of a field is contiguous)
  auto upload = [&](int za, int zb) -> bool {
    for (int v = 0; v < 5 && zb > za; ++v)
      if (cudaMemcpyAsync(din[v] + za * plane, static_cast<const char*>(I.U[v]) + za * plane, (zb - za) * plane,
                          cudaMemcpyHostToDevice, c->s_h2d) != cudaSuccess)
        return false;
    return true;
  };
  auto download = [&](int za, int zb) -> bool {
    for (int v = 0; v < 5 && zb > za; ++v)
      if (cudaMemcpyAsync(static_cast<char*>(O.U[v]) + za * plane, dout[v] + za * plane, (zb - za) * plane,
                          cudaMemcpyDeviceToHost, c->s_d2h) != cudaSuccess)
        return false;
    return true;
  };
  // the staging buffers may still be read or written by the previous call's work
  if (cudaEventRecord(c->ev_begin, c->stream) != cudaSuccess || cudaStreamWaitEvent(c->s_h2d, c->ev_begin) != cudaSuccess ||
      cudaStreamWaitEvent(c->s_d2h, c->ev_begin) != cudaSuccess)
    return HYDRO_ERR_CUDA;
  const int tail = S > 1 ? std::max(0, I.nz - 2) : I.nz;
  if (!upload(tail, I.nz)) return HYDRO_ERR_CUDA;
  for (int k = 0; k < S; ++k) {
    const int za = zs[k], zb = std::min(zs[k + 1], tail);
    // a slab's first two planes go first: with them the previous slab's step can start
    const int zh = std::min(za + 2, zb);
    if (!upload(za, zh) || cudaEventRecord(c->ev_halo[k], c->s_h2d) != cudaSuccess || !upload(zh, zb) ||
        cudaEventRecord(c->ev_copied[k], c->s_h2d) != cudaSuccess)
      return HYDRO_ERR_CUDA;
  }
  if (cudaMemsetAsync(c->d_stage_counters, 0, (size_t)S * sizeof(int), c->stream) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (dt_next_dev) {
    rc = reset_slots(c, dt_next_dev, 1, c->stream);
    if (rc) return rc;
  }
  const int per_sm = c->ops->batched_blocks_per_sm(c->tile_id, c->cfg.limiter);
  const int grid = std::max(1, std::min(tps, c->sm_count * per_sm));
  // slabs alternate between two compute streams, so that a slab's last partial wave of tiles runs
  // beside the next slab's first (the slabs write disjoint planes; dt_next is an order-free min)
  if (cudaEventRecord(c->ev_ready, c->stream) != cudaSuccess || cudaStreamWaitEvent(c->s_cmp2, c->ev_ready) != cudaSuccess)
    return HYDRO_ERR_CUDA;
  for (int k = 0; k < S; ++k) {
    const int za = zs[k], zb = zs[k + 1];
    cudaStream_t sk = (k & 1) ? c->s_cmp2 : c->stream;
    // slab k and its upper halo: the first two planes of slab k+1 (the last slab's halo wraps onto
    // slab 0, uploaded before it)
    if (cudaStreamWaitEvent(sk, k + 1 < S ? c->ev_halo[k + 1] : c->ev_copied[S - 1]) != cudaSuccess)
      return HYDRO_ERR_CUDA;
    c->launches += 1;
    if (c->ops->step_batched(c->tile_id, c->d_stage_io, c->d_stage_tiles + (size_t)k * tps, tps,
                             c->d_stage_counters + k, c->prm, dt_dev, dt_next_dev, zb - za, c->d_err, grid,
                             sk) != cudaSuccess)
      return HYDRO_ERR_CUDA;
    if (cudaEventRecord(c->ev_stepped[k], sk) != cudaSuccess ||
        cudaStreamWaitEvent(c->s_d2h, c->ev_stepped[k]) != cudaSuccess)
      return HYDRO_ERR_CUDA;
    if (!download(za, zb)) return HYDRO_ERR_CUDA;
  }
  if (cudaEventRecord(c->ev_end, c->s_d2h) != cudaSuccess || cudaStreamWaitEvent(c->stream, c->ev_end) != cudaSuccess)
    return HYDRO_ERR_CUDA;
  return HYDRO_OK;
}

int hydro_step_octs(hydro_ctx* c, void* const gathered[5], void* const out[5], long long ngroups, double dx,
                    const double* dt_dev) {
  if (!c || !gathered || !out || ngroups < 1 || !finite_pos(dx) || !dt_dev || ppm(c)) return HYDRO_ERR_ARG;
  const int es = elem_size(c);
  for (int v = 0; v < 5; ++v) {
    if (!gathered[v] || !out[v]) return HYDRO_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(gathered[v]) % es || reinterpret_cast<uintptr_t>(out[v]) % es) return HYDRO_ERR_ARG;
  }
  c->launches += 1;
  return cuda_status(c->ops->octs(gathered, out, ngroups, dx, c->prm, dt_dev, c->d_err, c->stream));
}

// The ghost fill from the coarse level after its step (coarse_old == nullptr), or at the fraction
// theta of its step between coarse_old and coarse.
static int fill_ghosts_impl(hydro_ctx* c, const hydro_patch* coarse, const hydro_patch* coarse_old, double theta,
                            const hydro_patch* fine, const int* fine_origins, int npatch) {
  if (!c || !coarse || !fine || !fine_origins || npatch < 1) return HYDRO_ERR_ARG;
  const hydro_patch& C = *coarse;
  if (!valid_patch(c, C) || C.ng != 0) return HYDRO_ERR_ARG;
  if (coarse_old) {
    const hydro_patch& O = *coarse_old;
    if (!valid_patch(c, O) || O.ng != 0 || !same_shape(O, C) || O.sy != C.sy || O.sz != C.sz) return HYDRO_ERR_ARG;
    if (!(theta >= 0.0 && theta <= 1.0)) return HYDRO_ERR_ARG;
  }
  std::vector<hydro::HostGhostPatch> set((size_t)npatch);
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch& F = fine[i];
    if (!valid_patch(c, F) || F.ng != 2 || F.dx != 0.5 * C.dx || overlaps(c, C, F)) return HYDRO_ERR_ARG;
    hydro::HostGhostPatch& g = set[i];
    for (int v = 0; v < 5; ++v) g.U[v] = F.U[v];
    g.nx = F.nx; g.ny = F.ny; g.nz = F.nz;
    g.ox = fine_origins[3 * i]; g.oy = fine_origins[3 * i + 1]; g.oz = fine_origins[3 * i + 2];
    g.sy = F.sy; g.sz = F.sz;
    const int o[3] = {g.ox, g.oy, g.oz}, nn[3] = {F.nx, F.ny, F.nz};
    long long cells = 1;
    for (int d = 0; d < 3; ++d) {  // coarse cells floor((o-2)/2) .. floor((o+n+1)/2)
      const long long lo = (long long)std::floor((o[d] - 2) / 2.0), hi = (long long)std::floor((o[d] + nn[d] + 1) / 2.0);
      if (lo < -0x3fffffffLL || hi > 0x3fffffffLL) return HYDRO_ERR_ARG;
      g.clo[d] = (int)lo;
      g.cm[d] = (int)(hi - lo + 1);
      cells *= g.cm[d];
    }
    if (cells > 0x7fffffff) return HYDRO_ERR_ARG;
  }
  std::vector<char> key;
  append(key, set.data(), set.size());
  SetCache::Entry* e = c->ghost_sets.find(key);
  if (!e) {
    std::vector<int2> blocks;
    for (int i = 0; i < npatch; ++i)
      for (int first = 0; first < set[i].cm[0] * set[i].cm[1] * set[i].cm[2]; first += 256)
        blocks.push_back(make_int2(i, first));
    if (blocks.size() > 0x7fffffff) return HYDRO_ERR_ARG;
    std::vector<char> bytes = key;
    const size_t off = append(bytes, blocks.data(), blocks.size());
    int rc;
    if (!(e = new_entry(c, c->ghost_sets, bytes.size(), &rc))) return rc;
    if (!upload(c, e->d, bytes.data(), bytes.size())) return HYDRO_ERR_CUDA;
    e->off[1] = off;
    e->n[0] = (int)blocks.size();
    c->ghost_sets.done(e, std::move(key));
  }
  if (int rc = graph_holds(c, e->graphs)) return rc;
  c->launches += 1;
  const HostPatchIO old = coarse_old ? make_io(*coarse_old, *coarse_old) : make_io(C, C);
  return cuda_status(hydro::launch_fill_ghosts(elem_size(c), reinterpret_cast<const hydro::HostGhostPatch*>(e->d),
                                               reinterpret_cast<const int2*>(e->d + e->off[1]), e->n[0], make_io(C, C),
                                               coarse_old ? &old : nullptr, theta, c->stream));
}

int hydro_fill_ghosts(hydro_ctx* c, const hydro_patch* coarse, const hydro_patch* fine, const int* fine_origins,
                      int npatch) {
  return fill_ghosts_impl(c, coarse, nullptr, 1.0, fine, fine_origins, npatch);
}

int hydro_fill_ghosts_time(hydro_ctx* c, const hydro_patch* coarse_old, const hydro_patch* coarse_new, double theta,
                           const hydro_patch* fine, const int* fine_origins, int npatch) {
  if (!coarse_old) return HYDRO_ERR_ARG;
  return fill_ghosts_impl(c, coarse_new, coarse_old, theta, fine, fine_origins, npatch);
}

// Copy tasks of the same-level exchange: for each destination patch, every periodic image of every
// patch interior (its own included) that meets its ghosted box.  Candidate sources come from a
// coarse spatial hash of the interiors (64-cell bins over the period).
static std::vector<hydro::HostCopyTask> exchange_tasks(const std::vector<hydro::HostGhostPatch>& P, const int per[3]) {
  const int n = (int)P.size();
  const int B = 64;
  int nb[3];
  for (int d = 0; d < 3; ++d) nb[d] = std::max(1, (per[d] + B - 1) / B);
  auto org = [&](int p, int d) { const int o[3] = {P[p].ox, P[p].oy, P[p].oz}; return ((o[d] % per[d]) + per[d]) % per[d]; };
  auto dim = [&](int p, int d) { return d == 0 ? P[p].nx : (d == 1 ? P[p].ny : P[p].nz); };
  std::vector<std::vector<int>> bins((size_t)nb[0] * nb[1] * nb[2]);
  // bins met by the positions [lo, hi) of axis d, each position wrapped into [0, period) first
  auto bins_of = [&](int lo, int hi, int d) {
    std::vector<int> out;
    for (int x = lo; x < hi; ++x) {
      const int b = (((x % per[d]) + per[d]) % per[d]) / B;
      if (out.empty() || out.back() != b)
        if (std::find(out.begin(), out.end(), b) == out.end()) out.push_back(b);
    }
    return out;
  };
  for (int p = 0; p < n; ++p) {
    const std::vector<int> bx = bins_of(org(p, 0), org(p, 0) + dim(p, 0), 0);
    const std::vector<int> by = bins_of(org(p, 1), org(p, 1) + dim(p, 1), 1);
    const std::vector<int> bz = bins_of(org(p, 2), org(p, 2) + dim(p, 2), 2);
    for (int z : bz)
      for (int y : by)
        for (int x : bx) bins[((size_t)z * nb[1] + y) * nb[0] + x].push_back(p);
  }
  std::vector<hydro::HostCopyTask> tasks;
  std::vector<int> seen(n, -1);
  for (int a = 0; a < n; ++a) {
    int glo[3], ghi[3];
    for (int d = 0; d < 3; ++d) {
      glo[d] = org(a, d) - 2;
      ghi[d] = org(a, d) + dim(a, d) + 2;
    }
    const std::vector<int> bx = bins_of(glo[0], ghi[0], 0), by = bins_of(glo[1], ghi[1], 1), bz = bins_of(glo[2], ghi[2], 2);
    std::vector<int> cand;
    for (int z : bz)
      for (int y : by)
        for (int x : bx)
          for (int q : bins[((size_t)z * nb[1] + y) * nb[0] + x])
            if (seen[q] != a) { seen[q] = a; cand.push_back(q); }
    for (int b : cand) {
      // per axis, the images (shift k periods) of b's interior that meet a's ghosted box, at most a
      // few of the five: their product instead of 125 tests per candidate
      struct Image { int k, lo, hi, s; } im[3][5];
      int ni[3] = {0, 0, 0};
      for (int d = 0; d < 3; ++d)
        for (int k = -2; k <= 2; ++k) {
          const int s = org(b, d) + k * per[d], lo = std::max(glo[d], s), hi = std::min(ghi[d], s + dim(b, d));
          if (lo < hi) im[d][ni[d]++] = {k, lo, hi, s};
        }
      for (int z = 0; z < ni[2]; ++z)
        for (int y = 0; y < ni[1]; ++y)
          for (int x = 0; x < ni[0]; ++x) {
            const Image m[3] = {im[0][x], im[1][y], im[2][z]};
            if (b == a && m[0].k == 0 && m[1].k == 0 && m[2].k == 0) continue;  // its own interior
            hydro::HostCopyTask t;
            t.dst = a;
            t.src = b;
            for (int d = 0; d < 3; ++d) {
              t.dlo[d] = m[d].lo - glo[d];
              t.slo[d] = m[d].lo - m[d].s + 2;
              t.n[d] = m[d].hi - m[d].lo;
            }
            tasks.push_back(t);
          }
    }
  }
  return tasks;
}

int hydro_patch_fluxes(hydro_ctx* c, const hydro_patch* patches, int npatch, const double* dt_dev,
                       void* const* registers, int accumulate) {
  if (!c || !patches || npatch < 1 || !dt_dev || !registers || ppm(c)) return HYDRO_ERR_ARG;
  std::vector<hydro::HostBoxFluxes> boxes((size_t)npatch);
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch& P = patches[i];
    if (!valid_patch(c, P) || P.ng != 2 || !registers[i]) return HYDRO_ERR_ARG;
    hydro::HostBoxFluxes& b = boxes[i];
    for (int v = 0; v < 5; ++v) b.U[v] = P.U[v];
    b.reg = registers[i];
    b.n[0] = P.nx; b.n[1] = P.ny; b.n[2] = P.nz;
    for (int d = 0; d < 3; ++d) b.o[d] = b.N[d] = 0;
    b.periodic = 0;
    b.dt_index = i;
    b.sy = P.sy; b.sz = P.sz;
    b.dx = P.dx;
  }
  return box_fluxes(c, 0, boxes, dt_dev, accumulate);
}

int hydro_level_fluxes(hydro_ctx* c, const hydro_patch* level, const int* box_origins, const int* box_dims, int nbox,
                       const double* dt_dev, void* const* registers, int accumulate) {
  if (!c || !level || !box_origins || !box_dims || nbox < 1 || !dt_dev || !registers || ppm(c)) return HYDRO_ERR_ARG;
  const hydro_patch& L = *level;
  if (!valid_patch(c, L) || L.ng != 0) return HYDRO_ERR_ARG;
  std::vector<hydro::HostBoxFluxes> boxes((size_t)nbox);
  for (int i = 0; i < nbox; ++i) {
    hydro::HostBoxFluxes& b = boxes[i];
    for (int v = 0; v < 5; ++v) b.U[v] = L.U[v];
    b.reg = registers[i];
    b.N[0] = L.nx; b.N[1] = L.ny; b.N[2] = L.nz;
    for (int d = 0; d < 3; ++d) {
      b.n[d] = box_dims[3 * i + d];
      b.o[d] = ((box_origins[3 * i + d] % b.N[d]) + b.N[d]) % b.N[d];  // wrapped into [0, N)
      if (b.n[d] < 1 || b.n[d] > b.N[d]) return HYDRO_ERR_ARG;
    }
    if (!b.reg) return HYDRO_ERR_ARG;
    b.periodic = 1;
    b.dt_index = 0;
    b.sy = L.sy; b.sz = L.sz;
    b.dx = L.dx;
  }
  return box_fluxes(c, 1, boxes, dt_dev, accumulate);
}

int hydro_reflux(hydro_ctx* c, const hydro_patch* coarse, const int* box_origins, const int* box_dims, int nbox,
                 void* const* coarse_registers, void* const* fine_registers) {
  if (!c || !coarse || !box_origins || !box_dims || nbox < 1 || !coarse_registers || !fine_registers)
    return HYDRO_ERR_ARG;
  const hydro_patch& C = *coarse;
  if (!valid_patch(c, C) || C.ng != 0) return HYDRO_ERR_ARG;
  std::vector<hydro::HostRefluxBox> boxes((size_t)nbox);
  std::vector<int2> tables[6];
  for (int i = 0; i < nbox; ++i) {
    hydro::HostRefluxBox& b = boxes[i];
    for (int d = 0; d < 3; ++d) {
      b.o[d] = box_origins[3 * i + d];
      b.n[d] = box_dims[3 * i + d];
      if (b.n[d] < 1) return HYDRO_ERR_ARG;
    }
    b.rc = coarse_registers[i];
    b.rf = fine_registers[i];
    if (!b.rc || !b.rf) return HYDRO_ERR_ARG;
    b.dx = C.dx;
    const long long faces[3] = {(long long)b.n[1] * b.n[2], (long long)b.n[0] * b.n[2], (long long)b.n[0] * b.n[1]};
    for (int t = 0; t < 6; ++t)
      for (long long k = 0; k * 256 < faces[t >> 1]; ++k) tables[t].push_back(make_int2(i, (int)k));
  }
  std::vector<char> bytes;
  const size_t ob = append(bytes, boxes.data(), boxes.size());
  size_t ot[6];
  int nb[6];
  for (int t = 0; t < 6; ++t) {
    if (tables[t].size() > 0x7fffffff) return HYDRO_ERR_ARG;
    ot[t] = append(bytes, tables[t].data(), tables[t].size());
    nb[t] = (int)tables[t].size();
  }
  const SetCache::Entry* e = upload_set(c, c->aux[2], std::move(bytes));
  if (!e) return HYDRO_ERR_CUDA;
  char* d = e->d;
  const int2* dt[6];
  for (int t = 0; t < 6; ++t) dt[t] = reinterpret_cast<const int2*>(d + ot[t]);
  c->launches += 6;
  return cuda_status(hydro::launch_reflux(elem_size(c), reinterpret_cast<const hydro::HostRefluxBox*>(d + ob), dt, nb,
                                          make_io(C, C), c->stream));
}

int hydro_average_down(hydro_ctx* c, const hydro_patch* coarse, const hydro_patch* fine, const int* fine_origins,
                       int npatch) {
  if (!c || !coarse || !fine || !fine_origins || npatch < 1) return HYDRO_ERR_ARG;
  const hydro_patch& C = *coarse;
  if (!valid_patch(c, C) || C.ng != 0) return HYDRO_ERR_ARG;
  std::vector<hydro::HostGhostPatch> set((size_t)npatch);
  std::vector<int2> blocks;
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch& F = fine[i];
    const int o[3] = {fine_origins[3 * i], fine_origins[3 * i + 1], fine_origins[3 * i + 2]};
    if (!valid_patch(c, F) || F.ng != 2 || overlaps(c, C, F)) return HYDRO_ERR_ARG;
    if ((F.nx | F.ny | F.nz | o[0] | o[1] | o[2]) & 1) return HYDRO_ERR_ARG;  // aligned with coarse cells
    hydro::HostGhostPatch& g = set[i];
    for (int v = 0; v < 5; ++v) g.U[v] = F.U[v];
    g.nx = F.nx; g.ny = F.ny; g.nz = F.nz;
    g.ox = o[0]; g.oy = o[1]; g.oz = o[2];
    for (int d = 0; d < 3; ++d) g.clo[d] = g.cm[d] = 0;
    g.sy = F.sy; g.sz = F.sz;
    const long long cells = (long long)(F.nx / 2) * (F.ny / 2) * (F.nz / 2);
    for (long long k = 0; k * 256 < cells; ++k) blocks.push_back(make_int2(i, (int)k));
  }
  std::vector<char> bytes;
  const size_t op = append(bytes, set.data(), set.size());
  const size_t obk = append(bytes, blocks.data(), blocks.size());
  const SetCache::Entry* e = upload_set(c, c->aux[3], std::move(bytes));
  if (!e) return HYDRO_ERR_CUDA;
  char* d = e->d;
  c->launches += 1;
  return cuda_status(hydro::launch_average_down(elem_size(c), reinterpret_cast<const hydro::HostGhostPatch*>(d + op),
                                                reinterpret_cast<const int2*>(d + obk), (int)blocks.size(),
                                                make_io(C, C), c->stream));
}

int hydro_exchange_ghosts(hydro_ctx* c, const hydro_patch* fine, const int* origins, int npatch, const int period[3]) {
  if (!c || !fine || !origins || !period || npatch < 1) return HYDRO_ERR_ARG;
  for (int d = 0; d < 3; ++d)
    if (period[d] < 1) return HYDRO_ERR_ARG;
  std::vector<hydro::HostGhostPatch> set((size_t)npatch);
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch& F = fine[i];
    if (!valid_patch(c, F) || F.ng != 2 || F.nx > period[0] || F.ny > period[1] || F.nz > period[2])
      return HYDRO_ERR_ARG;
    hydro::HostGhostPatch& g = set[i];
    for (int v = 0; v < 5; ++v) g.U[v] = F.U[v];
    g.nx = F.nx; g.ny = F.ny; g.nz = F.nz;
    g.ox = origins[3 * i]; g.oy = origins[3 * i + 1]; g.oz = origins[3 * i + 2];
    for (int d = 0; d < 3; ++d) g.clo[d] = g.cm[d] = 0;
    g.sy = F.sy; g.sz = F.sz;
  }
  std::vector<char> key;
  append(key, set.data(), set.size());
  append(key, period, 3);
  SetCache::Entry* e = c->xchg_sets.find(key);
  if (!e) {
    const std::vector<hydro::HostCopyTask> tasks = exchange_tasks(set, period);
    if (tasks.size() > 0x7fffffff) return HYDRO_ERR_ARG;
    std::vector<char> bytes;
    append(bytes, set.data(), set.size());
    const size_t off = append(bytes, tasks.data(), tasks.size());
    int rc;
    if (!(e = new_entry(c, c->xchg_sets, bytes.size(), &rc))) return rc;
    if (!upload(c, e->d, bytes.data(), bytes.size())) return HYDRO_ERR_CUDA;
    e->off[1] = off;
    e->n[0] = (int)tasks.size();
    c->xchg_sets.done(e, std::move(key));
  }
  if (int rc = graph_holds(c, e->graphs)) return rc;
  if (e->n[0] == 0) return HYDRO_OK;
  c->launches += 1;
  return cuda_status(hydro::launch_copy_boxes(elem_size(c), reinterpret_cast<const hydro::HostGhostPatch*>(e->d),
                                              reinterpret_cast<const hydro::HostCopyTask*>(e->d + e->off[1]), e->n[0],
                                              c->stream));
}

int hydro_step_octs_level(hydro_ctx* c, const hydro_patch* level, const int* origins_dev, long long ngroups,
                          void* const out[5], const double* dt_dev) {
  if (!c || !level || !origins_dev || !out || ngroups < 1 || !dt_dev || ppm(c)) return HYDRO_ERR_ARG;
  const hydro_patch& L = *level;
  if (!valid_patch(c, L) || L.ng != 0 || L.nx < 4 || L.ny < 4 || L.nz < 4) return HYDRO_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(origins_dev) % sizeof(int)) return HYDRO_ERR_ARG;
  const int es = elem_size(c);
  for (int v = 0; v < 5; ++v)
    if (!out[v] || reinterpret_cast<uintptr_t>(out[v]) % es) return HYDRO_ERR_ARG;
  c->launches += 1;
  return cuda_status(c->ops->octs_level(make_io(L, L), origins_dev, out, ngroups, c->prm, dt_dev, c->d_err, c->stream));
}

int hydro_octs_build(hydro_ctx* c, const int* pos_dev, int noct, const int dims[3], int* order_dev, int* nbr_dev) {
  if (!c || !pos_dev || !dims || !order_dev || noct < 1 || noct > (1 << 28)) return HYDRO_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(pos_dev) % sizeof(int) || reinterpret_cast<uintptr_t>(order_dev) % sizeof(int) ||
      reinterpret_cast<uintptr_t>(nbr_dev) % sizeof(int))
    return HYDRO_ERR_ARG;
  int bits = 0;
  for (int d = 0; d < 3; ++d) {
    if (dims[d] < 1 || dims[d] > 1024) return HYDRO_ERR_ARG;
    while ((1 << bits) < dims[d]) ++bits;
  }
  const size_t nwords = std::max<size_t>(1, ((size_t)1 << (3 * bits)) >> 5);
  const size_t nblocks = (nwords + 1023) / 1024;
  int rc = ensure_scratch(c, c->octs, (2 * nwords + nblocks) * sizeof(unsigned));
  if (rc) return rc;
  // Octs by key as well, where the key space is at most eight times the octs (a refined half of a level
  // per axis): beyond, clearing it costs more than the table's rank lookups.  A captured call, and one
  // without the memory, looks ranks up.
  const bool slots = nbr_dev && 32 * nwords <= 8 * (size_t)noct &&
                     eager_scratch(c, &c->d_octs_slots, &c->octs_slots_cap, 32 * nwords);
  unsigned* bitmap = reinterpret_cast<unsigned*>(c->octs.d);
  c->launches += nbr_dev ? 5 : 4;
  return cuda_status(hydro::launch_octs_build(pos_dev, noct, dims, bitmap, bitmap + nwords, bitmap + 2 * nwords, nwords,
                                              slots ? c->d_octs_slots : nullptr, order_dev, nbr_dev, c->d_err,
                                              c->stream));
}

int hydro_step_octs_table(hydro_ctx* c, void* const in[5], void* const out[5], int noct, const int* nbr_dev,
                          const int* list_dev, long long ngroups, double dx, const double* dt_dev) {
  if (!c || !in || !out || noct < 1 || !nbr_dev || !list_dev || ngroups < 1 || !finite_pos(dx) || !dt_dev || ppm(c))
    return HYDRO_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(nbr_dev) % sizeof(int) || reinterpret_cast<uintptr_t>(list_dev) % sizeof(int))
    return HYDRO_ERR_ARG;
  const int es = elem_size(c);
  const uintptr_t bytes = (uintptr_t)noct * 8 * es;
  for (int v = 0; v < 5; ++v) {
    if (!in[v] || !out[v]) return HYDRO_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(in[v]) % es || reinterpret_cast<uintptr_t>(out[v]) % es) return HYDRO_ERR_ARG;
  }
  for (int v = 0; v < 5; ++v)  // out is written while in is read as neighbours: no overlap
    for (int u = 0; u < 5; ++u) {
      const uintptr_t a = reinterpret_cast<uintptr_t>(out[v]), b = reinterpret_cast<uintptr_t>(in[u]);
      if (a < b + bytes && b < a + bytes) return HYDRO_ERR_ARG;
    }
  // A long list: its 4^3 cubes of octs are found first and stepped as boxes of 8^3 cells.  Lists too short
  // for one cube per SM keep the one-oct kernel, which needs no scratch, as does a captured call (its graph
  // then holds no memory of the context's) or one whose scratch cannot be allocated.
  hydro::OctCubes cubes;
  bool use = false;
  if (ngroups >= 64LL * c->sm_count && ngroups <= 0x7fffffffLL - 64) {
    const size_t ints = 2 + (size_t)ngroups / 64 + (size_t)ngroups;
    use = eager_scratch(c, &c->d_cubes, &c->cubes_cap, ints * sizeof(int) + (size_t)ngroups);
    if (use) {
      cubes.counts = reinterpret_cast<int*>(c->d_cubes);
      cubes.start = cubes.counts + 2;
      cubes.left = cubes.start + ngroups / 64;
      cubes.max_cubes = (int)(ngroups / 64);
      cubes.covered = reinterpret_cast<unsigned char*>(cubes.left + ngroups);
      if (hydro::find_oct_cubes(list_dev, ngroups, nbr_dev, noct, cubes, c->stream) != cudaSuccess) return HYDRO_ERR_CUDA;
      c->launches += 3;
    }
  }
  c->launches += 1;
  return cuda_status(c->ops->octs_table(in, nbr_dev, noct, list_dev, out, ngroups, dx, c->prm, dt_dev, c->d_err,
                                        use ? &cubes : nullptr, c->stream));
}

// Arguments of the MHD calls: a periodic box of nine contiguous fields in a context with a PLM
// limiter.
static bool mhd_args(const hydro_ctx* c, void* const* U, int nx, int ny, int nz, double dx) {
  if (!c || !U || nx < 1 || ny < 1 || nz < 1 || !finite_pos(dx)) return false;
  if ((long long)nx * ny * nz > 0x7fffffffLL) return false;
  if (ppm(c)) return false;
  const int es = elem_size(c);
  for (int v = 0; v < 9; ++v)
    if (!U[v] || reinterpret_cast<uintptr_t>(U[v]) % es) return false;
  return true;
}

static hydro::HostMhdBox mhd_box(void* const* in, void* const* out, int nx, int ny, int nz, double dx) {
  hydro::HostMhdBox h;
  for (int v = 0; v < 9; ++v) {
    h.in[v] = in[v];
    h.out[v] = out ? out[v] : nullptr;
  }
  h.nx = nx; h.ny = ny; h.nz = nz;
  h.dx = dx;
  return h;
}

int hydro_mhd_step(hydro_ctx* c, void* const in[9], void* const out[9], int nx, int ny, int nz, double dx,
                   const double* dt_dev, double* dt_next_dev) {
  if (!mhd_args(c, in, nx, ny, nz, dx) || !mhd_args(c, out, nx, ny, nz, dx) || !dt_dev) return HYDRO_ERR_ARG;
  const uintptr_t bytes = (uintptr_t)nx * ny * nz * elem_size(c);
  for (int v = 0; v < 9; ++v)  // out is written while in is read by other cells: no overlap
    for (int u = 0; u < 9; ++u) {
      const uintptr_t a = reinterpret_cast<uintptr_t>(out[v]), b = reinterpret_cast<uintptr_t>(in[u]);
      if (a < b + bytes && b < a + bytes) return HYDRO_ERR_ARG;
    }
  int rc = ensure_scratch(c, c->mhd, hydro::mhd_scratch_bytes(c->cfg.precision, nx, ny, nz, elem_size(c)));
  if (rc) return rc;
  if (dt_next_dev) {
    rc = reset_slots(c, dt_next_dev, 1, c->stream);
    if (rc) return rc;
  }
  c->launches += hydro::mhd_step_launches(c->cfg.precision);
  return cuda_status(hydro::launch_mhd_step(c->cfg.precision, mhd_box(in, out, nx, ny, nz, dx), c->prm, dt_dev,
                                            dt_next_dev, c->mhd.d, c->d_err, c->stream));
}

int hydro_mhd_cfl_dt(hydro_ctx* c, void* const U[9], int nx, int ny, int nz, double dx, double* dt_dev) {
  if (!mhd_args(c, U, nx, ny, nz, dx) || !dt_dev) return HYDRO_ERR_ARG;
  int rc = reset_slots(c, dt_dev, 1, c->stream);
  if (rc) return rc;
  c->launches += 1;
  return cuda_status(
      hydro::launch_mhd_cfl(c->cfg.precision, mhd_box(U, nullptr, nx, ny, nz, dx), c->prm, dt_dev, c->d_err, c->stream));
}

// A patch of the batched MHD calls: sizes, ghost layers (2; 0 also allowed for an output unless
// ghosts_only), strides and pointers.
static bool mhd_patch_ok(const hydro_ctx* c, const hydro_mhd_patch& p, bool ghosts_only) {
  if (p.nx < 1 || p.ny < 1 || p.nz < 1 || !finite_pos(p.dx)) return false;
  if (p.ng != 2 && !(p.ng == 0 && !ghosts_only)) return false;
  const long long gx = p.nx + 2LL * p.ng, gy = p.ny + 2LL * p.ng;
  if (p.sy < gx || p.sz < p.sy * gy) return false;
  if ((long long)(p.nx + 2) * (p.ny + 2) * (p.nz + 2) > 0x7fffff00LL) return false;
  const int es = elem_size(c);
  for (int v = 0; v < 9; ++v)
    if (!p.U[v] || reinterpret_cast<uintptr_t>(p.U[v]) % es) return false;
  return true;
}

static size_t mhd_patch_bytes(const hydro_ctx* c, const hydro_mhd_patch& p) {
  return (size_t)(p.nz + 2 * p.ng) * (size_t)p.sz * elem_size(c);
}

// Descriptors and the block table of a patch set, uploaded (or reused) as aux kind `kind`: with
// tiles, the fused step's tile records (patch, x0, y0, z0) when the precision has them, else 256
// extended cells of one patch per block; returns the device descriptors, table, count and the
// per-cell scratch elements.
static int mhd_patch_tables(hydro_ctx* c, int kind, const hydro_mhd_patch* in, const hydro_mhd_patch* out, int npatch,
                            bool tiles, const hydro::HostMhdPatch** d_patches, const void** d_blocks, int* nblocks,
                            size_t* scratch_elems) {
  std::vector<hydro::HostMhdPatch> set((size_t)npatch);
  std::vector<int2> blocks;
  std::vector<int4> recs;
  int tx = 0, ty = 0, zc = 0;
  tiles = tiles && hydro::mhd_patch_tiles(c->cfg.precision, &tx, &ty, &zc);
  long long off = 0;
  for (int i = 0; i < npatch; ++i) {
    const hydro_mhd_patch& I = in[i];
    const hydro_mhd_patch& O = out ? out[i] : in[i];
    hydro::HostMhdPatch& h = set[i];
    for (int v = 0; v < 9; ++v) {
      h.in[v] = I.U[v];
      h.out[v] = O.U[v];
    }
    h.nx = I.nx; h.ny = I.ny; h.nz = I.nz; h.gout = O.ng;
    h.isy = I.sy; h.isz = I.sz; h.osy = O.sy; h.osz = O.sz;
    h.dx = I.dx;
    h.scratch = off;
    if (tiles) {
      h.scratch = 0;
      for (int z = 0; z < I.nz; z += zc)
        for (int y = 0; y < I.ny; y += ty)
          for (int x = 0; x < I.nx; x += tx) recs.push_back(make_int4(i, x, y, z));
      continue;
    }
    const long long ec = (long long)(I.nx + 2) * (I.ny + 2) * (I.nz + 2);
    off += 81 * ec;
    for (long long f = 0; f < ec; f += 256) blocks.push_back(make_int2(i, (int)f));
  }
  if (blocks.size() > 0x7fffffff || recs.size() > 0x7fffffff) return HYDRO_ERR_ARG;
  std::vector<char> bytes;
  const size_t op = append(bytes, set.data(), set.size());
  const size_t ob = tiles ? append(bytes, recs.data(), recs.size()) : append(bytes, blocks.data(), blocks.size());
  const SetCache::Entry* e = upload_set(c, c->aux[kind], std::move(bytes));
  if (!e) return HYDRO_ERR_CUDA;
  char* d = e->d;
  *d_patches = reinterpret_cast<const hydro::HostMhdPatch*>(d + op);
  *d_blocks = d + ob;
  *nblocks = (int)(tiles ? recs.size() : blocks.size());
  *scratch_elems = (size_t)off;
  return HYDRO_OK;
}

int hydro_mhd_step_patches(hydro_ctx* c, const hydro_mhd_patch* in, const hydro_mhd_patch* out, int npatch,
                           const double* dt_dev, double* dt_next_dev) {
  if (!c || !in || !out || npatch < 1 || !dt_dev) return HYDRO_ERR_ARG;
  if (ppm(c)) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i) {
    const hydro_mhd_patch &I = in[i], &O = out[i];
    if (!mhd_patch_ok(c, I, true) || !mhd_patch_ok(c, O, false)) return HYDRO_ERR_ARG;
    if (I.nx != O.nx || I.ny != O.ny || I.nz != O.nz || I.dx != O.dx) return HYDRO_ERR_ARG;
    const size_t bi = mhd_patch_bytes(c, I), bo = mhd_patch_bytes(c, O);
    for (int v = 0; v < 9; ++v)  // the output is written while the input is read: no overlap
      for (int u = 0; u < 9; ++u) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(O.U[v]), b = reinterpret_cast<uintptr_t>(I.U[u]);
        if (a < b + bi && b < a + bo) return HYDRO_ERR_ARG;
      }
  }
  const hydro::HostMhdPatch* dp = nullptr;
  const void* db = nullptr;
  int nb = 0;
  size_t elems = 0;
  int rc = mhd_patch_tables(c, 4, in, out, npatch, true, &dp, &db, &nb, &elems);
  if (rc) return rc;
  rc = ensure_scratch(c, c->mhd, hydro::mhd_patch_consts_bytes(npatch) + elems * elem_size(c));
  if (rc) return rc;
  if (dt_next_dev) {
    rc = reset_slots(c, dt_next_dev, npatch, c->stream);
    if (rc) return rc;
  }
  c->launches += hydro::mhd_step_launches(c->cfg.precision);
  return cuda_status(hydro::launch_mhd_patches(c->cfg.precision, dp, db, nb, npatch, c->prm, dt_dev, dt_next_dev,
                                               c->mhd.d, c->d_err, c->stream));
}

int hydro_mhd_cfl_patches(hydro_ctx* c, const hydro_mhd_patch* p, int npatch, double* dt_dev) {
  if (!c || !p || npatch < 1 || !dt_dev) return HYDRO_ERR_ARG;
  if (ppm(c)) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i)
    if (!mhd_patch_ok(c, p[i], true)) return HYDRO_ERR_ARG;
  const hydro::HostMhdPatch* dp = nullptr;
  const void* db = nullptr;
  int nb = 0;
  size_t elems = 0;
  int rc = mhd_patch_tables(c, 5, p, nullptr, npatch, false, &dp, &db, &nb, &elems);
  if (rc) return rc;
  rc = reset_slots(c, dt_dev, npatch, c->stream);
  if (rc) return rc;
  c->launches += 1;
  return cuda_status(hydro::launch_mhd_patches_cfl(c->cfg.precision, dp, static_cast<const int2*>(db), nb, c->prm,
                                                   dt_dev, c->d_err, c->stream));
}

int hydro_adjoint_step(hydro_ctx* c, const hydro_patch* U_n, const double* dt_dev, const hydro_patch* lam_np1,
                       const hydro_patch* lam_n, int npatch) {
  if (!c || !U_n || !dt_dev || !lam_np1 || !lam_n || npatch < 1 || ppm(c)) return HYDRO_ERR_ARG;
  if (c->cfg.precision == HYDRO_MIXED) return HYDRO_ERR_ARG;
  // The double-float context runs the FP64 reverse sweep: on GB300 it is faster than the same
  // sweep in double-float arithmetic, whose register footprint (~240 per thread) leaves too few
  // warps per SM to cover the FP32 pipes' dependent chains; both keep the FP64 accuracy.
  const hydro::KernelOps* aops = c->cfg.precision == HYDRO_FP64_DF ? hydro::ops_for(HYDRO_FP64) : c->ops;
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch &U = U_n[i], &L = lam_np1[i], &O = lam_n[i];
    if (!valid_patch(c, U) || !valid_patch(c, L) || !valid_patch(c, O)) return HYDRO_ERR_ARG;
    if (U.ng != 0 || L.ng != 0 || O.ng != 0) return HYDRO_ERR_ARG;
    if (!same_shape(U, L) || !same_shape(U, O)) return HYDRO_ERR_ARG;
    if (overlaps(c, L, O) || overlaps(c, U, O)) return HYDRO_ERR_ARG;
  }
  for (int i = 0; i < npatch; ++i) {
    const hydro_patch &U = U_n[i], &L = lam_np1[i], &O = lam_n[i];
    const size_t need = aops->adjoint_scratch_bytes(U.nx, U.ny, U.nz);
    const int rc = ensure_scratch(c, c->adj, need);
    if (rc) return rc;
    void* outp[5];
    for (int v = 0; v < 5; ++v) outp[v] = O.U[v];
    HostPatchIO lam = make_io(L, O);
    c->launches += 2;
    cudaError_t e = aops->adjoint(make_io(U, O), lam, outp, c->prm, dt_dev + i, c->adj.d, c->adj.cap, c->d_err,
                                  c->stream);
    if (e == cudaErrorNotSupported) return HYDRO_ERR_STATE;
    if (e != cudaSuccess) return HYDRO_ERR_CUDA;
  }
  return HYDRO_OK;
}

int hydro_prim_to_cons(hydro_ctx* c, const hydro_patch* W, const hydro_patch* U, int npatch) {
  if (!c || !W || !U || npatch < 1) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i) {
    if (!valid_patch(c, W[i]) || !valid_patch(c, U[i]) || !same_shape(W[i], U[i]) || overlaps(c, W[i], U[i]))
      return HYDRO_ERR_ARG;
  }
  for (int i = 0; i < npatch; ++i) {
    void* o[5];
    for (int v = 0; v < 5; ++v) o[v] = U[i].U[v];
    c->launches += 1;
    cudaError_t e = c->ops->p2c(make_io(W[i], U[i]), o, c->prm, c->stream);
    if (e != cudaSuccess) return HYDRO_ERR_CUDA;
  }
  return HYDRO_OK;
}

int hydro_prim_to_cons_adjoint(hydro_ctx* c, const hydro_patch* W, const hydro_patch* lamU, const hydro_patch* lamW,
                               int npatch) {
  if (!c || !W || !lamU || !lamW || npatch < 1) return HYDRO_ERR_ARG;
  for (int i = 0; i < npatch; ++i) {
    if (!valid_patch(c, W[i]) || !valid_patch(c, lamU[i]) || !valid_patch(c, lamW[i])) return HYDRO_ERR_ARG;
    if (!same_shape(W[i], lamU[i]) || !same_shape(W[i], lamW[i])) return HYDRO_ERR_ARG;
    if (overlaps(c, W[i], lamW[i]) || overlaps(c, lamU[i], lamW[i])) return HYDRO_ERR_ARG;
  }
  for (int i = 0; i < npatch; ++i) {
    void* o[5];
    for (int v = 0; v < 5; ++v) o[v] = lamW[i].U[v];
    c->launches += 1;
    cudaError_t e = c->ops->p2c_adjoint(make_io(W[i], lamW[i]), make_io(lamU[i], lamU[i]), o, c->prm, c->stream);
    if (e != cudaSuccess) return HYDRO_ERR_CUDA;
  }
  return HYDRO_OK;
}

// The same arrays, sizes, strides and cell size: everything of a box that a captured step holds.
static bool same_box(const hydro_patch& a, const hydro_patch& b) {
  for (int v = 0; v < 5; ++v)
    if (a.U[v] != b.U[v]) return false;
  return a.nx == b.nx && a.ny == b.ny && a.nz == b.nz && a.sy == b.sy && a.sz == b.sz && a.dx == b.dx;
}

int hydro_run(hydro_ctx* c, const hydro_patch* a, const hydro_patch* b, int nsteps, double* dt_hist_dev,
              int use_graph) {
  if (!c || !a || !b || nsteps < 1 || !dt_hist_dev) return HYDRO_ERR_ARG;
  if (!valid_patch(c, *a) || !valid_patch(c, *b) || a->ng != 0 || b->ng != 0) return HYDRO_ERR_ARG;
  if (!same_shape(*a, *b) || overlaps(c, *a, *b)) return HYDRO_ERR_ARG;
  auto enqueue = [&](cudaStream_t s) -> int {
    int rc = reset_slots(c, dt_hist_dev, 1, s);
    if (rc) return rc;
    cudaError_t e = c->ops->cfl(nullptr, make_io(*a, *a), 1, c->prm, dt_hist_dev, c->d_err, s);
    c->launches += 1;
    if (e != cudaSuccess) return HYDRO_ERR_CUDA;
    for (int n = 0; n < nsteps; ++n) {
      const hydro_patch& src = (n % 2 == 0) ? *a : *b;
      const hydro_patch& dst = (n % 2 == 0) ? *b : *a;
      rc = step_one_uniform(c, src, dst, dt_hist_dev + n, dt_hist_dev + n + 1, s);
      if (rc) return rc;
    }
    return HYDRO_OK;
  };
  if (!use_graph) return enqueue(c->stream);
  const bool hit = c->graph && same_box(c->g_a, *a) && same_box(c->g_b, *b) && c->g_n == nsteps && c->g_dt == dt_hist_dev &&
                   c->g_tile == c->tile_id && c->g_zc == c->zchunk && c->g_tuned == c->tuned;
  if (!hit) {
    if (c->graph) cudaGraphExecDestroy(c->graph);
    c->graph = nullptr;
    const long long before = c->launches;
    if (cudaStreamBeginCapture(c->capture, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return HYDRO_ERR_CUDA;
    int rc = enqueue(c->capture);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(c->capture, &g);
    c->launches = before;  // capture launches nothing
    if (rc) {
      if (g) cudaGraphDestroy(g);
      return rc;
    }
    if (e != cudaSuccess) return HYDRO_ERR_CUDA;
    e = cudaGraphInstantiate(&c->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
      c->graph = nullptr;
      return HYDRO_ERR_CUDA;
    }
    c->g_a = *a;
    c->g_b = *b;
    c->g_n = nsteps;
    c->g_dt = dt_hist_dev;
    c->g_tile = c->tile_id;
    c->g_zc = c->zchunk;
    c->g_tuned = c->tuned;
  }
  c->launches += nsteps + 1;
  return cuda_status(cudaGraphLaunch(c->graph, c->stream));
}

int hydro_get_tuning(hydro_ctx* c, int* tile_id, int* zchunk) {
  if (!c) return HYDRO_ERR_ARG;
  if (tile_id) *tile_id = c->tile_id;
  if (zchunk) *zchunk = c->zchunk;
  return HYDRO_OK;
}

int hydro_set_tuning(hydro_ctx* c, int tile_id, int zchunk) {
  if (!c || tile_id < 0 || tile_id >= hydro::kNumTiles || zchunk < 1 || zchunk > 4096) return HYDRO_ERR_ARG;
  c->tile_id = tile_id;
  c->zchunk = zchunk;
  c->tuned = true;
  for (int k = 0; k < HYDRO_NUM_PATCH_CLASSES; ++k) c->cls_tile[k] = -1;
  return HYDRO_OK;
}

int hydro_get_class_tuning(hydro_ctx* c, int patch_class_id, int* tile_id, int* zchunk) {
  if (!c || patch_class_id < 0 || patch_class_id >= HYDRO_NUM_PATCH_CLASSES) return HYDRO_ERR_ARG;
  if (tile_id) *tile_id = class_tile(c, patch_class_id);
  if (zchunk) *zchunk = class_zc(c, patch_class_id);
  return HYDRO_OK;
}

int hydro_set_class_tuning(hydro_ctx* c, int patch_class_id, int tile_id, int zchunk) {
  if (!c || patch_class_id < 0 || patch_class_id >= HYDRO_NUM_PATCH_CLASSES) return HYDRO_ERR_ARG;
  if (tile_id == -1) {
    c->cls_tile[patch_class_id] = -1;
    return HYDRO_OK;
  }
  if (tile_id < 0 || tile_id >= hydro::kNumTiles || zchunk < 1 || zchunk > 4096) return HYDRO_ERR_ARG;
  c->cls_tile[patch_class_id] = tile_id;
  c->cls_zc[patch_class_id] = zchunk;
  return HYDRO_OK;
}

int hydro_autotune(hydro_ctx* c, const hydro_patch* in, const hydro_patch* out, int npatch, const double* dt_dev,
                   const char* cache_path) {
  if (!c || !in || !out || npatch < 1 || !dt_dev) return HYDRO_ERR_ARG;
  // signature of the patch set: count, precision and total cells
  long long cells = 0;
  for (int i = 0; i < npatch; ++i) cells += (long long)in[i].nx * in[i].ny * in[i].nz;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, c->device) != cudaSuccess) return HYDRO_ERR_CUDA;
  char key[512];
  std::snprintf(key, sizeof(key), "%s|sm%d|p%d|l%d|n%d|c%lld|g%d", prop.name, c->sm_count, c->cfg.precision,
                c->cfg.limiter, npatch, cells, in[0].ng);
  for (char* k = key; *k; ++k)
    if (*k == ' ') *k = '_';
  constexpr int NC = HYDRO_NUM_PATCH_CLASSES;
  if (cache_path) {
    // one line per tuning: key, tile, z chunk, then tile and z chunk of each patch-shape class (-1: none)
    if (FILE* f = std::fopen(cache_path, "r")) {
      char k2[512];
      int t, z, ct[NC], cz[NC];
      while (std::fscanf(f, "%511s %d %d %d %d %d %d %d %d", k2, &t, &z, &ct[0], &cz[0], &ct[1], &cz[1], &ct[2],
                         &cz[2]) == 3 + 2 * NC) {
        bool ok = std::strcmp(k2, key) == 0 && t >= 0 && t < hydro::kNumTiles && z >= 1;
        for (int k = 0; k < NC; ++k) ok = ok && ct[k] >= -1 && ct[k] < hydro::kNumTiles && (ct[k] < 0 || cz[k] >= 1);
        if (ok) {
          c->tile_id = t;
          c->zchunk = z;
          c->tuned = true;
          for (int k = 0; k < NC; ++k) {
            c->cls_tile[k] = ct[k];
            c->cls_zc[k] = cz[k];
          }
          std::fclose(f);
          return HYDRO_OK;
        }
      }
      std::fclose(f);
    }
  }
  const bool was_tuned = c->tuned;
  c->tuned = true;
  for (int k = 0; k < NC; ++k) c->cls_tile[k] = -1;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // time of 3 steps (after a warm-up that also builds the work-list) of a patch set at the current tuning
  auto time3 = [&](const hydro_patch* a, const hydro_patch* b, int n, const double* dt, float* ms) -> int {
    int rc = hydro_step(c, a, b, n, dt, nullptr);
    if (rc) return rc;
    cudaEventRecord(e0, c->stream);
    for (int r = 0; r < 3; ++r) hydro_step(c, a, b, n, dt, nullptr);
    cudaEventRecord(e1, c->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return HYDRO_ERR_CUDA;
    cudaEventElapsedTime(ms, e0, e1);
    return HYDRO_OK;
  };
  // the fastest tile shape and z chunk for a patch set (uniform tuning)
  auto sweep = [&](const hydro_patch* a, const hydro_patch* b, int n, const double* dt, int* bt, int* bz,
                   float* best) -> int {
    long long cl = 0;
    int maxnz = 1;
    for (int i = 0; i < n; ++i) {
      cl += (long long)a[i].nx * a[i].ny * a[i].nz;
      maxnz = std::max(maxnz, a[i].nz);
    }
    // short z chunks only pay on small grids, where the longer ones leave SMs without a block
    const int zcs[] = {2, 4, 8, 16, 32, 64, 128};
    *best = 1e30f;
    for (int t = 0; t < (ppm(c) ? 1 : hydro::kNumTiles); ++t) {  // the PPM kernel has one tile shape
      for (int zc : zcs) {
        if (zc > std::max(8, maxnz)) continue;
        if (zc < 8 && cl > (1LL << 22)) continue;
        c->tile_id = t;
        c->zchunk = zc;
        float ms = 0;
        int rc = time3(a, b, n, dt, &ms);
        if (rc) return rc;
        if (ms < *best) {
          *best = ms;
          *bt = t;
          *bz = zc;
        }
      }
    }
    return HYDRO_OK;
  };
  int bt = c->tile_id, bz = c->zchunk;
  float best = 1e30f;
  int rc = sweep(in, out, npatch, dt_dev, &bt, &bz, &best);
  // a tile shape per patch-shape class, when the set holds patches of more than one class: each
  // class's best shape on its own patches, kept if the whole set then steps faster
  std::vector<int> cls((size_t)npatch);
  int present = 0, cnt[NC] = {};
  for (int i = 0; i < npatch; ++i) cnt[cls[i] = patch_class(in[i])]++;
  for (int k = 0; k < NC; ++k) present += cnt[k] > 0;
  int ct[NC] = {-1, -1, -1}, cz[NC] = {0, 0, 0};
  if (!rc && !ppm(c) && present > 1) {
    rc = ensure_device(&c->d_cls_dt, &c->cls_dt_cap, (size_t)npatch);
    for (int k = 0; k < NC && !rc; ++k) {
      if (!cnt[k]) continue;
      std::vector<hydro_patch> a, b;
      for (int i = 0; i < npatch; ++i)
        if (cls[i] == k) {
          a.push_back(in[i]);
          b.push_back(out[i]);
          // the class's time steps, gathered in order (one small device copy each)
          if (cudaMemcpyAsync(c->d_cls_dt + a.size() - 1, dt_dev + i, sizeof(double), cudaMemcpyDeviceToDevice,
                              c->stream) != cudaSuccess)
            rc = HYDRO_ERR_CUDA;
        }
      float bk = 0;
      if (!rc) rc = sweep(a.data(), b.data(), (int)a.size(), c->d_cls_dt, &ct[k], &cz[k], &bk);
    }
    if (!rc) {
      c->tile_id = bt;
      c->zchunk = bz;
      for (int k = 0; k < NC; ++k) {
        c->cls_tile[k] = cnt[k] ? ct[k] : -1;
        c->cls_zc[k] = cz[k];
      }
      float ms = 0;
      rc = time3(in, out, npatch, dt_dev, &ms);
      if (!rc && !(ms < 0.99f * best))
        for (int k = 0; k < NC; ++k) c->cls_tile[k] = -1;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) {
    for (int k = 0; k < NC; ++k) c->cls_tile[k] = -1;
    c->tuned = was_tuned;
    return rc;
  }
  c->tile_id = bt;
  c->zchunk = bz;
  if (cache_path) {
    if (FILE* f = std::fopen(cache_path, "a")) {
      std::fprintf(f, "%s %d %d", key, bt, bz);
      for (int k = 0; k < NC; ++k) std::fprintf(f, " %d %d", c->cls_tile[k], c->cls_tile[k] >= 0 ? c->cls_zc[k] : 0);
      std::fprintf(f, "\n");
      std::fclose(f);
    }
  }
  return HYDRO_OK;
}

int hydro_get_error(hydro_ctx* c, unsigned* error_bits) {
  if (!c) return HYDRO_ERR_ARG;
  unsigned bits = 0;
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (cudaMemcpy(&bits, c->d_err, sizeof(unsigned), cudaMemcpyDeviceToHost) != cudaSuccess) return HYDRO_ERR_CUDA;
  if (error_bits) *error_bits = bits;
  return bits ? HYDRO_ERR_UNPHYSICAL : HYDRO_OK;
}

int hydro_clear_error(hydro_ctx* c) {
  if (!c) return HYDRO_ERR_ARG;
  return cuda_status(cudaMemsetAsync(c->d_err, 0, sizeof(unsigned), c->stream));
}

int hydro_launch_count(hydro_ctx* c, long long* count) {
  if (!c || !count) return HYDRO_ERR_ARG;
  *count = c->launches;
  return HYDRO_OK;
}

}  // extern "C"
