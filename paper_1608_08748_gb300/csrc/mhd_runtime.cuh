// mhd_runtime.cuh -- internal runtime of libmhd.so shared by its translation units: the simulation
// object, the executor that steps a set of boxes with one launch per kernel class, and the
// templated launchers.  The FP64 instances are compiled in mhd.cu, the FP32-bulk instances in
// mhd_f32.cu.
#pragma once
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>  // header-only; ranges cost nothing unless a profiler is attached

#include <vector>

#include "mhd.h"
#include "mhd_kernels.cuh"

namespace mhd_rt {
using namespace mhd;

inline unsigned nblk(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// The index-check flags of the translation unit that includes this header (MHD_CHECK builds; 0
// otherwise), read and optionally cleared.  Each translation unit has its own device word.
static inline unsigned check_flags_of_this_unit(bool clear) {
#ifdef MHD_CHECK
  unsigned v = 0;
  if (cudaMemcpyFromSymbol(&v, ::mhd::g_check_flags, sizeof(v)) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (clear) {
    const unsigned z = 0;
    cudaMemcpyToSymbol(::mhd::g_check_flags, &z, sizeof(z));
  }
  return v;
#else
  (void)clear;
  return 0;
#endif
}

// An NVTX range around the enqueueing of one stage of the step, so that a profiler can attribute
// and filter the kernels by the paper's stages (ncu --nvtx --nvtx-include "Lagrangian stage/").
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// kernel classes with their own launch shape
enum KClass { KC_PRIM = 0, KC_EFACE, KC_EDGES, KC_EUPD, KC_LFACE, KC_LUPD, KC_POST, NKC };
// profile class of each kernel class (include/mhd.h, enum mhd_kernel_class)
inline int profile_class(int kc) {
  const int m[NKC] = {MHD_K_PRIM, MHD_K_EULER_FACE, MHD_K_EDGES, MHD_K_EULER_UPDATE,
                      MHD_K_LAG_FACE, MHD_K_LAG_UPDATE, MHD_K_POST};
  return m[kc];
}
// profiler tags: PROF_KC_BASE + kernel class for the tiled kernels, MHD_K_SMALL for the rest
constexpr int PROF_KC_BASE = 100;
inline int report_class(int tag) { return tag >= PROF_KC_BASE ? profile_class(tag - PROF_KC_BASE) : tag; }
// domain of the tiles of each kernel class
// The Lagrangian faces run in pencils (kb_lag_pencil) where the parabolas are FP64: sharing the
// differences, slopes and edge values of neighbouring cells saves FP64 instructions, the bound of
// that path; the FP32 path keeps one thread per face (kb_lag_face).
template <typename T>
constexpr bool lag_in_pencils() { return sizeof(T) == 8; }

template <typename T>
inline int class_domain(int kc) {
  const int lag = lag_in_pencils<T>() ? DOM_LAG_PENCILS : DOM_FACES;
  const int m[NKC] = {DOM_CELLS, DOM_PENCILS, DOM_LATTICE, DOM_CELLS, lag, DOM_CELLS, DOM_CELLS};
  return m[kc];
}

// launch shape: threads per block (= tile size) and grid = min(tiles, grid_mult x SMs), or one
// block per tile when grid_mult == 0
struct LaunchCfg {
  int block = 256;
  int grid_mult = 0;
};
constexpr int NTILE_SIZES = 4;  // 64, 128, 256, 512
inline int tile_slot(int block) { return block == 64 ? 0 : block == 128 ? 1 : block == 256 ? 2 : 3; }

struct TileTable {
  int* d = nullptr;  // [box..., start...] in one allocation
  int n = 0;
  int first[4] = {0, 0, 0, 0};  // face tables: the tiles of direction q are first[q] .. first[q + 1]
};

// CUDA event pairs around launches while profiling
struct Profiler {
  bool on = false;
  std::vector<cudaEvent_t> ev;
  std::vector<int> cls;
};

struct PScope {
  Profiler* P;
  cudaStream_t st;
  PScope(Profiler* p, cudaStream_t s, int cls) : P(p), st(s) {
    if (!P || !P->on) return;
    cudaEvent_t e;
    cudaEventCreate(&e);
    cudaEventRecord(e, st);
    P->ev.push_back(e);
    P->cls.push_back(cls);
  }
  ~PScope() {
    if (!P || !P->on) return;
    cudaEvent_t e;
    cudaEventCreate(&e);
    cudaEventRecord(e, st);
    P->ev.push_back(e);
  }
};

// A set of boxes advanced together: one launch per kernel class covers every box.
template <typename T>
struct Exec {
  std::vector<Box<T>> h;  // host copies of the descriptors
  Box<T>* d = nullptr;    // device table
  int nb = 0;
  TileTable tab[NDOM][NTILE_SIZES];
  LaunchCfg cfg[NKC];
  int nsm = 152;
  Profiler* prof = nullptr;
  bool ions = false;      // some box has H+ (reactions 5-8): the kernels with the ion code
  bool x_stage = false;   // the FP32 x sweep may stage its rows in shared memory (kb_euler_x_staged)
};

// elements of a box in a domain (the face domains: of direction dir)
template <typename T>
long long domain_size(const Box<T>& B, int dom, int dir) {
  const Geom& g = B.g;
  long long e[3] = {g.n[0], g.n[1], g.n[2]};
  switch (dom) {
    case DOM_CELLS: return g.N;
    case DOM_FACES: e[dir] += 1; break;
    case DOM_PENCILS: e[dir] = B.pe.seg[dir]; break;
    case DOM_LAG_PENCILS: e[dir] = B.pl.seg[dir]; break;
    default: return g.NF;
  }
  return e[0] * e[1] * e[2];
}

template <typename T>
cudaError_t ensure_table(Exec<T>& X, int dom, int block) {
  TileTable& t = X.tab[dom][tile_slot(block)];
  if (t.d) return cudaSuccess;
  const int ndir = dom == DOM_CELLS || dom == DOM_LATTICE ? 1 : 3;
  std::vector<int> bx, st;
  for (int q = 0; q < ndir; ++q) {
    t.first[q] = (int)bx.size();
    for (int b = 0; b < X.nb; ++b) {
      const long long n = domain_size(X.h[b], dom, q);
      for (long long s = 0; s < n; s += block) {
        bx.push_back(b | (q << TILE_DIR_SHIFT));
        st.push_back((int)s);
      }
    }
  }
  for (int q = ndir; q < 4; ++q) t.first[q] = (int)bx.size();  // one direction: the others are empty
  t.n = (int)bx.size();
  if (t.n == 0) return cudaSuccess;
  cudaError_t e = cudaMalloc(&t.d, sizeof(int) * 2 * (size_t)t.n);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(t.d, bx.data(), sizeof(int) * t.n, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  return cudaMemcpy(t.d + t.n, st.data(), sizeof(int) * t.n, cudaMemcpyHostToDevice);
}

template <typename T>
cudaError_t ensure_tables(Exec<T>& X) {
  for (int kc = 0; kc < NKC; ++kc) {
    cudaError_t e = ensure_table(X, class_domain<T>(kc), X.cfg[kc].block);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// the tiles of the directions q0 .. q1 - 1 of a face table
template <typename T>
Tiles tiles_of_dirs(const Exec<T>& X, int dom, int block, int q0, int q1) {
  const TileTable& t = X.tab[dom][tile_slot(block)];
  Tiles r;
  r.box = t.d + t.first[q0];
  r.start = t.d + t.n + t.first[q0];
  r.n = t.first[q1] - t.first[q0];
  return r;
}

inline unsigned grid_of(const Tiles& t, const LaunchCfg& c, int nsm) {
  long long g = t.n;
  if (c.grid_mult > 0 && (long long)c.grid_mult * nsm < g) g = (long long)c.grid_mult * nsm;
  return (unsigned)(g > 0 ? g : 1);
}

// default launch shapes: the FP64 face kernels keep their pencils' cells in shared memory (0.6 and 0.5 KB a
// thread) besides up to 213 registers, so blocks of 64 threads fill an SM closer than larger ones: 4 and 7 of
// them against 2 and 3 of 128 (128^3 step: Lagrangian faces 3.04 -> 2.80 ms, Eulerian 9.26 -> 9.20).  The
// FP32 faces 128; the rest 256, one block per tile.  The FP32 path's
// HBM-bound cell kernels run grid-stride over their tiles with a few blocks per SM where that is faster
// (256^3 step, measured over 64-512 threads and 2-16 blocks per SM: Lagrangian update 0.98 ms with 12 blocks
// of 128 per SM, 1.20 with 8; Eulerian update 1.46 with 8, 1.52 one block per tile; edges 0.49 / 0.51;
// post stage 0.93 / 0.95; primitives 0.53 ms one block per tile, 0.60 with 4 blocks of 512).  The instances over
// many boxes take more registers (64 against 40 in the Lagrangian update, so 8 blocks of 128 fill an SM, and 12
// would leave a half-empty round) and a search for the box of each tile, which a grid-stride block shares
// (32 boxes of 32^3 to 96^3: Lagrangian update 0.65 ms with 8 blocks, 0.86 with 12; primitives 0.296 with 8 blocks
// of 256, 0.326 one block per tile).
template <typename T>
void default_cfgs(Exec<T>& X) {
  for (int kc = 0; kc < NKC; ++kc) X.cfg[kc] = LaunchCfg{256, 0};
  X.cfg[KC_EFACE].block = sizeof(T) == 8 ? 64 : 128;
  X.cfg[KC_LFACE].block = sizeof(T) == 8 ? 64 : 128;
  if constexpr (sizeof(T) == 4) {
    X.cfg[KC_PRIM] = LaunchCfg{256, 0};
    X.cfg[KC_EDGES] = LaunchCfg{512, 4};
    X.cfg[KC_EUPD] = LaunchCfg{128, 8};
    X.cfg[KC_LUPD] = LaunchCfg{128, 12};
    X.cfg[KC_POST] = LaunchCfg{128, 8};
    if (X.nb > 1) {
      X.cfg[KC_PRIM] = LaunchCfg{256, 8};
      X.cfg[KC_LUPD] = LaunchCfg{128, 8};
    }
  }
}

// The FP32 x sweep stages the window primitives of its tiles' rows in dynamic shared memory
// (kb_euler_x_staged): 16 bytes of barrier and six primitives of at most (block - 1) / S + 2 rows
// of n_x cells (S pencils per row).  It needs every box's n_x to be a multiple of 4 and the largest
// box's rows to fit in kXStageMax; 0 otherwise, and the launch takes the direct kernel.
constexpr size_t kXStageMax = 200 * 1024;
template <typename T>
size_t euler_x_stage_bytes(const Exec<T>& X, int block) {
  size_t m = 0;
  for (int b = 0; b < X.nb; ++b) {
    const int nx = X.h[b].g.n[0];
    if (nx % 4 != 0) return 0;
    const size_t rows = (size_t)((block - 1) / X.h[b].pe.seg[0] + 2);
    const size_t need = 16 + rows * 6 * (size_t)nx * sizeof(T);
    m = need > m ? need : m;
  }
  return m <= kXStageMax ? m : 0;
}

// Kernel attributes of the current device: dynamic shared memory above the 48 KB default for the
// Eulerian pencils that stream their parabolas (up to 256 threads per block).  A kernel template
// instantiated in two translation units is two kernels, so this is instantiated where the launches
// of T are (the float launchers live in their own translation unit).
template <typename T>
cudaError_t prepare_kernels() {
  if constexpr (sizeof(T) == 4) {
    return cudaFuncSetAttribute(kb_euler_x_staged<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kXStageMax);
  } else {
    const int eb = (int)pencil_smem_bytes(EULER_SLOTS, 256), lb = (int)pencil_smem_bytes(LAG_SLOTS, 256);
    const void* euler[2] = {(const void*)kb_euler_pencil<T, OneBox<T>>, (const void*)kb_euler_pencil<T, ManyBoxes<T>>};
    const void* lag[4] = {(const void*)kb_lag_pencil<T, OneBox<T>, false>, (const void*)kb_lag_pencil<T, OneBox<T>, true>,
                          (const void*)kb_lag_pencil<T, ManyBoxes<T>, false>, (const void*)kb_lag_pencil<T, ManyBoxes<T>, true>};
    cudaError_t e = cudaSuccess;
    for (const void* k : euler)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, eb);
    for (const void* k : lag)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, lb);
    return e;
  }
}

// The pencils of a face kernel.  A pencil has a cost of its own (one more cell and the priming of its
// streams, as much as `own` faces), so long ones suit large grids; on a small grid they leave SMs idle
// while each thread walks its pencil alone, and in between the last round of blocks decides.  The model:
// of the blocks on the busiest SM every `resident` make a round, a round takes (len + own), and a part
// of a round with k blocks the share first + (1 - first) k / resident of it.  Fitted to FP64 steps of 16^3
// to 96^3, 128x4x4 and 128x128x4 cells with 1 to 8 faces, it comes within 0.8 % (Eulerian, at worst 5 %) and 0.0 %
// (Lagrangian) of the best length's time on average: 8 faces against the chosen 1 is 0.34 against 0.08 ms of
// Eulerian faces at 128x4x4, 1 against the chosen 6 is 0.47 / 0.41 ms at 40^3, 1 against the chosen 7
// 4.9 / 3.9 ms at 96^3.  The faces' results do not depend on it.
struct PencilModel {
  int resident;
  double own, first;
};
constexpr PencilModel kEulerPencils64 = {4, 0.2, 0.8}, kLagPencils64 = {7, 0.8, 0.4}, kEulerPencils32 = {4, 1.5, 0.4};
template <typename T>
Pencils pencils_of(const Box<T>& b, int len) {
  Pencils P;
  for (int q = 0; q < 3; ++q) {
    P.seg[q] = (b.g.n[q] + len) / len;            // of the n + 1 faces of a line
    P.len[q] = (b.g.n[q] + P.seg[q]) / P.seg[q];  // shared out evenly
  }
  return P;
}
template <typename T>
int pencil_length(const Exec<T>& X, int block, const PencilModel& m) {
  int best = 1;
  double least = 0.0;
  for (int len = 1; len <= pencil_len<T>(); ++len) {
    long long blocks = 0;
    int longest = 1;
    for (const Box<T>& b : X.h) {
      const Pencils P = pencils_of(b, len);
      for (int q = 0; q < 3; ++q) {
        blocks += (b.g.N / b.g.n[q] * P.seg[q] + block - 1) / block;
        longest = longest > P.len[q] ? longest : P.len[q];
      }
    }
    const long long per_sm = (blocks + X.nsm - 1) / X.nsm;
    const int rest = (int)(per_sm % m.resident);
    const double part = rest > 0 ? m.first + (1.0 - m.first) * rest / m.resident : 0.0;
    const double cost = ((double)(per_sm / m.resident) + part) * (longest + m.own);
    if (len == 1 || cost < least) {
      best = len;
      least = cost;
    }
  }
  return best;
}
template <typename T>
void choose_pencils(Exec<T>& X) {
  const int le = pencil_length(X, X.cfg[KC_EFACE].block, sizeof(T) == 8 ? kEulerPencils64 : kEulerPencils32);
  const int ll = sizeof(T) == 8 ? pencil_length(X, X.cfg[KC_LFACE].block, kLagPencils64) : 1;
  for (Box<T>& b : X.h) {
    b.pe = pencils_of(b, le);
    b.pl = pencils_of(b, ll);
  }
}

template <typename T>
cudaError_t exec_init(Exec<T>& X, const std::vector<Box<T>>& boxes) {
  X.h = boxes;
  X.nb = (int)boxes.size();
  X.ions = false;
  for (const Box<T>& b : boxes) X.ions = X.ions || (b.ph.chem && b.ph.ions);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&X.nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = prepare_kernels<T>();
  if (e != cudaSuccess) return e;
  default_cfgs(X);
  choose_pencils(X);
  e = cudaMalloc(&X.d, sizeof(Box<T>) * (size_t)X.nb);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(X.d, X.h.data(), sizeof(Box<T>) * (size_t)X.nb, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  return ensure_tables(X);
}

template <typename T>
void exec_free(Exec<T>& X) {
  for (int d = 0; d < NDOM; ++d)
    for (int q = 0; q < NTILE_SIZES; ++q) {
      if (X.tab[d][q].d) cudaFree(X.tab[d][q].d);
      X.tab[d][q].d = nullptr;
      X.tab[d][q].n = 0;
    }
  if (X.d) cudaFree(X.d);
  X.d = nullptr;
  X.nb = 0;
  X.h.clear();
}

// ------------------------------------------------------------------------------------------------
// a launch whose blocks may start while the kernel before it in the stream drains
// (dependent_launch_begin); in a captured step a programmatic edge.  The small grids' steps are chains of
// 20 short kernels: 128x4x4 FP64 230 -> 224, 32^3 FP32 104 -> 99 us per step.
template <typename... P, typename... A>
void launch_dep(cudaStream_t st, unsigned grid, unsigned block, size_t smem, void (*kernel)(P...), A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, (P)args...);
}
// a kernel's two instances, for one box and for many
#define MHD_BOTH(kernel, ...) kernel<T, OneBox<T>, ##__VA_ARGS__>, kernel<T, ManyBoxes<T>, ##__VA_ARGS__>
// launch of the tiles of a domain (directions q0 .. q1 - 1 of the face tables; bytes: dynamic shared memory)
template <typename T, typename K1, typename KN, typename... A>
void launch_dirs(Exec<T>& X, cudaStream_t st, int kc, int dom, int q0, int q1, size_t bytes, K1 one, KN many, A... args) {
  const LaunchCfg& c = X.cfg[kc];
  const TileTable& t = X.tab[dom][tile_slot(c.block)];
  const Tiles tl = tiles_of_dirs(X, dom, c.block, q0, q1);
  const unsigned grid = grid_of(tl, c, X.nsm);
  PScope p(X.prof, st, PROF_KC_BASE + kc);  // the profiler records the kernel class
  if (X.nb == 1 && q0 == 0) {
    OneBox<T> src{X.h[0], tl.n, t.first[1], t.first[2]};
    launch_dep(st, grid, c.block, bytes, one, src, args...);
  } else {
    ManyBoxes<T> src{X.d, tl};
    launch_dep(st, grid, c.block, bytes, many, src, args...);
  }
}
template <typename T, typename K1, typename KN, typename... A>
void launch_k(Exec<T>& X, cudaStream_t st, int kc, int dom, size_t bytes, K1 one, KN many, A... args) {
  launch_dirs(X, st, kc, dom, 0, 3, bytes, one, many, args...);
}
template <typename T>
void launch_small(Exec<T>& X, cudaStream_t st, int which, double cfl = 0, double t_end = 0,
                  int fixed = 0, double tau = 0) {
  PScope p_(X.prof, st, MHD_K_SMALL);
  unsigned g = nblk(X.nb, 128);
  if (which == 0) launch_dep(st, g, 128, 0, kb_begin_step<T>, X.d, X.nb);
  if (which == 1) launch_dep(st, g, 128, 0, kb_end_step<T>, X.d, X.nb);
  if (which == 2) kb_set_params<T><<<g, 128, 0, st>>>(X.d, X.nb, cfl, t_end, fixed, tau);
  if (which == 3) kb_zero_dmax<T><<<g, 128, 0, st>>>(X.d, X.nb);
}

template <typename T>
void launch_euler_stage(Exec<T>& X, cudaStream_t st) {
  NvtxRange range("Eulerian stage with Flux-CT (Sec. 2.4, 2.5)");
  // self-gravity: a box with a potential (such sims step alone, never in a batch)
  const bool grav = X.nb == 1 && X.h[0].phi != nullptr;
  for (int r = 0; r < 3; ++r) {
    if (X.ions)
      launch_k(X, st, KC_PRIM, DOM_CELLS, 0, MHD_BOTH(kb_prim, true));
    else
      launch_k(X, st, KC_PRIM, DOM_CELLS, 0, MHD_BOTH(kb_prim, false));
    if constexpr (sizeof(T) == 8) {
      launch_k(X, st, KC_EFACE, DOM_PENCILS, pencil_smem_bytes(EULER_SLOTS, X.cfg[KC_EFACE].block), MHD_BOTH(kb_euler_pencil));
    } else if (const size_t xs = X.x_stage ? euler_x_stage_bytes(X, X.cfg[KC_EFACE].block) : 0) {
      {
        const LaunchCfg& c = X.cfg[KC_EFACE];
        const Tiles tl = tiles_of_dirs(X, DOM_PENCILS, c.block, 0, 1);
        PScope p(X.prof, st, PROF_KC_BASE + KC_EFACE);
        launch_dep(st, grid_of(tl, c, X.nsm), c.block, xs, kb_euler_x_staged<T>, X.d, tl);
      }
      launch_dirs(X, st, KC_EFACE, DOM_PENCILS, 1, 3, 0, MHD_BOTH(kb_euler_pencil));
    } else {
      launch_k(X, st, KC_EFACE, DOM_PENCILS, 0, MHD_BOTH(kb_euler_pencil));
    }
    launch_k(X, st, KC_EDGES, DOM_LATTICE, 0, MHD_BOTH(kb_edges));
    if (grav)
      launch_k(X, st, KC_EUPD, DOM_CELLS, 0, MHD_BOTH(kb_euler_update, true), r);
    else
      launch_k(X, st, KC_EUPD, DOM_CELLS, 0, MHD_BOTH(kb_euler_update, false), r);
  }
}

// fuse_last: the last substage's update is left to the fused update and post stage of the step
// (launch_lag_post)
template <typename T>
void launch_lag_stage(Exec<T>& X, cudaStream_t st, bool fuse_last) {
  NvtxRange range("Lagrangian stage (Sec. 2.6)");
  for (int r = 0; r < 3; ++r) {
    if constexpr (lag_in_pencils<T>()) {
      const size_t lag_bytes = pencil_smem_bytes(LAG_SLOTS, X.cfg[KC_LFACE].block);
      if (X.ions) launch_k(X, st, KC_LFACE, DOM_LAG_PENCILS, lag_bytes, MHD_BOTH(kb_lag_pencil, true));
      else launch_k(X, st, KC_LFACE, DOM_LAG_PENCILS, lag_bytes, MHD_BOTH(kb_lag_pencil, false));
    } else {
      if (X.ions) launch_k(X, st, KC_LFACE, DOM_FACES, 0, MHD_BOTH(kb_lag_face, true));
      else launch_k(X, st, KC_LFACE, DOM_FACES, 0, MHD_BOTH(kb_lag_face, false));
    }
    if (r == 2 && fuse_last) break;
    if (X.ions)
      launch_k(X, st, KC_LUPD, DOM_CELLS, 0, MHD_BOTH(kb_lag_update, true), r);
    else
      launch_k(X, st, KC_LUPD, DOM_CELLS, 0, MHD_BOTH(kb_lag_update, false), r);
  }
}

// per-cell stages (bit 0 chemistry, bit 1 heating/cooling) / regularisation / check / CFL of the
// new state (cell_stages = do_reg = check = 0: only the CFL denominator)
template <typename T>
void launch_post(Exec<T>& X, cudaStream_t st, int cell_stages, int do_reg, int check) {
  NvtxRange range("chemistry, heating/cooling, regularisation, CFL (Sec. 2.7-2.9, 2.3)");
  if (X.ions)
    launch_k(X, st, KC_POST, DOM_CELLS, 0, MHD_BOTH(kb_post, true), cell_stages, do_reg, check);
  else
    launch_k(X, st, KC_POST, DOM_CELLS, 0, MHD_BOTH(kb_post, false), cell_stages, do_reg, check);
}

// the last Lagrangian update with the post stage (kb_lag_update_post; the post stage's launch
// shape)
template <typename T>
void launch_lag_post(Exec<T>& X, cudaStream_t st, int cell_stages, int do_reg, int check) {
  NvtxRange range("last Lagrangian update + chemistry, heating/cooling, regularisation, CFL");
  if (X.ions)
    launch_k(X, st, KC_POST, DOM_CELLS, 0, MHD_BOTH(kb_lag_update_post, true), cell_stages, do_reg, check);
  else
    launch_k(X, st, KC_POST, DOM_CELLS, 0, MHD_BOTH(kb_lag_update_post, false), cell_stages, do_reg, check);
}

template <typename T>
void launch_step(Exec<T>& X, cudaStream_t st) {
  NvtxRange range("mhd step");
  launch_small(X, st, 0);
  launch_euler_stage(X, st);
  launch_lag_stage(X, st, true);
  launch_lag_post(X, st, 3, 1, 1);
  launch_small(X, st, 1);
}

// the max CFL denominator of the current state of every box
template <typename T>
cudaError_t launch_cfl(Exec<T>& X, cudaStream_t st) {
  launch_small(X, st, 3);
  launch_post(X, st, 0, 0, 0);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_set_params(Exec<T>& X, cudaStream_t st, double cfl, double t_end, int fixed, double tau) {
  launch_small(X, st, 2, cfl, t_end, fixed, tau);
  return cudaGetLastError();
}

}  // namespace mhd_rt

// ------------------------------------------------------------------------------------------------
struct mhd_sim {
  using Geom = mhd::Geom;
  using Phys = mhd::Phys;
  using Scalars = mhd::Scalars;
  Geom g;
  Phys ph;
  int precision = 0;
  int use_graph = 1;
  int x_stage = 0;  // MHD_OPT_X_STAGE
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  char* pool = nullptr;
  size_t pool_bytes = 0;
  char* staging = nullptr;  // 10 * N * 8 bytes for host transfers / dtype conversion
  Scalars* sc = nullptr;
  Scalars* sc_host = nullptr;  // pinned mirror
  int* hflags_host = nullptr;  // host-mapped error flags of the last finished step
  int* hflags_dev = nullptr;   // its device address
  double* diag_part = nullptr;
  double* diag_out = nullptr;
  double* diag_host = nullptr;  // pinned, 9 doubles
  int diag_blocks = 0;
  mhd::Box<double> b64;  // descriptors of this box (one of the two is used)
  mhd::Box<float> b32;
  mhd_rt::Exec<double> x64;  // executor of this box alone
  mhd_rt::Exec<float> x32;
  mhd_rt::Profiler prof;
  cudaGraphExec_t gexec = nullptr;
  bool graph_valid = false;
  bool exec_valid = false;
  bool params_dirty = true;
  double last_cfl = -1.0, last_tend = -1.0;
  bool has_state = false;
  int batched = 0;  // number of batches that reference this sim
  void* grav = nullptr;  // self-gravity resources (mhd_gravity.cu), allocated on first use
};

namespace mhd_rt {

// ------------------------------------------------------------------------------------------------
// self-gravity (mhd_gravity.cu): allocate and point the box at the potential; enqueue the Poisson
// solve of the current density; copy the potential out; release
int grav_prepare(mhd_sim* S);
int grav_solve(mhd_sim* S);
int grav_copy(mhd_sim* S, double* out);
void grav_free(mhd_sim* S);

// per-sim (non-batched) helpers: state transfer and diagnostics.  They take the sim's geometry
// (S->g), not the box descriptor's copy: that copy is refreshed only when the executor is rebuilt,
// so after a boundary option changes it still holds the old boundaries until the next step.
template <typename T, typename In>
cudaError_t load_state(mhd_sim* S, Box<T>& B, const In* const* p) {
  const Geom& g = S->g;
  k_load_state<T, In><<<nblk(g.N, 256), 256, 0, S->stream>>>(g, S->ph, S->sc, B.s, p[0], p[1], p[2], p[3], p[4],
                                                             p[5], p[6], p[7], p[8]);
  return cudaGetLastError();
}

template <typename T, typename Out>
cudaError_t store_state(mhd_sim* S, Box<T>& B, Out* const* p) {
  const Geom& g = S->g;
  k_store_state<T, Out><<<nblk(g.N, 256), 256, 0, S->stream>>>(g, B.s, p[0], p[1], p[2], p[3], p[4], p[5],
                                                                p[6], p[7], p[8]);
  return cudaGetLastError();
}

template <typename T>
cudaError_t set_faces(mhd_sim* S, Box<T>& B, const double* const* b) {
  const Geom& g = S->g;
  k_faces_copy<T><<<nblk(g.N, 256), 256, 0, S->stream>>>(g, B.s, b[0], b[1], b[2]);
  k_derive_eint<T><<<nblk(g.N, 256), 256, 0, S->stream>>>(g, B.s);
  return cudaGetLastError();
}

template <typename T>
cudaError_t store_full(mhd_sim* S, Box<T>& B, double* const* d) {
  k_store_full<T><<<nblk(S->g.N, 256), 256, 0, S->stream>>>(S->g, B.s, d[0], d[1], d[2], d[3]);
  return cudaGetLastError();
}

template <typename T>
cudaError_t load_full(mhd_sim* S, Box<T>& B, const double* const* d) {
  k_load_full<T><<<nblk(S->g.N, 256), 256, 0, S->stream>>>(S->g, B.s, d[0], d[1], d[2], d[3]);
  return cudaGetLastError();
}

template <typename T>
cudaError_t store_ions(mhd_sim* S, Box<T>& B, double* d) {
  k_store_ions<T><<<nblk(S->g.N, 256), 256, 0, S->stream>>>(S->g, B.s, d);
  return cudaGetLastError();
}

template <typename T>
cudaError_t load_ions(mhd_sim* S, Box<T>& B, const double* d) {
  k_load_ions<T><<<nblk(S->g.N, 256), 256, 0, S->stream>>>(S->g, B.s, d);
  return cudaGetLastError();
}

template <typename T>
cudaError_t diag_partial(mhd_sim* S, Box<T>& B) {
  k_diag_partial<T><<<S->diag_blocks, DIAG_THREADS, 0, S->stream>>>(S->g, B.s, S->diag_part);
  return cudaGetLastError();
}

// The FP32 instances live in mhd_f32.cu.
#ifndef MHD_RT_F32_TU
extern template cudaError_t prepare_kernels<float>();
extern template void launch_euler_stage<float>(Exec<float>&, cudaStream_t);
extern template void launch_lag_stage<float>(Exec<float>&, cudaStream_t, bool);
extern template void launch_step<float>(Exec<float>&, cudaStream_t);
extern template void launch_post<float>(Exec<float>&, cudaStream_t, int, int, int);
extern template cudaError_t launch_cfl<float>(Exec<float>&, cudaStream_t);
extern template cudaError_t launch_set_params<float>(Exec<float>&, cudaStream_t, double, double, int, double);
extern template void launch_small<float>(Exec<float>&, cudaStream_t, int, double, double, int, double);
extern template cudaError_t load_state<float, double>(mhd_sim*, Box<float>&, const double* const*);
extern template cudaError_t load_state<float, float>(mhd_sim*, Box<float>&, const float* const*);
extern template cudaError_t store_state<float, double>(mhd_sim*, Box<float>&, double* const*);
extern template cudaError_t store_state<float, float>(mhd_sim*, Box<float>&, float* const*);
extern template cudaError_t set_faces<float>(mhd_sim*, Box<float>&, const double* const*);
extern template cudaError_t store_full<float>(mhd_sim*, Box<float>&, double* const*);
extern template cudaError_t load_full<float>(mhd_sim*, Box<float>&, const double* const*);
extern template cudaError_t diag_partial<float>(mhd_sim*, Box<float>&);
extern template cudaError_t store_ions<float>(mhd_sim*, Box<float>&, double*);
extern template cudaError_t load_ions<float>(mhd_sim*, Box<float>&, const double*);
#endif

}  // namespace mhd_rt
