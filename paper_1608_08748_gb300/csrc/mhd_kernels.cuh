// mhd_kernels.cuh -- CUDA kernels of one time step (arXiv:1608.08748, Sec. 2), templated on the
// bulk type T.  Every kernel maps threadIdx.x to the x index so that all loads along any axis are
// coalesced; boundary cells are reached through the periodic / zero-gradient index map.
#pragma once
#include "mhd_device.cuh"

namespace mhd {

// SSP-RK3 (Sec. 2.2): Q = a Q^n + b Q + g tau R for the substages r = 0, 1, 2
__host__ __device__ __forceinline__ double RK3_A(int r) { return r == 0 ? 0.0 : (r == 1 ? 0.75 : 1.0 / 3.0); }
__host__ __device__ __forceinline__ double RK3_B(int r) { return r == 0 ? 1.0 : (r == 1 ? 0.25 : 2.0 / 3.0); }
__host__ __device__ __forceinline__ double RK3_G(int r) { return r == 0 ? 1.0 : (r == 1 ? 0.25 : 2.0 / 3.0); }

// primitives W of every cell: v (3), cell-centred B (3), p, gamma, sqrt(rho)   [Sec. 2 closure,
// Sec. 2.5 centring of B, Sec. 4.3 gamma_eff]
template <typename T>
struct Prim {
  T* v[3];
  T* B[3];
  T* p;
  T* g;
  T* sr;
};

// A pointer into global memory, said to the compiler.  The pointers of a descriptor in memory (ManyBoxes) are
// generic to it otherwise: its loads through them could then be of shared memory and stay behind the
// stores to the pencils' slots (FP64 Eulerian faces of ten boxes of 32^3 to 72^3: 4.60 -> 4.32 ns per cell and
// step; the other kernels have no such stores, and gain nothing).
template <typename P>
__device__ __forceinline__ P* as_global(P* p) {
  __builtin_assume(__isGlobal(p));
  return p;
}

// Eulerian face outputs of one direction: F_mn, F_mt1, F_mt2, F_E, V_n, eA, eB   (Sec. 2.4, 2.5)
template <typename T>
struct FaceOut {
  T* f[8];  // the Lagrangian fluxes use f[0..nv-1]
};

// ------------------------------------------------------------------------------------------------
// faces of a pencil and pencils along each axis
struct Pencils {
  int len[3], seg[3];
};

// Batched execution.  Every step kernel walks a table of tiles; a tile is blockDim.x consecutive
// elements (cells, faces of one direction, or lattice points) of one box, so a warp never spans
// two boxes.  Grid-stride over tiles: a grid smaller than the tile count makes the launch
// persistent.  A single simulation is a table of one box.
template <typename T>
struct Box {
  Geom g;
  Phys ph;
  Scalars* sc;
  State<T> s, s0;
  Prim<T> w;
  FaceOut<T> fo[3];  // Eulerian face outputs; the Lagrangian fluxes reuse fo[d].f[0..nv-1]
  T* e[3];
  int nv;            // advected fields of the Lagrangian stage (6; 7 with rho_H2; 8 with rho_H+)
  Pencils pe, pl;    // the Eulerian and the FP64 Lagrangian pencils (set by the executor, choose_pencils)
  const T* phi;      // gravitational potential of the step (nullptr: no self-gravity)
  int* hflags;       // host-mapped copy of the error flags, written at the end of every step
};

struct Tiles {
  const int* box;    // box of tile t; its direction (of the face tables) in the bits from TILE_DIR_SHIFT on
  const int* start;  // first element of tile t inside its box (and direction)
  int n;             // number of tiles
};
constexpr int TILE_DIR_SHIFT = 28;

// Where a kernel takes its boxes from: a table of boxes and of their tiles, or one box.  A simulation on its
// own passes its box by value: the descriptor then lies in the kernel's parameter bank, so its 60-odd
// pointers cost neither loads nor registers, and a tile's place is arithmetic.  Against a table of one
// box: 256^3 FP32 step 13.0 -> 12.1 ms (Eulerian faces 4.43 -> 4.09, every other kernel but the primitives
// 3 to 12 % less), 128^3 FP64 16.7 -> 16.5, 32^3 FP32 99 -> 85 us, 128x4x4 FP64 224 -> 214 us.
template <typename T>
struct ManyBoxes {
  const Box<T>* boxes;
  Tiles tl;
  __device__ __forceinline__ int count() const { return tl.n; }
  // the box of tile t, its direction and the tile's first element
  __device__ __forceinline__ const Box<T>& tile(int t, int& dir, idx_t& start) const {
    const int code = tl.box[t];
    dir = code >> TILE_DIR_SHIFT;
    start = tl.start[t];
    return boxes[code & ((1 << TILE_DIR_SHIFT) - 1)];
  }
};
template <typename T>
struct OneBox {
  Box<T> box;
  int n, first1, first2;  // tiles, and the first ones of the directions 1 and 2
  __device__ __forceinline__ int count() const { return n; }
  __device__ __forceinline__ const Box<T>& tile(int t, int& dir, idx_t& start) const {
    dir = (t >= first1) + (t >= first2);
    start = (t - (dir == 0 ? 0 : dir == 1 ? first1 : first2)) * (int)blockDim.x;
    return box;
  }
};

// domains of the tile tables; those of faces and pencils hold the three directions one after another,
// so one launch covers the three sweeps of a stage
enum { DOM_CELLS = 0, DOM_FACES = 1, DOM_LATTICE = 2, DOM_PENCILS = 3, DOM_LAG_PENCILS = 4, NDOM = 5 };

// Faces are solved in pencils of consecutive faces along the sweep direction: the thread carries the
// stream of the left cell from one face to the next, so every cell's parabolas are built once per
// direction (plus one extra cell and the stream's priming per pencil).  pencil_len<T>() is the longest
// pencil: on the 256^3 FP32 step 6 faces measured fastest (4.41 ms of Eulerian faces; 4.83 with 4, 4.55
// with 8 and with 12), on the 128^3 FP64 one 8.  Smaller grids take shorter pencils, see choose_pencils.
template <typename T>
__host__ __device__ constexpr int pencil_len() { return sizeof(T) == 4 ? 6 : 8; }

// a lattice index with the grid's precomputed divisors (t >= 0)
__device__ __forceinline__ void decode_lattice(const Geom& g, idx_t t, int c[3]) {
  const unsigned r = fdiv((unsigned)t, g.dn1[0]);
  c[0] = (int)((unsigned)t - r * g.dn1[0].d);
  const unsigned q = fdiv(r, g.dn1[1]);
  c[1] = (int)(r - q * g.dn1[1].d);
  c[2] = (int)q;
}
// a cell index with the precomputed divisors of n_x and n_y
__device__ __forceinline__ void decode_cell(const Geom& g, idx_t t, int c[3]) {
  const unsigned r = fdiv((unsigned)t, g.dn[0]);
  c[0] = (int)((unsigned)t - r * g.dn[0].d);
  const unsigned q = fdiv(r, g.dn[1]);
  c[1] = (int)(r - q * g.dn[1].d);
  c[2] = (int)q;
}

// A pencil of direction D: its faces f0 .. f0 + nfp - 1 along the axis, and the cells and faces of its
// line (cell i at base + i stride, face i at fbase + i fstride).
struct Line {
  idx_t base, stride, fbase, fstride;
  int n, bc;
  int f0, nfp;
  __device__ __forceinline__ idx_t cell(const Geom& g, int i) const {
    return MHD_CELL(g, base + wrap(i, n, bc) * stride);
  }
  __device__ __forceinline__ idx_t face(const Geom& g, int i) const { return MHD_LATTICE(g, fbase + i * fstride); }
};
// Pencil p of direction D.  In the FP64 x sweep the y index runs fastest, so the threads of a warp
// share one segment and its face count (the last segment of a row is shorter; the FP64 pipe, not the
// memory system, bounds those kernels); the FP32 x sweep keeps the segment fastest for coalescing (the
// y-fastest order measured 12.9 against 8.1 ms per 256^3 step there), and the y and z sweeps run x
// fastest as the cells do.  D is a run-time value, the same for the whole block: one body serves the
// three sweeps (three instances in one kernel spilled 364 bytes of registers in FP32, against 72).
template <typename T>
__device__ __forceinline__ Line line_of_pencil(const Box<T>& B, const Pencils& P, int D, idx_t p) {
  const Geom& g = B.g;
  const int S = P.seg[D], nx = g.n[0], ny = g.n[1];
  int seg, i = 0, j = 0, k = 0;
  if (D == 0) {
    if (sizeof(T) == 8) {
      j = p % ny;
      p /= ny;
      seg = p % S;
      k = p / S;
    } else {
      seg = p % S;
      p /= S;
      j = p % ny;
      k = p / ny;
    }
  } else {
    i = p % nx;
    p /= nx;
    if (D == 1) {
      seg = p % S;
      k = p / S;
    } else {
      j = p % ny;
      seg = p / ny;
    }
  }
  Line L;
  L.n = g.n[D];
  L.bc = g.bc[D];
  L.base = (k * ny + j) * nx + i;
  L.stride = D == 0 ? 1 : D == 1 ? nx : nx * ny;
  L.fbase = (k * (ny + 1) + j) * (nx + 1) + i;
  L.fstride = D == 0 ? 1 : D == 1 ? nx + 1 : (nx + 1) * (ny + 1);
  L.f0 = seg * P.len[D];
  L.nfp = min(P.len[D], L.n + 1 - L.f0);
  return L;
}

// Programmatic dependent launch: the step's kernels are launched so that a kernel's blocks may take their
// places while the one before it drains (launch_dep).  Every such kernel first waits until the one before it has
// finished and its writes are visible; as it does so before it reads or writes anything, the order of the
// memory accesses is that of plain launches.  The next kernel may come when a block ends: let in at the start, its
// waiting blocks crowd the places of the few running ones (128x4x4 FP64 step 262 against 224 us).
__device__ __forceinline__ void dependent_launch_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

#define MHD_TILE_LOOP(src) for (int t_ = blockIdx.x; t_ < (src).count(); t_ += gridDim.x)

// Bulk asynchronous copies from global into shared memory (the copy engine moves the bytes; the
// issuing thread spends one instruction per copy) completed on an mbarrier.  Both addresses are
// 16-byte aligned and the size a multiple of 16 bytes; every wait on the barrier is bounded.
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned dynamic_smem_bytes() {
  unsigned r;
  asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// the one arrival of a phase, announcing the bytes its copies will deliver
__device__ __forceinline__ void mbar_arrive_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// waits for the phase of the given parity, for about a second at most; false if it gave up
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity) {
  const long long t0 = clock64();
  for (unsigned it = 0; it < (1u << 26); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > 2000000000ll) break;
  }
  return false;
}
// the error flag of a bulk copy that did not complete in time (bit 2 of Scalars::flags)
constexpr int FLAG_COPY_TIMEOUT = 4;

// ------------------------------------------------------------------------------------------------
// primitives of one cell (IONS: the kernel may see boxes with H+, whose gamma_eff counts it)
template <typename T, bool IONS>
__device__ __forceinline__ void prim_cell(const Box<T>& B, idx_t c) {
  const Geom& g = B.g;
  int q[3];
  decode_cell(g, c, q);
  const T rho = B.s.rho[c];
  idx_t up[3] = {cmap(g, q[0] + 1, q[1], q[2]), cmap(g, q[0], q[1] + 1, q[2]), cmap(g, q[0], q[1], q[2] + 1)};
  T Bc[3], m[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Bc[d] = mul_t(T(0.5), add_t(B.s.b[d][c], B.s.b[d][up[d]]));
    m[d] = B.s.m[d][c];
  }
  const T eint = B.s.eint[c];
  // gamma_eff in the bulk type: the FP32-bulk path's fluxes are FP32
  T gmt = !B.ph.chem ? (T)B.ph.gamma
          : (IONS && B.ph.ions) ? gamma_eff(rho, B.s.rh2[c], B.s.rhp[c]) : gamma_eff(rho, B.s.rh2[c]);
  const T irho = rcp_t(rho);  // one reciprocal for the three velocities
#pragma unroll
  for (int d = 0; d < 3; ++d) B.w.B[d][c] = Bc[d];
#pragma unroll
  for (int d = 0; d < 3; ++d) B.w.v[d][c] = mul_t(m[d], irho);
  B.w.p[c] = mul_t(sub_t(gmt, T(1)), eint);
  B.w.g[c] = gmt;
  B.w.sr[c] = sqrt_t(rho);
}

template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(512) kb_prim(const __grid_constant__ SRC src) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t c;
    const Box<T>& B = src.tile(t_, dir, c);
    c += (idx_t)threadIdx.x;
    if (c < B.g.N) prim_cell<T, IONS>(B, c);
  }
}

// ------------------------------------------------------------------------------------------------
// the step's tau / h, and g tau / h of substage r, in the bulk type
__device__ __forceinline__ double tau_h_of(const Box<double>& B) { return B.sc->tau_h; }
__device__ __forceinline__ float tau_h_of(const Box<float>& B) { return B.sc->tau_h32; }
__device__ __forceinline__ double rk_gth(const Box<double>& B, int r) { return B.sc->gth[r]; }
// (in FP32 the stored value made the updates slower, 1.51 against 1.46 and 1.05 against 0.98 ms per step)
__device__ __forceinline__ float rk_gth(const Box<float>& B, int r) { return (float)(RK3_G(r) * B.sc->tau * B.ph.ih); }

// Dynamic shared memory of the FP64 pencils: slots of this thread (slot k at [k blockDim.x +
// threadIdx.x], so a warp's accesses are consecutive), then a Step 4 ring per warp.
extern __shared__ __align__(16) unsigned char pencil_smem_raw[];
__device__ __forceinline__ double& pencil_slot(int k) {
  return reinterpret_cast<double*>(pencil_smem_raw)[k * blockDim.x + threadIdx.x];
}

// Step 4 of the FP64 parabolas, gathered over the warp.  Step 4 acts on one parabola in ten or less, but
// nearly every warp has a lane where it does, so as a branch its FP64 instructions would cost every
// parabola.  The lanes put what it needs in a ring of the warp in shared memory instead, and when 32 have
// come together (or the results are wanted) the warp does them at once, one per lane.  The deviations wait
// in slots of the owner's column; a result does not depend on how the ring groups it.  All 32 lanes call
// push and flush together.  (With the parabolas in FP64, 128^3 FP64 step at the developed flow: as a branch
// 20.0, gathered 17.2 ms.)
struct Step4Ring {
  static constexpr int N = 64;  // at most 31 left over and 32 new
  static constexpr size_t BYTES = N * (4 * sizeof(long long) + 2 * sizeof(int));
  long long* val;  // the four words of the items, N each
  int* who;        // the owner's slot of A (that of B lies `off` further), and E
  int off;
  int head = 0, count = 0;
  __device__ __forceinline__ Step4Ring(int slots, int slots_to_B) : off(slots_to_B * (int)blockDim.x) {
    unsigned char* base = pencil_smem_raw + (size_t)slots * blockDim.x * sizeof(double) + (threadIdx.x >> 5) * BYTES;
    val = reinterpret_cast<long long*>(base);
    who = reinterpret_cast<int*>(base + 4 * N * sizeof(long long));
  }
  __device__ __forceinline__ void process(int n) {
    __syncwarp();
    const int lane = threadIdx.x & 31;
    if (lane < n) {
      const int i = (head + lane) & (N - 1);
      double* ab = reinterpret_cast<double*>(pencil_smem_raw) + who[i];
      const Dev<double> P =
          fix_step4(Dev<double>{ab[0], ab[off]}, val[i], val[N + i], val[2 * N + i], val[3 * N + i], who[N + i]);
      ab[0] = P.A;
      ab[off] = P.B;
    }
    head = (head + n) & (N - 1);
    count -= n;
    __syncwarp();
  }
  // slot: the slot of A (B is at slot + slots_to_B)
  __device__ __forceinline__ void push(bool cand, int slot, const FixStep4& st) {
    const unsigned m = __ballot_sync(0xffffffffu, cand);
    if (cand) {
      const int i = (head + count + __popc(m & ((1u << (threadIdx.x & 31)) - 1))) & (N - 1);
      val[i] = st.num;
      val[N + i] = st.s0;
      val[2 * N + i] = st.h3;
      val[3 * N + i] = fix_min_abs(st);
      who[i] = slot * blockDim.x + threadIdx.x;
      who[N + i] = st.E;
    }
    count += __popc(m);
    if (count >= 32) process(32);
  }
  __device__ __forceinline__ void flush() {
    if (count > 0) process(count);
  }
};
// shared memory of a block with the given slots per thread and a ring per warp
constexpr size_t pencil_smem_bytes(int slots, int block) {
  return (size_t)slots * block * sizeof(double) + (size_t)(block / 32) * Step4Ring::BYTES;
}
// the deviations of the middle cell of c (live: this lane has one): Steps 1 and 2 at once, into the slots,
// Step 4 into the ring; returns q_0 - q_{-1}
__device__ __forceinline__ double ring_dev(const FixCell c[5], bool live, Step4Ring& ring, int slotA, int slotB) {
  Dev<double> P;
  double left;
  FixStep4 st;
  const bool cand = fix_dev(c, P, left, st);
  pencil_slot(slotA) = P.A;
  pencil_slot(slotB) = P.B;
  ring.push(live && cand, slotA, st);
  return left;
}

// The FP64 Eulerian pencils keep of each primitive v the last cells in rings of slots: the values of four
// (10 v .. 10 v + 3), the integers of five (10 v + 4 .. 10 v + 8) and their exponents, 11 bits each, in one
// word (10 v + 9); the new cell's deviations in the slots 60 + v (A) and 66 + v (B), its value less the cell's on
// its left in 72 + v (from the integers, which the integer pipes have time for: 128^3 step 13.9 -> 13.7 ms).
constexpr int EULER_SLOTS = 10 * 6 + 18;
__device__ __forceinline__ long long& pencil_word(int k) {
  return reinterpret_cast<long long*>(pencil_smem_raw)[k * blockDim.x + threadIdx.x];
}

// The element at an unsigned 32-bit byte offset: one add to a base that all threads share instead of an index
// widened and scaled for each access (FP32 256^3 step: Lagrangian faces 3.25 -> 3.14 ms).  4 GiB of one field
// are 2^29 cells (2^30 in FP32), whose fields together, 330 bytes a cell and more, no device holds.
template <typename T>
__device__ __forceinline__ T& at_byte(T* p, unsigned byte) {
  return *reinterpret_cast<T*>(reinterpret_cast<char*>(p) + byte);
}
template <typename T>
__device__ __forceinline__ const T& at_byte(const T* p, unsigned byte) {
  return *reinterpret_cast<const T*>(reinterpret_cast<const char*>(p) + byte);
}

// The fluxes of one Eulerian face f of direction D from its Riemann solution q* = (V_n, V_t1, V_t2,
// B_t1, B_t2, P) and the face field B_n (the non-advective parts of Sec. 2, reading A12), and the
// two EMF contributions E = B x U of Sec. 2.5.
template <typename T>
__device__ __forceinline__ void store_face_fluxes(const FaceOut<T>& fo, idx_t f, T Bn, const T qs[6]) {
  const T Vn = qs[0], Vt1 = qs[1], Vt2 = qs[2], Bt1 = qs[3], Bt2 = qs[4], P = qs[5];
  const T Bn2 = mul_t(Bn, Bn);
  const T Fn = fma(T(0.5), fma(Bt1, Bt1, fma(Bt2, Bt2, -Bn2)), P);  // p* - B_n^2
  const T F1 = -mul_t(Bn, Bt1), F2 = -mul_t(Bn, Bt2);
  as_global(fo.f[0])[f] = Fn;
  as_global(fo.f[1])[f] = F1;
  as_global(fo.f[2])[f] = F2;
  as_global(fo.f[3])[f] = fma(Fn, Vn, fma(F1, Vt1, mul_t(F2, Vt2)));  // p* V_n - B_n (B . V)
  as_global(fo.f[4])[f] = Vn;
  as_global(fo.f[5])[f] = fma(Bn, Vt1, -mul_t(Bt1, Vn));
  as_global(fo.f[6])[f] = fma(Bt2, Vn, -mul_t(Bn, Vt2));
}

// The FP32 Eulerian pencil: each of the six primitives streams along the pencil in registers (a
// DevStream of seven values; the loop over the faces stays rolled, since eight unrolled copies of the
// Riemann solve overflow the instruction cache), and the left cell's deviations, density, gamma and
// sqrt(rho) are carried from the previous face: ten loads per face instead of forty-three.  Where all
// cells f0 - 3 .. f1 + 1 of the pencil lie inside the grid they are addressed as base + i * stride
// without the boundary map.
//
// STG (the x sweep only): the six window primitives of the pencil's row are read from shared memory,
// srow[v * fs + x] for x in [0, n_x), where the block staged them (kb_euler_x_staged); the boundary map
// then only wraps or clamps x within the row.
template <typename T, bool STG = false>
__device__ __forceinline__ void euler_pencil_window(const Box<T>& B, int D, idx_t p, const T* srow = nullptr,
                                                    int fs = 0) {
  const int D1 = D == 2 ? 0 : D + 1, D2 = D == 0 ? 2 : D - 1;
  const Geom& g = B.g;
  const Line L = line_of_pencil(B, B.pe, D, p);
  const int f0 = L.f0, nfp = L.nfp;
  const T tau_k = mul_t(tau_h_of(B), avg_scale<T>());
  const bool inside = f0 >= 3 && f0 + nfp + 2 <= L.n;
  auto cell_at = [&](int i) -> idx_t {
    if (inside) return MHD_CELL(g, L.base + i * L.stride);
    return L.cell(g, i);
  };
  const T* qv[6] = {as_global(B.w.v[D]),  as_global(B.w.v[D1]), as_global(B.w.v[D2]),
                    as_global(B.w.B[D1]), as_global(B.w.B[D2]), as_global(B.w.p)};
  // the six window primitives of cell i along the pencil
  auto load6 = [&](int i, T out[6]) {
    if constexpr (STG) {
      const int x = inside ? i : wrap(i, L.n, L.bc);
#pragma unroll
      for (int v = 0; v < 6; ++v) out[v] = srow[v * fs + x];
    } else {
      const idx_t q = cell_at(i);
#pragma unroll
      for (int v = 0; v < 6; ++v) out[v] = qv[v][q];
    }
  };
  DevStream<T> S[6];
  FaceSide<T> l, r;  // the face's two cells; l carries the previous face's right cell
  {
    T col[5][6];
#pragma unroll
    for (int o = 0; o < 5; ++o) load6(f0 - 3 + o, col[o]);
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      S[v].prime(col[0][v], col[1][v], col[2][v], col[3][v]);
      l.P[v] = S[v].next(col[4][v]);  // cell f0 - 1
    }
  }
  {
    const idx_t q = cell_at(f0 - 1);
    l.w[0] = B.s.rho[q];
    l.w[2] = B.w.g[q];
    l.w[5] = B.w.sr[q];
  }
  // the loads of a face are issued one face ahead, so that their latency overlaps the previous
  // face's Riemann solve: the new stencil cell i + 2 and the right cell i (density, gamma,
  // sqrt(rho), face field)
  T nq[6], nr, ng, ns, nb;
  {
    const idx_t cr = cell_at(f0);
    load6(f0 + 2, nq);
    nr = B.s.rho[cr];
    ng = B.w.g[cr];
    ns = B.w.sr[cr];
    nb = B.s.b[D][cr];
  }
#pragma unroll 1
  for (int k = 0; k < nfp; ++k) {
    {
      const int i = f0 + k;
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        l.q[v] = S[v].qm;  // cell i - 1
        r.P[v] = S[v].next(nq[v]);  // cell i
        r.q[v] = S[v].qm;
      }
      r.w[0] = nr;
      r.w[2] = ng;
      r.w[5] = ns;
      const T Bn = nb;
      if (k + 1 < nfp) {
        const idx_t cr = cell_at(i + 1);
        load6(i + 3, nq);
        nr = B.s.rho[cr];
        ng = B.w.g[cr];
        ns = B.w.sr[cr];
        nb = B.s.b[D][cr];
      }
      l.w[1] = l.q[5];
      l.w[3] = l.q[3];
      l.w[4] = l.q[4];
      r.w[1] = r.q[5];
      r.w[3] = r.q[3];
      r.w[4] = r.q[4];
      T qs[6];
      riemann(l, r, Bn, tau_k, qs);
      store_face_fluxes(B.fo[D], L.face(g, i), Bn, qs);
      l = r;
    }
  }
}

// Eulerian faces of direction D (Sec. 2.4): the face i_D - 1/2 lies between cells i_D - 1 and i_D.
// One thread takes the faces i_D in [s P, min((s+1) P, n_D + 1)), P = pe.len[D], of one pencil s (the
// other two indices in [0, n)); each cell's parabolas are built once and serve both its faces.
// Per face: the PPM parabolas of (v_n, v_t1, v_t2, B_t1, B_t2, p) of the two cells, the Riemann
// solve, and the non-advective fluxes with the two EMF contributions E = B x U (Sec. 2.5).  This is
// the FP64 form; the FP32 form is euler_pencil_window.  The lanes of a warp go through the pencil
// together (Step4Ring); live: this lane has a pencil.
__device__ __forceinline__ void euler_pencil(const Box<double>& B, int D, idx_t p, bool live) {
  const int D1 = D == 2 ? 0 : D + 1, D2 = D == 0 ? 2 : D - 1;
  const Geom& g = B.g;
  const Line L = line_of_pencil(B, B.pe, D, p);
  const int f0 = L.f0, nfp = live ? L.nfp : 0;
  const double tau_k = mul_t(tau_h_of(B), avg_scale<double>());
  const double* qv[6] = {B.w.v[D], B.w.v[D1], B.w.v[D2], B.w.B[D1], B.w.B[D2], B.w.p};
  // the pointers of the loop by value: behind a reference each would be loaded again after the stores to the
  // slots, which might change it for all the compiler knows (128^3 step 13.6 -> 13.5 ms, ten boxes 4.66 -> 4.60
  // ns per cell)
  const double *rho = as_global(B.s.rho), *gam = as_global(B.w.g), *sr = as_global(B.w.sr),
               *bn = as_global(B.s.b[D]);
  const FaceOut<double> fo = B.fo[D];
  auto cell_at = [&](int i) { return L.cell(g, i); };
  Step4Ring ring(EULER_SLOTS, 6);
  // cell j of the pencil (j = 0 is cell f0 - 3): its value in ring place j % 4, its integer in j % 5
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    long long es = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double q = as_global(qv[v])[cell_at(f0 - 3 + j)];
      const FixCell c = fix_cell(q);
      pencil_slot(10 * v + j) = q;
      pencil_word(10 * v + 4 + j) = c.n;
      es |= (long long)c.e << (11 * (j + 1));
    }
    pencil_word(10 * v + 9) = es;
  }
  FaceSide<double> l, r;  // the face's two cells; l.P carries the previous face's right cell
#pragma unroll 1
  for (int k = -1; k < pencil_len<double>(); ++k) {  // cell f0 + k, then (from k = 0 on) the face on its left
    const int i = f0 + k;
    const bool on = k < nfp;
    if (!__any_sync(0xffffffffu, on)) break;
    const idx_t cn = cell_at(on ? i + 2 : f0);
    const int w4 = (k + 1) & 3;  // the new cell's place in the value rings: cell f0 + k + 2 is j = k + 5
    int w5[5];                   // the window's places in the integer rings: the cells j = k + 1 .. k + 5
    w5[0] = (k + 1) % 5;
#pragma unroll
    for (int o = 1; o < 5; ++o) w5[o] = w5[o - 1] == 4 ? 0 : w5[o - 1] + 1;
#pragma unroll 1
    for (int v = 0; v < 6; ++v) {
      const double q = as_global(qv[v])[cn];
      FixCell c[5];
      c[4] = fix_cell(q);
      const long long es = ((unsigned long long)pencil_word(10 * v + 9) >> 11) | ((long long)c[4].e << 44);
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        c[o].n = pencil_word(10 * v + 4 + w5[o]);
        c[o].e = (int)(es >> (11 * o)) & 0x7ff;
      }
      pencil_slot(10 * v + w4) = q;
      pencil_word(10 * v + 4 + w5[4]) = c[4].n;
      pencil_word(10 * v + 9) = es;
      pencil_slot(72 + v) = ring_dev(c, on, ring, 60 + v, 66 + v);
    }
    ring.flush();
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      l.q[v] = pencil_slot(10 * v + ((k + 2) & 3));  // cell i - 1: j = k + 2
      r.q[v] = pencil_slot(10 * v + ((k + 3) & 3));  // cell i
      r.P[v].A = pencil_slot(60 + v);
      r.P[v].B = pencil_slot(66 + v);
    }
    if (k >= 0 && on) {
      const idx_t cl = cell_at(i - 1), cr = cell_at(i);
      l.w[0] = rho[cl];
      l.w[1] = l.q[5];
      l.w[2] = gam[cl];
      l.w[3] = l.q[3];
      l.w[4] = l.q[4];
      l.w[5] = sr[cl];
      r.w[0] = rho[cr];
      r.w[1] = r.q[5];
      r.w[2] = gam[cr];
      r.w[3] = r.q[3];
      r.w[4] = r.q[4];
      r.w[5] = sr[cr];
      const double Bn = bn[cr];
      double d[6], qs[6];
#pragma unroll
      for (int v = 0; v < 6; ++v) d[v] = pencil_slot(72 + v);
      riemann(l, r, d, Bn, tau_k, qs);
      store_face_fluxes(fo, L.face(g, i), Bn, qs);
    }
#pragma unroll
    for (int v = 0; v < 6; ++v) l.P[v] = r.P[v];
  }
}

// The FP32 x sweep with the window primitives of its rows staged in shared memory.  A tile is
// blockDim.x consecutive x pencils (the segments of a row fastest), so its pencils lie in rows
// r_lo .. r_hi of the box (row r = k n_y + j, the cells r n_x .. r n_x + n_x - 1).  The six window
// primitives of those rows are brought into shared memory by bulk copies, one per row and
// primitive, issued by the lanes of the first warp; the threads then read their windows there
// instead of with global loads whose lanes lie 12 cells apart (12 cache lines per warp load).  Rows
// need n_x a multiple of 4 (16-byte rows) and the launch's dynamic shared memory to hold them
// (16 bytes of barrier, then [primitive][row][x]): the launcher takes this kernel only where every
// box qualifies, and a tile that does not (which the launcher rules out) is flagged, not solved.
// The results are those of kb_euler_pencil bit for bit.  It is opt-in (MHD_OPT_X_STAGE): on
// GB300 the x sweep measured slower with it (119 against 111 us per 128^3 launch), since the shared
// memory takes L1 capacity from the sweep's other strided accesses (L1 hit rate 38 -> 16 %), and
// staging all ten input fields as well (72 KB per block) kept the concurrent y and z sweeps' blocks
// off the SMs.
template <typename T>
__global__ void __launch_bounds__(256, 2) kb_euler_x_staged(const Box<T>* __restrict__ boxes, Tiles tl) {
  dependent_launch_begin();
  T* rows = reinterpret_cast<T*>(pencil_smem_raw + 16);
  const unsigned bar = smem_u32(pencil_smem_raw), rows_s = smem_u32(rows);
  const unsigned cap = dynamic_smem_bytes();
  if (threadIdx.x == 0 && cap >= 16) mbar_init(bar);
  __syncthreads();
  unsigned parity = 0;
  for (int t_ = blockIdx.x; t_ < tl.n; t_ += gridDim.x) {
    const Box<T>& B = boxes[tl.box[t_] & ((1 << TILE_DIR_SHIFT) - 1)];
    const int nx = B.g.n[0], S = B.pe.seg[0];
    const idx_t total = (idx_t)S * B.g.n[1] * B.g.n[2];
    const idx_t p0 = tl.start[t_], p = p0 + (idx_t)threadIdx.x;
    const idx_t pe = p0 + (idx_t)blockDim.x < total ? p0 + (idx_t)blockDim.x : total;
    const int r_lo = p0 / S, nrows = (int)((pe - 1) / S) - r_lo + 1;
    const unsigned bytes = (unsigned)nrows * 6u * (unsigned)nx * (unsigned)sizeof(T);
    if (nx % 4 != 0 || 16u + bytes > cap) {  // the same for every thread of the block
      if (threadIdx.x == 0) atomicOr(&B.sc->flags, FLAG_COPY_TIMEOUT);
      continue;
    }
    __syncthreads();  // every thread is done with the previous tile's rows
    if (threadIdx.x < 32) {
      if (threadIdx.x == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect(bar, bytes);
      }
      const T* src[6] = {B.w.v[0], B.w.v[1], B.w.v[2], B.w.B[1], B.w.B[2], B.w.p};
      for (int q = (int)threadIdx.x; q < 6 * nrows; q += 32) {
        const int v = q / nrows, lr = q - v * nrows;
        bulk_copy_g2s(rows_s + (unsigned)((v * nrows + lr) * nx) * (unsigned)sizeof(T),
                      src[v] + (size_t)(r_lo + lr) * nx, (unsigned)nx * (unsigned)sizeof(T), bar);
      }
    }
    const unsigned phase = parity;
    parity ^= 1u;
    const bool ok = mbar_wait_bounded(bar, phase);
    if (__syncthreads_or(!ok)) {
      // a copy did not arrive in time: flag it, give the copies in flight one more bounded wait,
      // and leave
      if (threadIdx.x == 0) atomicOr(&B.sc->flags, FLAG_COPY_TIMEOUT);
      mbar_wait_bounded(bar, phase);
      return;
    }
    if (p < total) euler_pencil_window<T, true>(B, 0, p, rows + (int)(p / S - r_lo) * nx, nrows * nx);
  }
}

// The three sweeps in one launch: they read the same cells and write separate arrays, so a sweep's
// last wave overlaps the next sweep's first, and the small grids pay one launch instead of three.
template <typename T>
__device__ __forceinline__ idx_t pencil_count(const Box<T>& B, const Pencils& P, int dir) {
  return (idx_t)(dir == 0 ? P.seg[0] : B.g.n[0]) * (dir == 1 ? P.seg[1] : B.g.n[1]) * (dir == 2 ? P.seg[2] : B.g.n[2]);
}

template <typename T, typename SRC>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1) kb_euler_pencil(const __grid_constant__ SRC src) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t p;
    const Box<T>& B = src.tile(t_, dir, p);
    p += (idx_t)threadIdx.x;
    const idx_t total = pencil_count(B, B.pe, dir);
    if constexpr (sizeof(T) == 8)
      euler_pencil(B, dir, p < total ? p : total - 1, p < total);
    else if (p < total)
      euler_pencil_window<T>(B, dir, p);
  }
}

// App. C: edge EMFs.  E_d at the corner (i_{d+1} - 1/2, i_{d+2} - 1/2) of lattice point c, for
// c_d in [0, n_d) and c_{d+1}, c_{d+2} in [0, n]: the mean of the two faces of direction d+1 and
// the two of direction d+2 that share the edge.
template <typename T>
__device__ __forceinline__ void edges_point(const Box<T>& B, idx_t t) {
  const Geom& g = B.g;
  int c[3];
  decode_lattice(g, t, c);
  T e[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
    e[d] = T(0);
    if (c[d] >= g.n[d]) continue;
    int a[3] = {c[0], c[1], c[2]};
    a[d2] = wrap(c[d2], g.n[d2], g.bc[d2]);
    int alo[3] = {c[0], c[1], c[2]};
    alo[d2] = wrap(c[d2] - 1, g.n[d2], g.bc[d2]);
    const T f1 = add_t(B.fo[d1].f[5][fidx(g, alo[0], alo[1], alo[2])], B.fo[d1].f[5][fidx(g, a[0], a[1], a[2])]);
    int b[3] = {c[0], c[1], c[2]};
    b[d1] = wrap(c[d1], g.n[d1], g.bc[d1]);
    int blo[3] = {c[0], c[1], c[2]};
    blo[d1] = wrap(c[d1] - 1, g.n[d1], g.bc[d1]);
    const T f2 = add_t(B.fo[d2].f[6][fidx(g, blo[0], blo[1], blo[2])], B.fo[d2].f[6][fidx(g, b[0], b[1], b[2])]);
    e[d] = mul_t(T(0.25), add_t(f1, f2));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (c[d] < g.n[d]) B.e[d][t] = e[d];
}

template <typename T, typename SRC>
__global__ void __launch_bounds__(512) kb_edges(const __grid_constant__ SRC src) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t t;
    const Box<T>& B = src.tile(t_, dir, t);
    t += (idx_t)threadIdx.x;
    if (t < B.g.NF) edges_point(B, t);
  }
}

// SSP-RK3 combination of Sec. 2.2 for one value: a Q^n + b Q + g tau R, with g tau R = gth S for a
// flux-difference sum S (R = S / h, gth = g tau / h once per thread).  The first substage has
// a = 0, b = g = 1 and returns Q + gth S; its caller stores Q^n (the stage's start value, the Q it
// read) in the RK register, which later substages read as q0.  (FP64 rounds a Q^n, FP32 b Q: against
// 64-bit arithmetic as written the other FP64 order is 20 % further off after one step.)
template <typename T>
__device__ __forceinline__ T rk_value(T q, T q0, T a, T b, T gth, T S, int r) {
  if constexpr (sizeof(T) == 8) return fma(gth, S, r == 0 ? q : fma(b, q, mul_t(a, q0)));
  else return fma(gth, S, r == 0 ? q : fma(a, q0, mul_t(b, q)));
}

// The cell kernels (primitives, edge EMFs, and the two updates in FP32) issue every load of a cell
// before its first store.  A thread stores only its own cell (or edge), which no load of the kernel
// reads, so the order is free; the compiler cannot prove that (all fields are plain pointers), and
// a store between two loads costs the thread one DRAM latency per stored field.  The FP64 updates
// keep the order field by field: holding all their loads would double their registers and halve
// the resident warps, and at the FP64 path's sizes that costs more than the latencies.
template <typename T>
__host__ __device__ constexpr bool update_loads_first() { return sizeof(T) == 4; }
// Eulerian update of one cell: finite-volume R of m, rho E, rho eps (Sec. 2.4 + A12), Flux-CT of
// the cell's three faces (Sec. 2.5), SSP-RK3 combination (Sec. 2.2) with stage r.
template <typename T, bool GRAV>
__device__ __forceinline__ void euler_update_cell(const Box<T>& B, idx_t c, int r) {
  const Geom& g = B.g;
  int q[3];
  decode_cell(g, c, q);
  const T a = (T)RK3_A(r), bb = (T)RK3_B(r), gth = rk_gth(B, r);
  idx_t f0 = fidx(g, q[0], q[1], q[2]);
  idx_t fup[3] = {fidx(g, q[0] + 1, q[1], q[2]), fidx(g, q[0], q[1] + 1, q[2]), fidx(g, q[0], q[1], q[2] + 1)};
  T acc[5];  // m_x, m_y, m_z, rho E, -h div V
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
    const FaceOut<T>& o = B.fo[d];
    auto sum = [&](T& a, int v) {
      const T df = sub_t(o.f[v][f0], o.f[v][fup[d]]);
      a = d == 0 ? df : add_t(a, df);
    };
    sum(acc[d], 0);
    sum(acc[d1], 1);
    sum(acc[d2], 2);
    sum(acc[3], 3);
    sum(acc[4], 4);
  }
  T Rv[5];  // h R: the flux-difference sums, and -(gamma - 1) rho eps h div V
#pragma unroll
  for (int v = 0; v < 4; ++v) Rv[v] = acc[v];
  Rv[4] = mul_t(mul_t(sub_t(B.w.g[c], T(1)), B.s.eint[c]), acc[4]);
  if (GRAV) {
    // self-gravity (Sec. 2): -rho grad Phi and -rho v . grad Phi, central differences of the
    // potential of the step (periodic box); a separate instance, so that the update without
    // gravity keeps its registers
    const idx_t dn[3] = {cmap(g, q[0] - 1, q[1], q[2]), cmap(g, q[0], q[1] - 1, q[2]), cmap(g, q[0], q[1], q[2] - 1)};
    const idx_t upc[3] = {cmap(g, q[0] + 1, q[1], q[2]), cmap(g, q[0], q[1] + 1, q[2]), cmap(g, q[0], q[1], q[2] + 1)};
    const T rho = B.s.rho[c];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T gd = mul_t(sub_t(B.phi[dn[d]], B.phi[upc[d]]), T(0.5));  // h (-d Phi / dx_d)
      Rv[d] = fma(rho, gd, Rv[d]);
      Rv[3] = fma(B.s.m[d][c], gd, Rv[3]);
    }
  }
  T* qq[5] = {B.s.m[0], B.s.m[1], B.s.m[2], B.s.E, B.s.eint};
  T* q0[5] = {B.s0.m[0], B.s0.m[1], B.s0.m[2], B.s0.E, B.s0.eint};
  // Flux-CT: d b_d / dt = -(curl E)_d on the face i_d - 1/2 of this cell
  auto curl_of = [&](int d) {
    const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
    return sub_t(sub_t(B.e[d1][fup[d2]], B.e[d1][f0]), sub_t(B.e[d2][fup[d1]], B.e[d2][f0]));
  };
  if constexpr (update_loads_first<T>()) {
    T qv[5], q0v[5], bv[3], b0v[3], curl[3];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      qv[v] = qq[v][c];
      q0v[v] = r ? q0[v][c] : T(0);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      bv[d] = B.s.b[d][c];
      b0v[d] = r ? B.s0.b[d][c] : T(0);
      curl[d] = curl_of(d);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if (r == 0) q0[v][c] = qv[v];
      qq[v][c] = rk_value(qv[v], q0v[v], a, bb, gth, Rv[v], r);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (r == 0) B.s0.b[d][c] = bv[d];
      B.s.b[d][c] = rk_value(bv[d], b0v[d], a, bb, gth, curl[d], r);
    }
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const T qv = qq[v][c], q0v = r ? q0[v][c] : T(0);
      if (r == 0) q0[v][c] = qv;
      qq[v][c] = rk_value(qv, q0v, a, bb, gth, Rv[v], r);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T curl = curl_of(d);
      const T bv = B.s.b[d][c], b0v = r ? B.s0.b[d][c] : T(0);
      if (r == 0) B.s0.b[d][c] = bv;
      B.s.b[d][c] = rk_value(bv, b0v, a, bb, gth, curl, r);
    }
  }
}

template <typename T, typename SRC, bool GRAV>
__global__ void __launch_bounds__(512) kb_euler_update(const __grid_constant__ SRC src, int r) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t c;
    const Box<T>& B = src.tile(t_, dir, c);
    c += (idx_t)threadIdx.x;
    if (c < B.g.N) euler_update_cell<T, GRAV>(B, c, r);
  }
}

// ------------------------------------------------------------------------------------------------
// Sec. 2.6 Lagrangian face flux for direction D: F = v_n q(-|v_n| tau) (v_n >= 0, left cell) or
// v_n q(|v_n| tau) (right cell) with v_n the sqrt(rho)-weighted mean of the cell velocities.
template <typename T, bool IONS>
__device__ __forceinline__ void lag_face(const Box<T>& B, int D, idx_t t) {
  const Geom& g = B.g;
  // face t of direction D: x runs over n_x (+ 1 in the x sweep) values, y over n_y (+ 1 in the y sweep)
  const FastDiv d0 = D == 0 ? g.dn1[0] : g.dn[0], d1 = D == 1 ? g.dn1[1] : g.dn[1];
  const unsigned r0 = fdiv((unsigned)t, d0);
  const int i = (int)((unsigned)t - r0 * d0.d), k = (int)fdiv(r0, d1), j = (int)(r0 - (unsigned)k * d1.d);
  const T tau_k = mul_t(tau_h_of(B), avg_scale<T>());
  const int nx = g.n[0], ny = g.n[1], n = g.n[D];
  const int a = D == 0 ? i : D == 1 ? j : k;
  const idx_t stride = D == 0 ? 1 : (D == 1 ? nx : nx * ny);
  const idx_t cc = (k * ny + j) * nx + i;
  idx_t cell[6];
  if (a >= 3 && a + 2 < n) {
    // the whole stencil inside the grid: a stride from this face's right cell, no boundary map
#pragma unroll
    for (int o = 0; o < 6; ++o) cell[o] = MHD_CELL(g, cc + (o - 3) * stride);
  } else {
    const idx_t line = cc - a * stride;
#pragma unroll
    for (int o = 0; o < 6; ++o) cell[o] = MHD_CELL(g, line + wrap(a + o - 3, n, g.bc[D]) * stride);
  }
  idx_t cl = cell[2], cr = cell[3];
  // v_l sqrt(rho_l) = m_l / sqrt(rho_l) and sqrt(rho) = rho / sqrt(rho): two 1/sqrt and a division
  T rl = B.s.rho[cl], rr = B.s.rho[cr];
  T isl = rsqrt_t(rl), isr = rsqrt_t(rr);
  const T vn = mul_t(fma(B.s.m[D][cr], isr, mul_t(B.s.m[D][cl], isl)), rcp_t(fma(rr, isr, mul_t(rl, isl))));
  const AvgCoef<T> kc = avg_coef(mul_t(abs_b(vn), tau_k));
  const T* q[7] = {B.s.rho, B.s.m[0], B.s.m[1], B.s.m[2], B.s.E, B.s.eint, B.s.rh2};
  const idx_t f = fidx(g, i, j, k);
  const int o0 = vn >= T(0) ? 0 : 1;  // upwind cell: stencil cells o0 .. o0 + 4
  // the upwind average as q + kA A + kB B on either side
  const T kA = o0 == 0 ? kc.p : -kc.r, kB = o0 == 0 ? kc.r : -kc.p;
  const int nv = B.nv;
  unsigned st[5];
#pragma unroll
  for (int o = 0; o < 5; ++o) st[o] = (unsigned)(o0 == 0 ? cell[o] : cell[o + 1]) * (unsigned)sizeof(T);
  const unsigned fb = (unsigned)f * (unsigned)sizeof(T);
  auto flux = [&](const T* u, int v) {
    const T qc = at_byte(u, st[2]);
    const Dev<T> P = dev_of(at_byte(u, st[0]), at_byte(u, st[1]), qc, at_byte(u, st[3]), at_byte(u, st[4]));
    at_byte(B.fo[D].f[v], fb) = vn * fma(kB, P.B, fma(kA, P.A, qc));
  };
#pragma unroll
  for (int v = 0; v < 7; ++v) {
    if (v >= nv) break;
    flux(q[v], v);
  }
  if (IONS) {
#pragma unroll 1
    for (int v = 7; v < nv; ++v) flux(B.s.rhp, v);  // rho_H+ (ions on)
  }
}

// At most 32 registers, a full SM: the instance over many boxes would take 40 (32 boxes of 32^3 to 96^3: 1.85 ->
// 1.73 ms per step, in spite of 56 bytes of spills; that of one box takes 32 by itself).
template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(256, 8) kb_lag_face(const __grid_constant__ SRC src) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t t;
    const Box<T>& B = src.tile(t_, dir, t);
    t += (idx_t)threadIdx.x;
    if (t < (idx_t)(B.g.n[0] + (dir == 0)) * (B.g.n[1] + (dir == 1)) * (B.g.n[2] + (dir == 2)))
      lag_face<T, IONS>(B, dir, t);
  }
}

// The same fluxes in FP64 for the faces i_D - 1/2, i_D in [s P, min((s+1) P, n_D + 1)), P = pl.len[D],
// of one pencil s: the face velocities first, then field by field the deviations of the pencil's cells from a
// window of five integers that slides along D, Step 4 gathered over the warp (Step4Ring), then each face's
// average of its upwind cell.  Slots: v_n and the two average coefficients of each face, then A, B and the value of each cell.
constexpr int LAG_FACES = pencil_len<double>(), LAG_CELLS = LAG_FACES + 1;
constexpr int LAG_SLOTS = 3 * LAG_FACES + 3 * LAG_CELLS;
template <bool IONS>
__device__ __forceinline__ void lag_pencil(const Box<double>& B, int D, idx_t p, bool live) {
  const Geom& g = B.g;
  const Line L = line_of_pencil(B, B.pl, D, p);
  const int f0 = L.f0, nfp = live ? L.nfp : 0;
  const double tau_k = mul_t(tau_h_of(B), avg_scale<double>());
  auto cell_at = [&](int i) { return L.cell(g, i); };
  constexpr int VN = 0, KP = LAG_FACES, KR = 2 * LAG_FACES, CA = 3 * LAG_FACES, CB = CA + LAG_CELLS, CQ = CB + LAG_CELLS;
  Step4Ring ring(LAG_SLOTS, LAG_CELLS);
  // per face: v_n and the coefficients of the average over the upwind fraction y = |v_n| tau / h,
  // q + p A + r B of the left cell (v_n >= 0) or q - r A - p B of the right cell: with (X, Z) = (A, B)
  // or (-B, -A) both are q + p X + r Z.  v_n = (v_l sqrt(rho_l) + v_r sqrt(rho_r)) / (sqrt(rho_l) +
  // sqrt(rho_r)) from the per-cell m / sqrt(rho) and rho / sqrt(rho) = sqrt(rho), each formed once and
  // carried to the next face
  double al, bl;
  {
    const idx_t c0 = cell_at(f0 - 1);
    const double r0 = B.s.rho[c0], is0 = rsqrt_n(r0);
    al = mul_t(B.s.m[D][c0], is0);
    bl = mul_t(r0, is0);
  }
#pragma unroll 2
  for (int k = 0; k < nfp; ++k) {
    const idx_t cr = cell_at(f0 + k);
    const double rr = B.s.rho[cr], isr = rsqrt_n(rr);
    const double ar = mul_t(B.s.m[D][cr], isr), br = mul_t(rr, isr);
    const double vn = mul_t(add_t(al, ar), rcp_t(add_t(bl, br)));
    al = ar;
    bl = br;
    const AvgCoef<double> kc = avg_coef(mul_t(abs_b(vn), tau_k));
    pencil_slot(VN + k) = vn;
    pencil_slot(KP + k) = kc.p;
    pencil_slot(KR + k) = kc.r;
  }
  __syncwarp();
  const int nv = B.nv;
#pragma unroll 1
  for (int v = 0; v < nv; ++v) {
    const double* a = v == 0 ? B.s.rho : v < 4 ? B.s.m[v - 1] : v == 4 ? B.s.E : v == 5 ? B.s.eint
                      : (IONS && v == 7) ? B.s.rhp : B.s.rh2;
    a = as_global(a);
    FixCell w[5];
    double qa = a[cell_at(f0 - 1)], qb = a[cell_at(f0)];  // the values of the next two cells
    w[1] = fix_cell(a[cell_at(f0 - 3)]);
    w[2] = fix_cell(a[cell_at(f0 - 2)]);
    w[3] = fix_cell(qa);
    w[4] = fix_cell(qb);
    double q1 = a[cell_at(f0 + 1)];  // one cell ahead, so that its latency overlaps the cell before
#pragma unroll 1
    for (int c = 0; c < LAG_CELLS; ++c) {  // cell f0 - 1 + c
      const bool on = c <= nfp && live;
      if (!__any_sync(0xffffffffu, on)) break;
      const double qn = q1;
      q1 = a[cell_at(c < nfp ? f0 + 2 + c : f0)];
      pencil_slot(CQ + c) = qa;
      qa = qb;
      qb = qn;
#pragma unroll
      for (int o = 0; o < 4; ++o) w[o] = w[o + 1];
      w[4] = fix_cell(qn);
      ring_dev(w, on, ring, CA + c, CB + c);
    }
    ring.flush();
    double* out = as_global(B.fo[D].f[v]);
#pragma unroll 2
    for (int k = 0; k < nfp; ++k) {
      const double vn = pencil_slot(VN + k);
      const bool left = !sign_bit_b(vn);  // v_n = -0: a zero flux either way
      const int c = left ? k : k + 1;
      const double A = pencil_slot(CA + c), Bv = pencil_slot(CB + c);
      const double X = left ? A : neg_b(Bv), Z = left ? Bv : neg_b(A);
      out[L.face(g, f0 + k)] = mul_t(vn, fma(pencil_slot(KR + k), Z, fma(pencil_slot(KP + k), X, pencil_slot(CQ + c))));
    }
    __syncwarp();
  }
}

template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(256, 1) kb_lag_pencil(const __grid_constant__ SRC src) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t p;
    const Box<double>& B = src.tile(t_, dir, p);
    p += (idx_t)threadIdx.x;
    const idx_t total = pencil_count(B, B.pl, dir);
    lag_pencil<IONS>(B, dir, p < total ? p : total - 1, p < total);
  }
}

// IONS: up to 8 advected fields (rho_H+ last), else up to 7
template <typename T, bool IONS>
__device__ __forceinline__ void lag_update_cell(const Box<T>& B, idx_t c, int r) {
  const Geom& g = B.g;
  int q[3];
  decode_cell(g, c, q);
  const T a = (T)RK3_A(r), bb = (T)RK3_B(r), gth = rk_gth(B, r);
  idx_t f0 = fidx(g, q[0], q[1], q[2]);
  idx_t fup[3] = {fidx(g, q[0] + 1, q[1], q[2]), fidx(g, q[0], q[1] + 1, q[2]), fidx(g, q[0], q[1], q[2] + 1)};
  T* qq[8] = {B.s.rho, B.s.m[0], B.s.m[1], B.s.m[2], B.s.E, B.s.eint, B.s.rh2, B.s.rhp};
  T* q0[8] = {B.s0.rho, B.s0.m[0], B.s0.m[1], B.s0.m[2], B.s0.E, B.s0.eint, B.s0.rh2, B.s0.rhp};
  const int nv = B.nv;
  constexpr int NV = IONS ? 8 : 7;
  auto sum_of = [&](int v) {
    T acc = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T df = sub_t(B.fo[d].f[v][f0], B.fo[d].f[v][fup[d]]);
      acc = d == 0 ? df : add_t(acc, df);
    }
    return acc;
  };
  if constexpr (update_loads_first<T>()) {
    // the fields in two halves, each with its loads before its stores: all seven at once kept 21
    // values and the flux sums live at the 64 registers the compiler chose, and measured slower
    // (1.34 against 1.25 ms per 256^3 step)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      constexpr int H = (NV + 1) / 2;
      T acc[H], qv[H], q0v[H];
#pragma unroll
      for (int i = 0; i < H; ++i) {
        const int v = h * H + i;
        acc[i] = qv[i] = q0v[i] = T(0);
        if (v < NV && v < nv) {
          acc[i] = sum_of(v);
          qv[i] = qq[v][c];
          if (r) q0v[i] = q0[v][c];
        }
      }
#pragma unroll
      for (int i = 0; i < H; ++i) {
        const int v = h * H + i;
        if (v < NV && v < nv) {
          if (r == 0) q0[v][c] = qv[i];
          qq[v][c] = rk_value(qv[i], q0v[i], a, bb, gth, acc[i], r);
        }
      }
    }
  } else {

#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (v >= nv) break;
      const T acc = sum_of(v);
      const T qv = qq[v][c], q0v = r ? q0[v][c] : T(0);
      if (r == 0) q0[v][c] = qv;
      qq[v][c] = rk_value(qv, q0v, a, bb, gth, acc, r);
    }
  }
}

template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(512) kb_lag_update(const __grid_constant__ SRC src, int r) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t c;
    const Box<T>& B = src.tile(t_, dir, c);
    c += (idx_t)threadIdx.x;
    if (c < B.g.N) lag_update_cell<T, IONS>(B, c, r);
  }
}

// ------------------------------------------------------------------------------------------------
// warp-aggregated helpers
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The CFL denominator of the new state of one cell for the next tau (Sec. 2.3).  All lanes of the warp
// call it (candidate marks those with a physical cell): the FP64 denominator is evaluated only where the
// FP32 screen (cfl_estimate_f32) cannot exclude the cell from the box's maximum; D stays 0 elsewhere.
//
// The screen: a finite estimate raised by 2^-12 below a lower bound of the maximum excludes the cell: any
// finite estimate lowered by 2^-12 (whose cell is evaluated unless it is excluded too), or the FP64
// maximum reached so far.  The warp's largest goes into the box's dlow before the test, and what the
// other warps have put there by then comes back, so that the first wave's warps need not each
// evaluate their own largest cell.
template <typename T>
__device__ __forceinline__ void cfl_of_cell(const Phys& ph, Scalars* sc, bool candidate, bool ions, T rho, const T m[3],
                                            const T Bc[3], T eint, T rh2, T rhp, double& D) {
  float D32 = 0.0f;  // 0: no candidate
  if (candidate)
    D32 = cfl_estimate_f32((float)rho, (float)m[0], (float)m[1], (float)m[2], (float)Bc[0], (float)Bc[1],
                           (float)Bc[2], (float)eint,
                           gamma_minus_one_f32(ph.chem, ph.gamma, (float)rho, (float)rh2, (float)rhp));
  float bound = warp_max_f(D32 <= 3.0e38f ? D32 : 0.0f) * (1.0f - 0x1p-12f);
  if ((threadIdx.x & 31) == 0) {
    const int mine = __float_as_int(bound);
    int low = *(volatile int*)&sc->dlow;
    if (mine > low) low = max(mine, atomicMax(&sc->dlow, mine));
    bound = __int_as_float(low);
  }
  bound = __shfl_sync(0xffffffffu, bound, 0);
  bound = fmaxf(bound, __double2float_rd(__longlong_as_double(*(volatile long long*)&sc->dmax)));
  if (candidate && !(D32 * (1.0f + 0x1p-12f) < bound)) {
    // FP64 CFL of the new state (FP32 fields widened)
    double gm = ph.chem ? gamma_eff((double)rho, (double)rh2) : ph.gamma;
    if (ions) gm = gamma_eff((double)rho, (double)rh2, (double)rhp);
    D = cfl_denominator((double)rho, (double)m[0], (double)m[1], (double)m[2], (double)Bc[0],
                        (double)Bc[1], (double)Bc[2], gm * ((gm - 1.0) * (double)eint));
  }
}
// the warp's share of the largest FP64 CFL denominator
__device__ __forceinline__ void cfl_warp_reduce(Scalars* sc, double D) {
  if (__any_sync(0xffffffffu, D > 0.0)) {
    D = warp_max(D);
    if ((threadIdx.x & 31) == 0) atomicMax(&sc->dmax, (unsigned long long)__double_as_longlong(D));
  }
}

// Per cell, after the Lagrangian stage: chemistry (Sec. 2.7, FP64), heating/cooling (Sec. 2.8,
// FP64, when on), regularisation (Sec. 2.9), the non-physical check, and the CFL denominator of the
// new state for the next tau (Sec. 2.3).  cell_stages selects the per-cell stages (bit 0
// chemistry, bit 1 heating/cooling; the full step runs both), do_reg the regularisation;
// cell_stages = do_reg = 0 computes only the CFL denominator.  All lanes of the warp call it (valid
// marks those with a cell).  Returns the flags via the warp-aggregated atomics of the caller.
template <typename T, bool IONS>
__device__ __forceinline__ void post_cell(const Box<T>& B, idx_t c, bool valid, int cell_stages,
                                          int do_reg, double& D, int& bad, unsigned& vb) {
  const Geom& g = B.g;
  const Phys& ph = B.ph;
  const bool ions = IONS && ph.ions;
  const State<T>& s = B.s;
  T rho = T(0), m[3] = {T(0), T(0), T(0)}, Bc[3] = {T(0), T(0), T(0)}, eint = T(0), rh2 = T(0), rhp = T(0);
  if (valid) {
    int q[3];
    decode_cell(g, c, q);
    const double tau = B.sc->tau;
    bool fp64_chem = (cell_stages & 1) && ph.chem;
    if constexpr (sizeof(T) == 4) {
      if (fp64_chem && !ions) {
        float r;
        if (chem_cell_pairs(ph, B.sc->ts, s.rho[c], s.eint[c], s.rh2[c], r)) {
          s.rh2[c] = r;
          fp64_chem = false;
        }
      }
    }
    if (fp64_chem) {
      const ChemOut co = chem_cell<IONS>(ph, (double)s.rho[c], (double)s.eint[c], (double)s.rh2[c],
                                         ions ? (double)s.rhp[c] : 0.0, tau);
      s.rh2[c] = (T)co.rh2;
      if (ions) s.rhp[c] = (T)co.rhp;
    }
    if ((cell_stages & 2) && ph.chem && ph.heatcool) {
      const double d = heatcool_delta<IONS>(ph, (double)s.rho[c], (double)s.eint[c], (double)s.rh2[c],
                                            ions ? (double)s.rhp[c] : 0.0, tau);
      s.E[c] = (T)((double)s.E[c] + d);
      s.eint[c] = (T)((double)s.eint[c] + d);
    }
    idx_t up[3] = {cmap(g, q[0] + 1, q[1], q[2]), cmap(g, q[0], q[1] + 1, q[2]),
                   cmap(g, q[0], q[1], q[2] + 1)};
#pragma unroll
    for (int d = 0; d < 3; ++d) Bc[d] = mul_t(T(0.5), add_t(s.b[d][c], s.b[d][up[d]]));
    rho = s.rho[c];
#pragma unroll
    for (int d = 0; d < 3; ++d) m[d] = s.m[d][c];
    T E = s.E[c];
    eint = s.eint[c];
    if (do_reg) {
      const T m2 = fma(m[2], m[2], fma(m[1], m[1], mul_t(m[0], m[0])));
      const T kin = mul_t(T(0.5), m2) / rho;
      const T mag = mul_t(T(0.5), fma(Bc[2], Bc[2], fma(Bc[1], Bc[1], mul_t(Bc[0], Bc[0]))));
      const T e = sub_t(sub_t(E, kin), mag);
      T f = e / E;
      bool entropy_branch = f >= T(1e-3);
      if (ph.regul_mode == 2) entropy_branch = !entropy_branch;
      if (entropy_branch) {
        if (ph.regul_mode != 0 || e > eint) eint = e;
      } else {
        T v2 = mul_t(T(2), sub_t(sub_t(E, eint), mag)) / rho;
        if (v2 < T(0)) v2 = T(0);
        T vnew = sqrt(v2);
        T vold = sqrt(m2) / rho;
        if (vold > T(0)) {
          T scl = vnew / vold;
#pragma unroll
          for (int d = 0; d < 3; ++d) m[d] = m[d] * scl;
        }
        vb = 1;
      }
      s.eint[c] = eint;
#pragma unroll
      for (int d = 0; d < 3; ++d) s.m[d][c] = m[d];
    }
    if (ph.chem) rh2 = s.rh2[c];
    if (ions) rhp = s.rhp[c];
    T vals[11] = {rho, m[0], m[1], m[2], E, eint, rh2, s.b[0][c], s.b[1][c], s.b[2][c], rhp};
#pragma unroll
    for (int k = 0; k < 11; ++k)
      if (!isfinite(vals[k])) bad = 1;
    if (!(rho > T(0)) || !(eint > T(0))) bad = 1;
  }
  cfl_of_cell(ph, B.sc, valid && !bad, ions, rho, m, Bc, eint, rh2, rhp, D);
}

// the warp's share of the post stage's box scalars: the largest FP64 CFL denominator, the
// non-physical flag and the count of velocity-branch regularisations
template <typename T>
__device__ __forceinline__ void post_warp_reduce(const Box<T>& B, double D, int bad, unsigned vb, int check) {
  if (!check) bad = 0;
  cfl_warp_reduce(B.sc, D);
  int anybad = __any_sync(0xffffffffu, bad);
  unsigned nvb = __popc(__ballot_sync(0xffffffffu, vb));
  if ((threadIdx.x & 31) == 0) {
    if (anybad) atomicOr(&B.sc->flags, 1);
    if (nvb) atomicAdd(&B.sc->vel_branch, (unsigned long long)nvb);
  }
}

template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(512) kb_post(const __grid_constant__ SRC src, int cell_stages,
                                               int do_reg, int check) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t c;
    const Box<T>& B = src.tile(t_, dir, c);
    c += (idx_t)threadIdx.x;
    double D = 0.0;
    int bad = 0;
    unsigned vb = 0;
    post_cell<T, IONS>(B, c, c < B.g.N, cell_stages, do_reg, D, bad, vb);
    post_warp_reduce(B, D, bad, vb, check);
  }
}

// The last Lagrangian substage (r = 2) and the post stage of a step in one pass.  A cell's update
// reads the face fluxes and the cell's own fields, and its post stage reads only the cell's own
// fields and the face field b, which neither changes; so one thread takes both, in program order,
// and the update's HBM traffic overlaps the post stage's FP64 work.
template <typename T, typename SRC, bool IONS>
__global__ void __launch_bounds__(512) kb_lag_update_post(const __grid_constant__ SRC src,
                                                          int cell_stages, int do_reg, int check) {
  dependent_launch_begin();
  MHD_TILE_LOOP(src) {
    int dir;
    idx_t c;
    const Box<T>& B = src.tile(t_, dir, c);
    c += (idx_t)threadIdx.x;
    const bool valid = c < B.g.N;
    if (valid) lag_update_cell<T, IONS>(B, c, 2);
    double D = 0.0;
    int bad = 0;
    unsigned vb = 0;
    post_cell<T, IONS>(B, c, valid, cell_stages, do_reg, D, bad, vb);
    post_warp_reduce(B, D, bad, vb, check);
  }
}

// tau of the step from the device-resident max denominator (Sec. 2.3; min over cells of
// CFL h / D equals CFL h / max D since rounding is monotone), truncated at t_end (A18).
template <typename T>
__global__ void kb_begin_step(const Box<T>* __restrict__ boxes, int nb) {
  dependent_launch_begin();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  Scalars* sc = boxes[b].sc;
  const double dx = boxes[b].ph.dx;
  if (!sc->fixed_tau) {
    double Dm = __longlong_as_double((long long)sc->dmax);
    double tau = sc->cfl * dx / Dm;
    if (sc->t_end > 0.0 && tau > sc->t_end - sc->t) tau = sc->t_end - sc->t;
    sc->tau = tau;
  }
  sc->tau_h = sc->tau / dx;
  sc->tau_h32 = (float)sc->tau_h;
  for (int r = 0; r < 3; ++r) sc->gth[r] = RK3_G(r) * sc->tau * boxes[b].ph.ih;
  const double ts = sc->tau * (ChemConst::PC / ChemConst::KMS);
  sc->ts[0] = (float)ts;
  sc->ts[1] = (float)(ts - (double)sc->ts[0]);
  if (!(sc->tau > 0.0)) sc->flags |= 2;
  sc->dmax = 0ull;  // the post kernel of this step accumulates the next state's denominator
  sc->dlow = 0;
}

template <typename T>
__global__ void kb_end_step(const Box<T>* __restrict__ boxes, int nb) {
  dependent_launch_begin();
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  Scalars* sc = boxes[b].sc;
  sc->t = sc->t + sc->tau;
  sc->steps += 1;
  // the host reads this word without synchronising (mhd_step with dt = NULL)
  if (boxes[b].hflags) *(volatile int*)boxes[b].hflags = sc->flags;
}

template <typename T>
__global__ void kb_set_params(const Box<T>* __restrict__ boxes, int nb, double cfl, double t_end,
                              int fixed_tau, double tau) {
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  Scalars* sc = boxes[b].sc;
  sc->cfl = cfl;
  sc->t_end = t_end;
  sc->fixed_tau = fixed_tau;
  if (fixed_tau) sc->tau = tau;
}

template <typename T>
__global__ void kb_zero_dmax(const Box<T>* __restrict__ boxes, int nb) {
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  boxes[b].sc->dmax = 0ull;
  boxes[b].sc->dlow = 0;
}

// ------------------------------------------------------------------------------------------------
// set_state helpers
// (a + b) / 2 of two inputs in FP64, rounded to T; of two floats to a float the FP32 sum and halving give
// the same value
template <typename T, typename In>
__device__ __forceinline__ T half_sum(In a, In b) {
  if constexpr (sizeof(T) == 4 && sizeof(In) == 4) return 0.5f * (a + b);
  else return (T)(0.5 * ((double)a + (double)b));
}
// The state from cell-centred input in one pass: the cell fields, the faces b_d(i_d - 1/2) = (B_d(i_d - 1) +
// B_d(i_d)) / 2 (A17), rho eps = rho E - |m|^2 / (2 rho) - |B_cell|^2 / 2 with B_cell from the stored
// faces, whose upper one is formed again from the input (with an open boundary the upper face of
// the last cell is its lower one), and the first tau's CFL denominator (the box's scalars are zero).  As
// five launches (cells, faces, rho eps, the scalars' reset, the CFL pass) mhd_set_state from device memory
// took 1.27 ms for 256^3 cells of FP32 and 0.068 ms for 32^3, as one 0.41 and 0.044 ms.  (The half sums of
// floats in FP64 alone cost 0.6 ms: each conversion takes the FP64 pipe as long as an FMA.)
template <typename T, typename In>
__global__ void __launch_bounds__(256) k_load_state(Geom g, Phys ph, Scalars* sc, State<T> s, const In* rho_,
                                                    const In* mx, const In* my, const In* mz, const In* E_,
                                                    const In* Bx, const In* By, const In* Bz, const In* rh2) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool valid = c < g.N;
  T rho = T(0), m[3] = {T(0), T(0), T(0)}, B[3] = {T(0), T(0), T(0)}, eint = T(0), h2 = T(0);
  bool bad = false;
  if (valid) {
    int q[3];
    decode_cell(g, (idx_t)c, q);
    const In* Bi[3] = {Bx, By, Bz};
    T b[3];
    m[0] = (T)mx[c];
    m[1] = (T)my[c];
    m[2] = (T)mz[c];
    rho = (T)rho_[c];
    const T E = (T)E_[c];
    if (rh2) h2 = (T)rh2[c];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      int lo[3] = {q[0], q[1], q[2]}, hi[3] = {q[0], q[1], q[2]};
      lo[d] -= 1;
      hi[d] += 1;
      const In Bc = Bi[d][c];
      b[d] = half_sum<T>(Bi[d][cmap(g, lo[0], lo[1], lo[2])], Bc);
      const bool last = g.bc[d] != 0 && hi[d] == g.n[d];
      const T up = last ? b[d] : half_sum<T>(Bc, Bi[d][cmap(g, hi[0], hi[1], hi[2])]);
      B[d] = T(0.5) * (b[d] + up);
    }
    const T kin = T(0.5) * (m[0] * m[0] + m[1] * m[1] + m[2] * m[2]) / rho;
    const T mag = T(0.5) * (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
    eint = E - kin - mag;
    s.rho[c] = rho;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      s.m[d][c] = m[d];
      s.b[d][c] = b[d];
    }
    s.E[c] = E;
    s.eint[c] = eint;
    if (s.rh2) s.rh2[c] = h2;
    if (s.rhp) s.rhp[c] = T(0);
    const T vals[10] = {rho, m[0], m[1], m[2], E, eint, ph.chem ? h2 : T(0), b[0], b[1], b[2]};
#pragma unroll
    for (int k = 0; k < 10; ++k)
      if (!isfinite(vals[k])) bad = true;
    if (!(rho > T(0)) || !(eint > T(0))) bad = true;
  }
  double D = 0.0;
  cfl_of_cell(ph, sc, valid && !bad, ph.chem && ph.ions, rho, m, B, eint, ph.chem ? h2 : T(0), T(0), D);
  cfl_warp_reduce(sc, D);
}

template <typename T>
__global__ void k_faces_copy(Geom g, State<T> s, const double* bx, const double* by, const double* bz) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.N) return;
  s.b[0][c] = (T)bx[c];
  s.b[1][c] = (T)by[c];
  s.b[2][c] = (T)bz[c];
}

// rho eps = rho E - |m|^2 / (2 rho) - |B_cell|^2 / 2 with B_cell from the faces
template <typename T>
__global__ void k_derive_eint(Geom g, State<T> s) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.N) return;
  int i = (int)(c % g.n[0]);
  long long r = c / g.n[0];
  int j = (int)(r % g.n[1]);
  int k = (int)(r / g.n[1]);
  long long up[3] = {cmap(g, i + 1, j, k), cmap(g, i, j + 1, k), cmap(g, i, j, k + 1)};
  T B[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) B[d] = T(0.5) * (s.b[d][c] + s.b[d][up[d]]);
  T rho = s.rho[c];
  T kin = T(0.5) * (s.m[0][c] * s.m[0][c] + s.m[1][c] * s.m[1][c] + s.m[2][c] * s.m[2][c]) / rho;
  T mag = T(0.5) * (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
  s.eint[c] = s.E[c] - kin - mag;
}

template <typename T, typename Out>
__global__ void k_store_state(Geom g, State<T> s, Out* rho, Out* mx, Out* my, Out* mz, Out* E,
                              Out* Bx, Out* By, Out* Bz, Out* rh2) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.N) return;
  int i = (int)(c % g.n[0]);
  long long r = c / g.n[0];
  int j = (int)(r % g.n[1]);
  int k = (int)(r / g.n[1]);
  long long up[3] = {cmap(g, i + 1, j, k), cmap(g, i, j + 1, k), cmap(g, i, j, k + 1)};
  Out* B[3] = {Bx, By, Bz};
#pragma unroll
  for (int d = 0; d < 3; ++d) B[d][c] = (Out)(T(0.5) * (s.b[d][c] + s.b[d][up[d]]));
  rho[c] = (Out)s.rho[c];
  mx[c] = (Out)s.m[0][c];
  my[c] = (Out)s.m[1][c];
  mz[c] = (Out)s.m[2][c];
  E[c] = (Out)s.E[c];
  if (rh2) rh2[c] = s.rh2 ? (Out)s.rh2[c] : Out(0);
}

template <typename T>
__global__ void k_store_full(Geom g, State<T> s, double* eint, double* bx, double* by, double* bz) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.N) return;
  eint[c] = (double)s.eint[c];
  bx[c] = (double)s.b[0][c];
  by[c] = (double)s.b[1][c];
  bz[c] = (double)s.b[2][c];
}

// rho_H+ in and out (FP64 interface)
template <typename T>
__global__ void k_load_ions(Geom g, State<T> s, const double* rhp) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c < g.N) s.rhp[c] = (T)rhp[c];
}

template <typename T>
__global__ void k_store_ions(Geom g, State<T> s, double* rhp) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c < g.N) rhp[c] = (double)s.rhp[c];
}

template <typename T>
__global__ void k_load_full(Geom g, State<T> s, const double* eint, const double* bx,
                            const double* by, const double* bz) {
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= g.N) return;
  s.eint[c] = (T)eint[c];
  s.b[0][c] = (T)bx[c];
  s.b[1][c] = (T)by[c];
  s.b[2][c] = (T)bz[c];
}

// ------------------------------------------------------------------------------------------------
// FP64 diagnostics: fixed-shape tree reduction (block partials, then one block) -> deterministic.
// Partial layout per block: 8 sums + 1 max.
constexpr int DIAG_THREADS = 256;

template <typename T>
__global__ void __launch_bounds__(DIAG_THREADS) k_diag_partial(Geom g, State<T> s, double* part) {
  __shared__ double sh[9][DIAG_THREADS];
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (c < g.N) {
    int i = (int)(c % g.n[0]);
    long long r = c / g.n[0];
    int j = (int)(r % g.n[1]);
    int k = (int)(r / g.n[1]);
    long long up[3] = {cmap(g, i + 1, j, k), cmap(g, i, j + 1, k), cmap(g, i, j, k + 1)};
    v[0] = (double)s.rho[c];
    v[1] = (double)s.m[0][c];
    v[2] = (double)s.m[1][c];
    v[3] = (double)s.m[2][c];
    v[4] = (double)s.E[c];
    v[5] = (double)s.b[0][c];
    v[6] = (double)s.b[1][c];
    v[7] = (double)s.b[2][c];
    double div = ((double)s.b[0][up[0]] - (double)s.b[0][c]) + ((double)s.b[1][up[1]] - (double)s.b[1][c]) +
                 ((double)s.b[2][up[2]] - (double)s.b[2][c]);
    v[8] = fabs(div);
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = DIAG_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
#pragma unroll
      for (int q = 0; q < 8; ++q) sh[q][threadIdx.x] = sh[q][threadIdx.x] + sh[q][threadIdx.x + w];
      sh[8][threadIdx.x] = fmax(sh[8][threadIdx.x], sh[8][threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 9) part[(long long)blockIdx.x * 9 + threadIdx.x] = sh[threadIdx.x][0];
}

static __global__ void __launch_bounds__(DIAG_THREADS) k_diag_final(const double* part, int nblocks, double* out) {
  __shared__ double sh[9][DIAG_THREADS];
  double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nblocks; b += DIAG_THREADS) {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = v[q] + part[(long long)b * 9 + q];
    v[8] = fmax(v[8], part[(long long)b * 9 + 8]);
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = DIAG_THREADS / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
#pragma unroll
      for (int q = 0; q < 8; ++q) sh[q][threadIdx.x] = sh[q][threadIdx.x] + sh[q][threadIdx.x + w];
      sh[8][threadIdx.x] = fmax(sh[8][threadIdx.x], sh[8][threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 9) out[threadIdx.x] = sh[threadIdx.x][0];
}

}  // namespace mhd
