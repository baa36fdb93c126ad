// Internal declarations of libnsi_assemble: the handle, status helpers and the
// per-element arithmetic shared by the kernels.  Nothing here is part of the
// public ABI (include/nsi_assemble.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/nsi_assemble.h"

namespace nsi {

// ---------------------------------------------------------------- status ---
void set_error(const std::string& msg);
nsi_status fail(nsi_status s, const std::string& msg);
nsi_status cuda_fail(cudaError_t e, const char* what);

#define NSI_CUDA(call)                                   \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return nsi::cuda_fail(e_, #call); \
  } while (0)

// device error word bits (set by kernels built with debug checks)
enum : unsigned { ERR_BAD_INDEX = 1u, ERR_NOT_IN_PATTERN = 2u, ERR_STAR = 4u };

// Row-gather ("pull") map, built at create time: for CSR row i, one 16-bit
// word per element that contains node i (the row's star): the positions,
// inside row i's column list, of the element's other three nodes (5 bits
// each), ordered so that (i, j1, j2, j3) is an even permutation of the
// element's node order (hence a positively oriented tet).  The kernels read
// the element walk encoded from these words (WALK_* below) and the edge-fan
// map.  Rows longer than 32 entries cannot be encoded: "long rows" (DIAG_LONG).
constexpr int STAR_BITS = 5;
constexpr int STAR_MAX_ROW = 1 << STAR_BITS;
// an element with |d1||d2||d3| > EXACT_RATIO |det| (edge vectors from any of
// its nodes) is "badly shaped": in the mixed modes the rows of its nodes are
// recomputed in double after the assembly
constexpr double EXACT_RATIO = 16.0;
// One step of a row's element walk (one byte): the row position of the node
// it brings into the window, whether the element formed by the window and that
// node is evaluated, the element's orientation in window order, and which
// window node leaves afterwards.
constexpr unsigned WALK_POS = 31u;       // bits 0-4: row position of the new node
constexpr unsigned WALK_ELEM = 1u << 5;  // the step evaluates element (p, q, c)
constexpr unsigned WALK_NEG = 1u << 6;   // (p, q, c) is an odd permutation of the element's order
constexpr unsigned WALK_EVQ = 1u << 7;   // q leaves (next window (p, c)); else p leaves (next window (q, c))

// Element-position map, for the element-centric kernels: per element one
// 64-bit word holding, for every ordered pair (a, b) of its local nodes with
// b != a, the position of node b inside the CSR row of node a, 5 bits each,
// at bit 5 * (3a + (b < a ? b : b - 1)); the diagonal positions come from
// diag_pos.  Built for meshes whose rows have at most 32 entries (others scan
// the row).
constexpr int ELEM_POS_BITS = 5;
__host__ __device__ inline int elem_pos_slot(int a, int b) { return 3 * a + (b < a ? b : b - 1); }

// Edge-fan map: for every off-diagonal CSR entry (i, j), the ring of nodes
// around the edge (i, j) -- the other two nodes of every element containing
// both i and j, chained in cyclic order so that consecutive ring nodes k, l
// form the positively oriented element (i, j, k, l) -- as positions inside
// row i.  One 32-bit word per entry: ring positions in bits 0..23 (4 bits
// each, up to 6 of them), ring size in bits 24..26, bit 27 set when the ring
// is closed (interior edge: as many elements as ring nodes) and clear when it
// is open (boundary edge: one element fewer).  The diagonal entry has word 0.
// Meshes with rows longer than 16 entries, rings longer than 6 nodes or
// non-manifold edge fans do not get the map and use the per-row star kernel.
constexpr int FAN_MAX_ROW = 16;
constexpr int FAN_MAX_RING = 6;
constexpr int FAN_BLOCK = 256;  // CSR entries (threads) per fan block

// vector types with explicit alignment (CUDA 13 deprecates the unsuffixed double4)
struct alignas(32) D4 {
  double x, y, z, w;
};

struct GatherPlan {
  int rows_per_block = 0;     // the plan's name: 32, 64, 96 or 128
  int warps = 0;              // warps per block, each with row groups of its own
  int max_block_steps = 0;    // max over the groups of the walk bytes of a group's rows
  int w = 0;                  // slots per row (>= the off-diagonal entries of the longest row the kernels
                              // take, and large enough for the staging)
  bool long_group = false;    // a group has more entries, a long row's among them, than its staging holds
};
// A mesh of fewer rows has four lanes per row in the row gather, which then
// reads the nodes' own data in a single launch; others have two lanes (or one)
// and a packing launch with the row gather started as it ends.  Assembly, us,
// two -> four: 2,197 rows mixed64 8.3 -> 6.2, FP64 39 -> 25; 9,261 rows 10.3 ->
// 8.2 and 41 -> 41; 12,167 rows 10.3 -> 8.3 and 55 -> 59; 15,625 rows 10.3 -> 10.3
// and 61 -> 70; 19,683 rows 10.3 -> 12.0 and 74 -> 80 (time step and nodal
// outputs cross at the same sizes): the line is FP64's.
constexpr int64_t SMALL_MESH_ROWS = 10000;
// From here on FP64 has one lane per row.  Below, two lanes' smaller groups fill
// the last round better at most sizes; above, the merge's additions weigh more.
// Assembly, us, one -> two lanes: 68,921 rows 246 -> 232, 79,507 264 -> 274,
// 91,125 323 -> 299, 103,823 348 -> 337, 110,592 351 -> 356, 125,000 412 -> 403,
// 148,877 491 -> 474, 166,375 516 -> 526, 185,193 584 -> 581, 205,379 656 -> 643,
// 226,981 686 -> 704, 287,496 853 -> 884.
constexpr int64_t LARGE_FP64_ROWS = 215000;
constexpr int SMEM_MAX = 200 * 1024;  // shared memory of one block

// diag_pos value of a row the row gather leaves out ("long row": more than
// 32 entries, or a star whose walk does not encode): the kernels give it no
// elements and zero its slice, or leave it out where it is longer than their
// staging; rows64_kernel computes it afterwards
constexpr uint8_t DIAG_LONG = 0xff;

// What a launch of the row gather computes: the assembly, the time step with
// cached geometry, the nodal outputs.
enum { ASSEMBLE = 0, STEP = 1, NODAL = 2 };

// Shared-memory layout of one warp's group of the row gather: R rows, W slots
// per row (the off-diagonal entries of the longest row of the mesh), H lanes
// per row, L entries of staging and S walk bytes.  Slot q of row t lives at
// index q * R + t ("row-interleaved"), so the lanes of a warp touch consecutive
// records whichever slot each row uses: the element loop is free of
// shared-memory bank conflicts.
//   nb0   T[4] per slot: edge vector d = x_j - x_i and u_x of the neighbour
//   nb1   T[2] per slot: u_y, u_z
//   acc   H planes of accumulators per slot (ab bytes each): A and the three
//         sums of c_i (time step: A; nodal outputs: none)
//   walk  the walk bytes (copied as aligned 4-byte words, so S + 8 bytes)
//   info  the next group's row bounds and diagonal positions
// After the element loop, nb0 and nb1 are reused to stage the finished values
// for the coalesced write-out (4 T per entry, in CSR order, or row t's from
// t * (W + 1) on), and past them for the next group's column indices.
// The host sizes launches by it and hands the kernels its offsets.
struct GatherSmem {
  int R, W, L, S, H, tb, ab;
  static size_t up16(size_t x) { return (x + 15) & ~size_t(15); }
  size_t N() const { return (size_t)R * W; }
  size_t nb1() const { return up16((size_t)4 * tb * N()); }
  size_t acc() const { return up16(nb1() + (size_t)2 * tb * N()); }
  size_t plane() const { return (size_t)ab * N(); }
  size_t walk() const { return up16(acc() + plane() * H); }
  size_t info() const { return up16(walk() + (size_t)S + 8); }
  // (a multiple of 32: the next warp's nb0 holds 32-byte aligned FP64 vectors)
  size_t total() const { return (info() + 8 * (size_t)(R + 1) + R + 31) & ~size_t(31); }
  // the column indices of the next group's entries, past the staged entries
  size_t cols() const { return up16((size_t)4 * tb * L); }
  bool group_fits() const { return cols() + (size_t)4 * L <= acc(); }
};

// the layout of a group of 32 / H rows whose staging holds W + 1 entries of each
inline GatherSmem gather_smem(int precision, int mode, int H, int W, int S) {
  GatherSmem g;
  g.R = 32 / H;
  g.W = W;
  g.L = g.R * (W + 1);
  g.S = S;
  g.H = H;
  g.tb = precision == NSI_FP64 ? 8 : 4;
  g.ab = mode == ASSEMBLE ? 4 * g.tb : mode == STEP ? g.tb : 0;
  return g;
}
// the slots of a mesh whose longest row has `slots` off-diagonal entries: those,
// or more where the staging would not fit nb0 and nb1
inline int group_slots(int precision, int H, int slots) {
  int W = slots;
  while (!gather_smem(precision, ASSEMBLE, H, W, 0).group_fits()) ++W;
  return W;
}

int gather_kernel_regs(int precision);  // registers per thread of the row-gather kernel

}  // namespace nsi

struct NsiHandle {
  int device = 0;
  int64_t n = 0, E = 0, nnz = 0;
  int precision = NSI_FP64;
  int scatter = NSI_SCATTER_AUTO;
  int block = 256;
  int debug = 0;
  int max_row = 0;
  int n_colors = 0;
  bool gather_ok = false;
  int64_t device_bytes = 0;

  // CSR pattern
  int32_t* row_ptr = nullptr;  // [n+1]
  int32_t* col_idx = nullptr;  // [nnz]
  // connectivity copy and colouring
  int4* lnods = nullptr;        // [E]
  int32_t* color_elems = nullptr;  // [E] element ids grouped by colour
  std::vector<int64_t> color_off;  // host [n_colors + 1]
  // row-gather map: every row's element walk (one byte per step)
  uint32_t* walk_ptr = nullptr;  // [n+1]
  uint8_t* walk = nullptr;      // [walk_ptr[n] + 8]
  int nsub = 2;                 // sub-walks per row
  bool packs() const { return nsub != 4; }  // the row gather reads packed node records (else the nodes' own data)
  uint8_t* diag_pos = nullptr;  // [n + 32] position of the diagonal inside its row (rows <= 32 entries)
  unsigned long long* elem_pos = nullptr;  // [E] element-position map (rows <= 32 entries), or null
  // edge-fan map (one word per CSR entry) and its block partition of the rows
  bool fan_ok = false;
  uint32_t* fan = nullptr;      // [nnz]
  int32_t* fan_blk = nullptr;   // [fan_blocks + 1] first row of every fan block
  int64_t fan_blocks = 0;
  bool use_fan = false;         // row-gather mode runs the edge-fan kernel
  bool atomic_agg = false;      // atomic mode runs the warp-aggregated atomics (else one atomic per value)
  int64_t long_rows = 0;        // rows the row gather leaves out, recomputed by rows64_kernel
  int32_t* long_list = nullptr;  // [long_rows] their node ids
  int32_t* long_ptr = nullptr;   // [long_rows + 1] into long_inc
  uint32_t* long_inc = nullptr;  // element * 4 + local index of the row's node
  int64_t n_bad = 0;            // mixed modes: badly shaped elements (the adjoint and residual take them in double)
  int32_t* bad_list = nullptr;  // [n_bad] their ids
  uint32_t* bad_mask = nullptr; // [ceil(E / 32)] one bit per element, or null when there are none
  // mixed modes: the rows of badly shaped elements, recomputed in double: first
  // those with a walk (exact_rows of them, at most exact_slots off-diagonal
  // entries), then the rest (exact_rest)
  int64_t exact_rows = 0, exact_rest = 0;
  int exact_slots = 0;
  int32_t* exact_list = nullptr;  // [exact_rows + exact_rest] their node ids
  int32_t* exact_ptr = nullptr;   // [exact_rows + exact_rest + 1] into exact_inc
  uint32_t* exact_inc = nullptr;  // element * 4 + local index of the row's node
  // the stabilised block's row kernel: every row's star as row positions of
  // each element's other three nodes (five bits each, the row's node and the
  // three in a positively oriented order), and its warp tasks (one row, or two
  // consecutive rows of at most 16 entries), each described by two int4:
  // {first row, CSR start of the first row, of the second, end} and
  // {star start of the first row, of the second, end, diagonal positions |
  // rows << 16 | long << 24}
  uint16_t* star_word = nullptr;  // [incidences]
  int4* star_task = nullptr;      // [2 n_star_tasks]
  int64_t n_star_tasks = 0;
  nsi::GatherPlan plan;         // the launch plan in use
  nsi::GatherPlan plans[4];     // the distinct launches (warps per block, ascending), by the first name of each
  int n_plans = 0;
  std::atomic<int> resident[3][4] = {};  // row gather by mode and warps per block: blocks resident at once (0: not known)
  // coordinates: double4 for FP64, float4 hi + float4 lo for the mixed modes
  nsi::D4* xyz64 = nullptr;
  float4* xyz_hi = nullptr;
  float4* xyz_lo = nullptr;
  // per-call node records for the row-gather kernel (one 32-byte record per node
  // in the mixed modes, 64 bytes in FP64): coordinates and velocity of a node
  // in one or two DRAM sectors, rebuilt at the start of every gather call
  void* rec = nullptr;
  int rec_bytes = 0;
  // optional profiling events around the main assembly kernel
  cudaEvent_t ev_start = nullptr, ev_stop = nullptr;
  // device error word
  unsigned* err = nullptr;
  // staging for nsi_assemble_host (allocated on first use)
  void* stage = nullptr;
  size_t stage_bytes = 0;
  // host-buffer calls: the CSR row starts on the host, and a stream and
  // events on which finished chunks of the outputs go to the host while the
  // next chunk is assembled
  std::vector<int32_t> row_ptr_host;  // [n+1]
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t chunk_ev[8] = {};
};

namespace nsi {

// --------------------------------------------------- element arithmetic ---
// For a positively oriented tet with edge vectors d1, d2, d3 leaving vertex 0,
// the cofactor vectors c_b = det(J) grad N_b are
//   c1 = d2 x d3,  c2 = d3 x d1,  c3 = d1 x d2,  c0 = -(c1 + c2 + c3),
// det J = d1 . c1 and |T| = det J / 6.  With them the Galerkin P1 terms are
//   convection  rho int N_a (u_h . grad N_b) = rho/120 (S + u_a) . c_b,
//               S = sum_c u_c  (exact P1 mass moments int N_a N_c = |T|(1+d_ac)/20,
//               which the 4-point Gauss rule integrates exactly)
//   viscous     mu |T| grad N_a . grad N_b  = mu / (6 det) c_a . c_b
//   lumped mass rho |T| / (4 dt)            = rho det / (24 dt)
//   pressure gradient  -int d_d N_a N_b     = -c_a[d] / 24  (every b)
//   lumped RHS  rho |T| u^n_a / (4 dt)      = rho det / (24 dt) u^n_a
template <typename T>
struct V3 {
  T x, y, z;
};
template <typename T>
__host__ __device__ __forceinline__ V3<T> cross(const V3<T>& a, const V3<T>& b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
template <typename T>
__host__ __device__ __forceinline__ T dot(const V3<T>& a, const V3<T>& b) {
  return a.x * b.x + a.y * b.y + a.z * b.z;
}
template <typename T>
__host__ __device__ __forceinline__ V3<T> add(const V3<T>& a, const V3<T>& b) {
  return {a.x + b.x, a.y + b.y, a.z + b.z};
}
template <typename T>
__host__ __device__ __forceinline__ V3<T> sub(const V3<T>& a, const V3<T>& b) {
  return {a.x - b.x, a.y - b.y, a.z - b.z};
}

// ------------------------------------------------ f32 -> f64 without DP ops ---
// GB300 executes double-precision instructions (including conversions) at a
// small fraction of the single-precision rate, so the mixed modes build their
// double outputs from integer operations on the IEEE-754 bit patterns.

// Exact float -> double (every float is a double).  Subnormal floats are
// renormalised; inf/nan keep their class.
__device__ __forceinline__ long long f32_to_f64_bits(float f) {
  unsigned u = __float_as_uint(f);
  unsigned sign = u & 0x80000000u;
  unsigned e = (u >> 23) & 0xffu;
  unsigned m = u & 0x7fffffu;
  unsigned e64;
  if (e == 0u) {
    if (m == 0u) return (long long)((unsigned long long)sign << 32);
    int lz = __clz(m) - 8;  // shift that brings the leading 1 to bit 23
    m = (m << lz) & 0x7fffffu;
    e64 = 897u - (unsigned)lz;  // 1 - 127 + 1023 - lz
  } else if (e == 0xffu) {
    e64 = 0x7ffu;
  } else {
    e64 = e + 896u;  // 1023 - 127
  }
  unsigned hi = sign | (e64 << 20) | (m >> 3);
  unsigned lo = m << 29;
  return (long long)(((unsigned long long)hi << 32) | lo);
}


// error-free sum: s + e == a + b exactly (Knuth's TwoSum, 6 float ops)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

}  // namespace nsi
