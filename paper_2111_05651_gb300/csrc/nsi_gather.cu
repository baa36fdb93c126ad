// The row gather: the assembly (A, G, rhs), the time step with cached
// geometry (A = A_static + C(u), rhs) and the paper's per-node outputs, for
// one mesh or a batch of meshes.
//
//   pack_kernel, batched_pack_kernel  the call's node records
//   gather_persistent_kernel          one mesh, a persistent grid of warps
//   batched_kernel                    many meshes in one persistent launch
//
// A warp takes groups of 32 / H consecutive CSR rows, H lanes per row.  The
// elements around a row's node (its star) are ordered at create along walks of
// neighbouring elements and cut into `nsub` sub-walks; each of the row's lanes
// follows its own and adds into its own accumulators, and the lanes' sums are
// merged in a fixed order, so results do not depend on timing.  Every output
// is written once, in memory order; there are no atomics and no zeroing.
//
// What bounds it, and why H lanes per row: a walk is a serial chain of element
// evaluations, and the slots it works on (edge vectors, velocities and
// accumulators of a row's neighbours) are in shared memory, which limits the
// resident warps.  One lane per row kept 32 rows of slots per warp (20 KB, 11
// warps per SM) behind chains of 24 elements; two lanes per row keep 16 rows
// and a second set of accumulators (13 KB, 16 warps) behind chains of 12, and
// the neighbours' records come as one 256-bit load each, in registers under the
// previous group's write-out, instead of two 16-byte copies through shared
// memory (100^3 cube, us, one lane per row -> two: mixed64 277 -> 270 in random
// and 269 -> 221 in natural node order, mixed32 228 -> 224, time step 275 ->
// 195, nodal outputs 216 -> 121; 47x61x38 mixed32 39.6 -> 31.4).  The records
// bypass L1 (allocating there costs 407 us: 115 KB of sectors in flight per SM
// through the 28 KB that shared memory leaves).  What is left is the shared
// memory's data path (72% busy: 650 wavefronts of a group's 16 rows) and issue
// (59%), and in random node order the rate of scattered 32-byte requests (50 us
// against natural order; loading still earlier changes nothing).
//
// A small mesh has four lanes per row: its groups do not fill the chip, so the
// chain is the time (8^3 cube in FP64: 66 us with one lane, 27 with four; at
// 100^3 four cost mixed64 374 us).  FP64 is bound by the FP64 pipe (one warp
// instruction in 18 cycles, 97-100% busy): a large mesh has one lane per row,
// which saves the merge's additions (100^3: 2977 us, with two 3057, before all
// this 3023).  SMALL_MESH_ROWS and LARGE_FP64_ROWS have the sizes around the lines.
#include <algorithm>
#include <mutex>

#include "nsi_device.cuh"

namespace nsi {

namespace {

constexpr int MAX_WARPS = 4;  // warps per block

// --------------------------------------------------------------- copies ---
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// A node's record in registers: 32 bytes (mixed) or 64 (FP64) by 256-bit loads
// (records are 32-byte aligned and written by an earlier launch).
template <int P>
struct NodeRec {
  uint4 a, b;
  __device__ __forceinline__ void load(const void* rec, int64_t j) {
    load_record<false>(static_cast<const unsigned*>(rec) + 8 * j, a, b);
  }
  // the record's words from the node's own data, without a packed record
  template <typename Mesh>
  __device__ __forceinline__ void gather(const Mesh& m, const FieldView& f, int64_t j) {
    const uint4 hi = __ldg(reinterpret_cast<const uint4*>(m.xyz_hi + j));
    const uint4 lo = __ldg(reinterpret_cast<const uint4*>(m.xyz_lo + j));
    const V3<float> u = load_vec<float>(f.u, j);
    a = make_uint4(hi.x, hi.y, hi.z, __float_as_uint(u.x));
    b = make_uint4(__float_as_uint(u.y), __float_as_uint(u.z), (lo.x >> 16) | (lo.y & 0xffff0000u),
                   lo.z & 0xffff0000u);
  }
  // edge vector from node o to this one
  __device__ __forceinline__ V3<float> minus(const NodeRec& o) const {
    const V3<float> h{__uint_as_float(a.x) - __uint_as_float(o.a.x), __uint_as_float(a.y) - __uint_as_float(o.a.y),
                      __uint_as_float(a.z) - __uint_as_float(o.a.z)};
    return add(h, sub(record_lo(__uint_as_float(b.z), __uint_as_float(b.w)),
                      record_lo(__uint_as_float(o.b.z), __uint_as_float(o.b.w))));
  }
  __device__ __forceinline__ V3<float> vel() const {
    return {__uint_as_float(a.w), __uint_as_float(b.x), __uint_as_float(b.y)};
  }
};
template <>
struct NodeRec<NSI_FP64> {
  double x, y, z, ux, uy, uz;
  __device__ __forceinline__ void load(const void* rec, int64_t j) {
    const double* r = static_cast<const double*>(rec) + 8 * j;
    load_record<false>(r, x, y, z);
    load_record<false>(r + 4, ux, uy, uz);
  }
  template <typename Mesh>
  __device__ __forceinline__ void gather(const Mesh& m, const FieldView& f, int64_t j) {
    const D4 p = m.xyz64[j];
    const V3<double> u = load_vec<double>(f.u, j);
    x = p.x, y = p.y, z = p.z;
    ux = u.x, uy = u.y, uz = u.z;
  }
  __device__ __forceinline__ V3<double> minus(const NodeRec& o) const { return {x - o.x, y - o.y, z - o.z}; }
  __device__ __forceinline__ V3<double> vel() const { return {ux, uy, uz}; }
};

// -------------------------------------------------------------- kernel I/O ---
// the layout of a warp's shared memory (GatherSmem) as the kernels take it:
// byte offsets of its regions, the bytes of one accumulator plane, R * W, and
// the limits that the bounds checks compare with.  Kernel parameters are
// operands of the instructions that use them and take no registers.
struct GroupLay {
  int nb1, acc, plane, walk, info, cols, total, N, W, L, S;
  GroupLay() = default;
  explicit GroupLay(const GatherSmem& g)
      : nb1((int)g.nb1()), acc((int)g.acc()), plane((int)(g.ab * g.N())), walk((int)g.walk()), info((int)g.info()),
        cols((int)g.cols()), total((int)g.total()), N((int)g.N()), W(g.W),
        L(g.L), S(g.S) {}
};
// what the kernels read of a mesh
struct WalkMesh {
  int64_t n, nnz;
  const int32_t* row_ptr;
  const int32_t* col_idx;
  const uint32_t* walk_ptr;
  const uint8_t* walk;
  const uint8_t* diag_pos;
  const D4* xyz64;
  const float4* xyz_hi;
  const float4* xyz_lo;
  void* rec;
  unsigned* err;
};
// outputs by mode (kmr = rho/24, the density mass per det)
template <int MODE>
struct WalkOut;
template <>
struct WalkOut<ASSEMBLE> {
  void *A, *G, *rhs;
};
template <>
struct WalkOut<STEP> {
  void *A, *rhs;
  const void* A_static;
};
template <>
struct WalkOut<NODAL> {
  void *rhs, *dt_rho, *mass_rho;
  double kmr;
  float kmrf;
};
template <int MODE>
struct WalkItem {
  WalkMesh m;
  FieldView f;
  WalkOut<MODE> o;
  int group0;  // the first of the mesh's row groups in the launch
};

// ------------------------------------------------------------ the sub-walk ---
// Products that are rounded, and cross and dot products with their
// multiply-adds spelt out: the single-mesh and the batched kernel are compiled
// apart and give the same bits.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <typename T>
__device__ __forceinline__ V3<T> cross_fma(const V3<T>& a, const V3<T>& b) {
  return {fma(a.y, b.z, -mul_rn(a.z, b.y)), fma(a.z, b.x, -mul_rn(a.x, b.z)), fma(a.x, b.y, -mul_rn(a.y, b.x))};
}
template <typename T>
__device__ __forceinline__ T dot_fma(const V3<T>& a, const V3<T>& b) {
  return fma(a.z, b.z, fma(a.y, b.y, mul_rn(a.x, b.x)));
}

// Accumulators of a row's slots in shared memory, one plane per lane of the
// row: the sums of A and of the pressure gradient (-c_i / 24) of each entry
// (mixed: a float4 (G_x, G_y, G_z, A); FP64 two planes (A, G_x), (G_y, G_z));
// the time step only A.  A slot is touched by one lane until the merge.
template <int P, int MODE>
struct Slots;
// paired float arithmetic: one instruction for two lanes of a float2
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

template <int P>
struct Slots<P, ASSEMBLE> {
  float4* a;
  struct V {
    float2 g, r;  // (G_x, G_y), (G_z, A)
  };
  __device__ __forceinline__ Slots(unsigned char* p, size_t) : a(reinterpret_cast<float4*>(p)) {}
  static __device__ __forceinline__ V zero_value() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
  __device__ __forceinline__ V load(int k) const {
    const float4 v = a[k];
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
  }
  __device__ __forceinline__ void store(int k, const V& v) { a[k] = make_float4(v.g.x, v.g.y, v.r.x, v.r.y); }
  static __device__ __forceinline__ V sum(const V& x, const V& y) { return {add2(x.g, y.g), add2(x.r, y.r)}; }
};
template <>
struct Slots<NSI_FP64, ASSEMBLE> {
  T2<double>*a0, *a1;
  struct V {
    T2<double> x, y;  // (A, G_x), (G_y, G_z)
  };
  __device__ __forceinline__ Slots(unsigned char* p, size_t N)
      : a0(reinterpret_cast<T2<double>*>(p)), a1(reinterpret_cast<T2<double>*>(p) + N) {}
  static __device__ __forceinline__ V zero_value() { return {{0.0, 0.0}, {0.0, 0.0}}; }
  __device__ __forceinline__ V load(int k) const { return {a0[k], a1[k]}; }
  __device__ __forceinline__ void store(int k, const V& v) {
    a0[k] = v.x;
    a1[k] = v.y;
  }
  static __device__ __forceinline__ V sum(const V& x, const V& y) {
    return {{x.x.x + y.x.x, x.x.y + y.x.y}, {x.y.x + y.y.x, x.y.y + y.y.y}};
  }
};
template <int P>
struct Slots<P, STEP> {
  using V = typename Prec<P>::T;
  V* a;
  __device__ __forceinline__ Slots(unsigned char* p, size_t) : a(reinterpret_cast<V*>(p)) {}
  static __device__ __forceinline__ V zero_value() { return V(0); }
  __device__ __forceinline__ V load(int k) const { return a[k]; }
  __device__ __forceinline__ void store(int k, V v) { a[k] = v; }
  static __device__ __forceinline__ V sum(V x, V y) { return x + y; }
};
template <int P>
struct Slots<P, NODAL> {
  struct V {};
  __device__ __forceinline__ Slots(unsigned char*, size_t) {}
  static __device__ __forceinline__ V zero_value() { return {}; }
  __device__ __forceinline__ V load(int) const { return {}; }
  __device__ __forceinline__ void store(int, V) {}
  static __device__ __forceinline__ V sum(V, V) { return {}; }
};

// One lane's sub-walk of one row, node i as the origin: segments of
// neighbouring elements.  A window of two neighbours (p, q) stays in registers
// with their edge vectors, velocities and accumulators; every step brings one
// node c in from shared memory, evaluates the element (i, p, q, c), then
// writes back the accumulator of the node that leaves the window; c always
// becomes q, and p keeps its node or takes q's.  With
// c_p = d_q x d_c, c_q = d_c x d_p, c_c = d_p x d_q (cofactors of the
// Jacobian, calculate_cartesian_derivatives, for the order (p, q, c)),
// det = d_p . c_p and c_i = -(c_p + c_q + c_c), the element adds
//   A(i,x) += w . c_x  (x = p, q, c),  w = rho/120 (2 u_i + u_p + u_q + u_c) + mu/(6 det) c_i
// (p's velocity carries the 2 u_i; in FP64 the staged velocities carry the
// factor rho/120 too, which saves its products on the FP64 pipe; in float, where
// a product per velocity would add its rounding to every term, it is taken in
// the step; the time step has no viscous part),
// -c_i / 24 (= -|T| grad N_i / 4, the element's G(i, x)) to the three
// pressure-gradient sums and det to the lumped mass sum (scaled after the
// walk).  For the order (p, q, c) an odd permutation of the element's own, det
// and every cofactor change sign, w does not, so every contribution is
// multiplied by -1.  M = -c_c is carried from the previous step: after q
// leaves, the window (p, c) has d_p x d_c = -c_q; after p leaves, (q, c) has
// d_q x d_c = c_p.
template <int P, int MODE>
struct WalkNode {
  int k;  // slot (in rows of the group)
  V3<typename Prec<P>::T> d, v;
  typename Slots<P, MODE>::V a;
};

template <int P, int RW, int MODE>
__device__ __forceinline__ void walk_lane(const uint8_t* __restrict__ st, int nbytes,
                                          const T4<typename Prec<P>::T>* nb0, const T2<typename Prec<P>::T>* nb1,
                                          Slots<P, MODE>& acc, const V3<typename Prec<P>::T>& u2i,
                                          typename Prec<P>::T kc, typename Prec<P>::T kmu, Acc<P>& detsum) {
  using T = typename Prec<P>::T;
  using Node = WalkNode<P, MODE>;
  constexpr T kg = T(-1.0 / 24.0);  // the pressure-gradient sums are accumulated scaled
  auto load = [&](unsigned w) {
    Node nd;
    nd.k = (int)(w & WALK_POS) * RW;
    const T4<T> x = nb0[nd.k];
    nd.d = V3<T>{x.x, x.y, x.z};
    if constexpr (MODE != NODAL) {
      const T2<T> y = nb1[nd.k];
      nd.v = V3<T>{x.w, y.x, y.y};
      nd.a = acc.load(nd.k);
    }
    return nd;
  };
  for (int s = 0; s < nbytes;) {
    // a segment: two filling bytes with the element count in their upper
    // bits, then one byte per element
    const unsigned f1 = st[s], f2 = st[s + 1];
    const int cnt = (int)((f1 >> 5) | ((f2 >> 5) << 3));
    const uint8_t* e = st + s + 2;
    s += 2 + cnt;
    Node p = load(f1), n0 = load(f2);
    V3<T> M{};
    bool flip = false;  // FP64: c_c is M, not -M
    if constexpr (MODE != NODAL) {
      M = cross_fma(n0.d, p.d);
      p.v = add(u2i, p.v);
    }
    unsigned w = e[0];
    Node n1 = load(w), n2;
    // The next step's node is loaded while this element is evaluated (never
    // one of p, q, c: the walk is encoded that way; the last step reloads its
    // own node, unused).
    auto step = [&](Node& q, Node& c, Node& nx, int i) {
      const unsigned wn = e[i + 1 < cnt ? i + 1 : i];
      nx = load(wn);
      const bool neg = (w & WALK_NEG) != 0u, evq = (w & WALK_EVQ) != 0u;
      const T f = neg ? T(-1) : T(1);
      const V3<T> cp = cross_fma(q.d, c.d);
      const T det = dot_fma(p.d, cp);
      if constexpr (P == NSI_MIXED_F32_ACC64) detsum.add(f * det);
      else detsum.v = fma(f, det, detsum.v);
      if constexpr (MODE != NODAL) {
        const V3<T> cq = cross_fma(c.d, p.d);
        V3<T> w3{p.v.x + q.v.x + c.v.x, p.v.y + q.v.y + c.v.y, p.v.z + q.v.z + c.v.z};
        if constexpr (MODE == ASSEMBLE) {
          V3<T> ci;
          if constexpr (P == NSI_FP64) {
            const T sg = flip ? T(-1) : T(1);
            ci = V3<T>{fma(sg, M.x, -(cp.x + cq.x)), fma(sg, M.y, -(cp.y + cq.y)), fma(sg, M.z, -(cp.z + cq.z))};
          } else {
            ci = V3<T>{M.x - (cp.x + cq.x), M.y - (cp.y + cq.y), M.z - (cp.z + cq.z)};
          }
          const T kv = mul_rn(kmu, rcp_fast(det));
          if constexpr (P == NSI_FP64)
            w3 = V3<T>{fma(kv, ci.x, w3.x), fma(kv, ci.y, w3.y), fma(kv, ci.z, w3.z)};
          else
            w3 = V3<T>{fma(kc, w3.x, mul_rn(kv, ci.x)), fma(kc, w3.y, mul_rn(kv, ci.y)), fma(kc, w3.z, mul_rn(kv, ci.z))};
          const T fg = neg ? -kg : kg;
          const T ap = dot_fma(w3, cp), aq = dot_fma(w3, cq), ac = dot_fma(w3, M);
          if constexpr (P == NSI_FP64) {
            auto upd = [&](typename Slots<P, MODE>::V& a, T fs, T v) {
              a.x.x = fma(fs, v, a.x.x);
              a.x.y = fma(fg, ci.x, a.x.y);
              a.y.x = fma(fg, ci.y, a.y.x);
              a.y.y = fma(fg, ci.z, a.y.y);
            };
            upd(p.a, f, ap);
            upd(q.a, f, aq);
            upd(c.a, neg != flip ? T(1) : T(-1), ac);
          } else {
            const float2 gg = make_float2(fg, fg), cxy = make_float2(ci.x, ci.y);
            auto upd = [&](typename Slots<P, MODE>::V& a, float fs, float v) {
              a.g = fma2(gg, cxy, a.g);
              a.r = fma2(make_float2(fg, fs), make_float2(ci.z, v), a.r);
            };
            upd(p.a, f, ap);
            upd(q.a, f, aq);
            upd(c.a, -f, ac);
          }
        } else {
          const T one = P == NSI_FP64 ? T(1) : kc, fk = neg ? -one : one;
          p.a = fma(fk, dot_fma(w3, cp), p.a);
          q.a = fma(fk, dot_fma(w3, cq), q.a);
          c.a = fma(neg != flip ? one : -one, dot_fma(w3, M), c.a);
        }
        if constexpr (P == NSI_FP64) {  // (a negated double is an operation of the FP64 pipe, its bound)
          M = V3<T>{evq ? cq.x : cp.x, evq ? cq.y : cp.y, evq ? cq.z : cp.z};
          flip = !evq;
        } else {
          M = V3<T>{evq ? cq.x : -cp.x, evq ? cq.y : -cp.y, evq ? cq.z : -cp.z};
        }
        if (evq) acc.store(q.k, q.a);
        else acc.store(p.k, p.a);
      }
      if (!evq) {
        p = q;
        if constexpr (MODE != NODAL) p.v = add(u2i, q.v);
      }
      w = wn;
    };
    // q, c and the node in flight rotate through n0, n1, n2: three steps per
    // iteration bring them back to their places, so the newest node never
    // moves between registers (only p's update depends on the walk)
    int i = 0;
    for (; i + 3 <= cnt; i += 3) {
      step(n0, n1, n2, i);
      step(n1, n2, n0, i + 1);
      step(n2, n0, n1, i + 2);
    }
    if (i < cnt) {
      step(n0, n1, n2, i);
      if (i + 1 < cnt) {
        step(n1, n2, n0, i + 1);
        acc.store(n2.k, n2.a);
      } else {
        acc.store(n1.k, n1.a);
      }
    } else {
      acc.store(n0.k, n0.a);
    }
    acc.store(p.k, p.a);
  }
}

// every byte of a row's sub-walks within the row's bytes and its slots (debug)
__device__ __forceinline__ bool walk_ok(const uint8_t* st, int nbytes, int nsub, int slots) {
  if (nbytes == 0) return true;
  if (nbytes < nsub) return false;
  int at = nsub;
  for (int k = 0; k < nsub; ++k) {
    const int end = at + st[k];
    if (end > nbytes) return false;
    while (at < end) {
      if (at + 2 >= end) return false;
      const int cnt = (st[at] >> 5) | ((st[at + 1] >> 5) << 3);
      if (cnt < 1 || at + 2 + cnt > end) return false;
      for (int b = 0; b < 2 + cnt; ++b)
        if ((int)(st[at + b] & WALK_POS) >= slots) return false;
      at += 2 + cnt;
    }
  }
  return at == nbytes;
}

// ---------------------------------------------------------------- groups ---
// One row of a group, as each of its lanes sees it.
struct GroupRow {
  int32_t rs, re;  // CSR bounds
  uint32_t w0, w1;  // walk bounds
  int dp;
};
// the bounds and diagonal positions of rows [r0, r0 + RW) into shared memory
// (rows past the mesh's end get its last bound)
template <int RW>
__device__ __forceinline__ void copy_rows(const WalkMesh& m, unsigned char* info, int64_t r0, int lane) {
  int32_t* b = reinterpret_cast<int32_t*>(info);
  for (int k = lane; k <= RW; k += 32) {
    const int64_t i = min(r0 + k, m.n);
    cp_async4(b + k, m.row_ptr + i);
    cp_async4(b + RW + 1 + k, m.walk_ptr + i);
  }
  if (lane < RW / 4) cp_async4(b + 2 * (RW + 1) + lane, m.diag_pos + r0 + 4 * lane);  // (padded past n)
}
template <int RW>
__device__ __forceinline__ GroupRow read_row(const unsigned char* info, int t) {
  const int32_t* b = reinterpret_cast<const int32_t*>(info);
  GroupRow r;
  r.rs = b[t];
  r.re = b[t + 1];
  r.w0 = (uint32_t)b[RW + 1 + t];
  r.w1 = (uint32_t)b[RW + 2 + t];
  r.dp = info[8 * (RW + 1) + t];
  return r;
}
// slots of a row: its off-diagonal entries (none for a long row, which
// rows64_kernel computes)
__device__ __forceinline__ int row_slots(const GroupRow& r) {
  return r.dp == DIAG_LONG ? 0 : max(0, r.re - r.rs - 1);
}
// row position of slot s (the diagonal has none)
__device__ __forceinline__ int slot_pos(int s, int dp) { return s + (s >= dp ? 1 : 0); }

// the walk bytes of the group's rows into shared memory, as aligned words
__device__ __forceinline__ void copy_walk(const WalkMesh& m, unsigned char* dst, uint32_t w0, uint32_t w1, int lane) {
  const uint32_t off = w0 & 3u;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(m.walk + (w0 - off));
  const int words = (int)((w1 - w0 + off + 3) >> 2);
  for (int k = lane; k < words; k += 32) cp_async4(reinterpret_cast<uint32_t*>(dst) + k, src + k);
}

template <int P>
__device__ __forceinline__ Acc<P> scaled(const Acc<P>& s, typename Prec<P>::T c) {
  Acc<P> r;
  if constexpr (P == NSI_MIXED_F32_ACC64) {
    const float p = __fmul_rn(s.hi, c);  // c * (hi + lo), product error kept
    r.hi = p;
    r.lo = fmaf(s.lo, c, fmaf(s.hi, c, -p));
  } else {
    r.v = s.v * c;
  }
  return r;
}
// a + (the same accumulator of the lane `off` away): the error terms first (a
// commutative sum), so that both lanes of a pair hold bitwise the same value
template <int P>
__device__ __forceinline__ void merge_lanes(Acc<P>& a, int off) {
  if constexpr (P == NSI_MIXED_F32_ACC64) {
    const float hi = __shfl_xor_sync(0xffffffffu, a.hi, off), lo = __shfl_xor_sync(0xffffffffu, a.lo, off);
    a.lo += lo;
    a.add(hi);
  } else {
    a.v += __shfl_xor_sync(0xffffffffu, a.v, off);
  }
}

// The group loop of one warp: groups g, g + stride, ... below g_end; `src`
// gives a group's mesh.  H lanes per row: lane = h * RW + t works on row t.
// The next group's row bounds are copied under the current walk, its walk
// bytes and column indices under the merge, and its records are loaded under
// the write-out.
// LONG: the mesh has groups whose entries, because of a long row among them, are
// more than the staging holds.  (Kernels of their own: the time step of a mesh
// without such groups took 88 us instead of 86.)
// DIRECT: the nodes' coordinates and velocities are read where they are (five
// loads a node) instead of from packed records (one), which saves a small mesh
// the packing launch; the values are the same.
template <int P, int H, int MODE, bool DEBUG, bool DIRECT, bool LONG, typename Source>
__device__ __forceinline__ void group_loop(const Source& src, int g, int stride, int g_end, unsigned char* smem,
                                           const GroupLay& lay) {
  using T = typename Prec<P>::T;
  using Out = typename Prec<P>::Out;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int RW = 32 / H;
  int lane = threadIdx.x & 31, t = lane & (RW - 1), h = lane / RW;
  if (g >= g_end) return;  // warp-uniform
  // The lane's place, made opaque between the phases of a group: otherwise the
  // compiler keeps every phase's addresses in registers over the whole loop.
  auto refresh = [&]() { asm volatile("" : "+r"(lane), "+r"(t), "+r"(h)); };
  auto nb0 = [&]() { return reinterpret_cast<T4<T>*>(smem) + t; };
  auto nb1 = [&]() { return reinterpret_cast<T2<T>*>(smem + lay.nb1) + t; };
  // one lane's accumulators
  auto slots = [&](int p) { return Slots<P, MODE>(smem + lay.acc + p * lay.plane, lay.N); };

  constexpr int UT = P == NSI_FP64 || H == 1 ? 4 : 16 / H;  // records of a lane in flight

  auto copy_cols = [&](const WalkMesh& m, int32_t c0, int32_t c1) {
    if (LONG && c1 - c0 > lay.L) return;  // read where they are
    for (int k = lane; k < c1 - c0; k += 32) cp_async4(reinterpret_cast<int32_t*>(smem + lay.cols) + k, m.col_idx + c0 + k);
  };
  // a row's record and its slots' s0, s0 + H, ... (UT per lane); STAGED: by the
  // column indices in shared memory, where the group's entries from c0 to c1 are
  // unless they are more than the staging holds
  struct Recs {
    NodeRec<P> me, r[UT];
  };
  auto load_recs = [&](Recs& v, const WalkItem<MODE>& of, const GroupRow& r, int32_t c0, int32_t c1, int64_t i, int s0,
                       bool staged) {
    const WalkMesh& m = of.m;
    const int ns = row_slots(r);
    const int32_t self = (int32_t)min(i, m.n - 1);
    auto load = [&](NodeRec<P>& to, int64_t j) {
      if constexpr (DIRECT) to.gather(m, of.f, j);
      else to.load(m.rec, j);
    };
    // (all columns first: the records' loads keep their place among each other)
    int32_t k[UT];
    auto columns = [&](const int32_t* col) {
#pragma unroll
      for (int c = 0; c < UT; ++c) {
        const int s = s0 + c * H;
        k[c] = s < ns ? col[slot_pos(s, r.dp)] : self;  // (past the row: its own, unused)
        if (DEBUG && (k[c] < 0 || k[c] >= m.n)) {
          atomicOr(m.err, ERR_BAD_INDEX);
          k[c] = self;
        }
      }
    };
    if (staged && (!LONG || c1 - c0 <= lay.L)) columns(reinterpret_cast<const int32_t*>(smem + lay.cols) + (r.rs - c0));
    else columns(m.col_idx + r.rs);
    if (s0 == h) load(v.me, self);
#pragma unroll
    for (int c = 0; c < UT; ++c) load(v.r[c], k[c]);
  };
  // the group's slots: edge vectors from the row's node, velocities, zeroed
  // sums; 2 u_i of the row's own node (FP64: all velocities times rho/120)
  V3<T> u2i;
  auto put = [&](Recs& v, const WalkItem<MODE>& of, const GroupRow& r, int64_t i) {
    const T kc = kc_of<T>(of.f);
    auto scale = [&](const V3<T>& u) {
      if constexpr (P == NSI_FP64) return V3<T>{mul_rn(kc, u.x), mul_rn(kc, u.y), mul_rn(kc, u.z)};
      else return u;
    };
    const V3<T> ui = scale(v.me.vel());
    u2i = add(ui, ui);
    const int ns = DEBUG ? min(row_slots(r), lay.W) : row_slots(r);
#pragma unroll 1
    for (int s0 = h; s0 < ns; s0 += UT * H) {
      if (s0 != h) load_recs(v, of, r, 0, 0, i, s0, false);
#pragma unroll
      for (int c = 0; c < UT; ++c) {
        if (s0 + c * H >= ns) break;
        const int k = (s0 + c * H) * RW;
        const V3<T> d = v.r[c].minus(v.me);
        if constexpr (MODE == NODAL) {
          nb0()[k] = T4<T>{d.x, d.y, d.z, T(0)};
        } else {
          const V3<T> u = scale(v.r[c].vel());
          nb0()[k] = T4<T>{d.x, d.y, d.z, u.x};
          nb1()[k] = T2<T>{u.y, u.z};
        }
      }
    }
    if constexpr (MODE != NODAL)
      for (int b = 16 * lane; b < H * lay.plane; b += 16 * 32)
        *reinterpret_cast<float4*>(smem + lay.acc + b) = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
  };
  // the first group
  int at = src.find(g);
  GroupRow row;
  int32_t base, end;
  uint32_t wb, we;
  {
    const WalkMesh& m = src.item(at).m;
    const int64_t r0 = (int64_t)(g - src.item(at).group0) * RW;
    copy_rows<RW>(m, smem + lay.info, r0, lane);
    cp_async_wait_all();
    __syncwarp();
    row = read_row<RW>(smem + lay.info, t);
    base = __shfl_sync(FULL, row.rs, 0), end = __shfl_sync(FULL, row.re, RW - 1);
    wb = __shfl_sync(FULL, row.w0, 0), we = __shfl_sync(FULL, row.w1, RW - 1);
    if (!DEBUG || we - wb <= (uint32_t)lay.S) copy_walk(m, smem + lay.walk, wb, we, lane);
    copy_cols(m, base, end);
    cp_async_wait_all();
    __syncwarp();
    Recs v;
    if constexpr (!DIRECT) wait_for_previous();
    load_recs(v, src.item(at), row, base, end, r0 + t, h, true);
    __syncwarp();
    put(v, src.item(at), row, r0 + t);
  }
  while (true) {
    const WalkMesh& m = src.item(at).m;
    const FieldView& f = src.item(at).f;
    const WalkOut<MODE>& o = src.item(at).o;
    const int64_t i = (int64_t)(g - src.item(at).group0) * RW + t;
    const bool valid = i < m.n;
    const int ns = row_slots(row);
    // The group's entries are staged as they lie in memory; where a long row
    // (hundreds of entries, which rows64_kernel computes) makes them more than
    // the staging holds, every other row in a place of its own.  gb: the row's
    // first entry in the group's slice, lb: in the staging.
    const bool dense = !LONG || end - base <= lay.L;  // warp-uniform
    const int Ld = dense ? end - base : 0, gb = row.rs - base;
    const int lb = dense ? gb : t * (lay.W + 1);
    bool fits = true;
    if (DEBUG) {
      fits = we - wb <= (uint32_t)lay.S && !__any_sync(FULL, ns > lay.W || (ns > 0 && row.dp > ns));
      if (!fits && lane == 0) atomicOr(m.err, ERR_STAR);
    }
    const T kmass = kmass_of<T>(f);
    refresh();

    // the next group's row bounds, in flight during the walk
    const int gn = g + stride;
    const bool more = gn < g_end;  // warp-uniform
    const int atn = more ? src.find(gn) : at;
    if (more) copy_rows<RW>(src.item(atn).m, smem + lay.info, (int64_t)(gn - src.item(atn).group0) * RW, lane);

    // 1. the row's sub-walk h
    refresh();
    Acc<P> detsum;
    detsum.zero();
    if (fits && ns > 0) {
      Slots<P, MODE> acc = slots(h);
      if constexpr (MODE == ASSEMBLE && P == NSI_FP64) {
        acc.a0 += t;
        acc.a1 += t;
      } else if constexpr (MODE != NODAL) {
        acc.a += t;
      }
      const uint8_t* st = (smem + lay.walk) + (row.w0 - wb) + (wb & 3u);
      const int nb = (int)(row.w1 - row.w0);
      if (DEBUG && !walk_ok(st, nb, H, ns)) {
        atomicOr(m.err, ERR_STAR);
      } else if (nb > 0) {
        // (each lane finds its bytes first: the row's lanes walk together)
        int b = H;
        for (int k = 0; k < h; ++k) b += st[k];
        walk_lane<P, RW, MODE>(st + b, st[h], nb0(), nb1(), acc, u2i, kc_of<T>(f), kmu_of<T>(f), detsum);
      }
    }
    __syncwarp();

    // the next group's walk bytes and column indices
    refresh();
    GroupRow rown = row;
    int32_t basen = 0, endn = 0;
    uint32_t wbn = 0, wen = 0;
    if (more) {
      cp_async_wait_all();
      __syncwarp();
      const WalkMesh& mn = src.item(atn).m;
      rown = read_row<RW>(smem + lay.info, t);
      basen = __shfl_sync(FULL, rown.rs, 0), endn = __shfl_sync(FULL, rown.re, RW - 1);
      wbn = __shfl_sync(FULL, rown.w0, 0), wen = __shfl_sync(FULL, rown.w1, RW - 1);
      if (!DEBUG || wen - wbn <= (uint32_t)lay.S) copy_walk(mn, smem + lay.walk, wbn, wen, lane);
      copy_cols(mn, basen, endn);
    }
    V3<T> un{T(0), T(0), T(0)};
    if (valid) un = load_vec<T>(f.un, i);
    // the time step's A_static: the lane's first entries and the diagonal,
    // read before the slice is written (A may be A_static)
    constexpr int NS = 8;
    [[maybe_unused]] Out as[NS], sd = Out(0);
    if constexpr (MODE == STEP) {
      const Out* As = static_cast<const Out*>(o.A_static) + base;
#pragma unroll
      for (int c = 0; c < NS; ++c)
        if (lane + 32 * c < Ld) as[c] = As[lane + 32 * c];
      if (h == 0 && ns > 0) sd = As[gb + row.dp];
    }
#pragma unroll
    for (int off = RW; off < 32; off <<= 1) merge_lanes<P>(detsum, off);

    // 2. the lanes' sums merged, the diagonal from the partition of unity
    // (sum_b grad N_b = 0):
    //   A(i,i) = lumped mass - sum_{j != i} A(i,j)   (convection + viscous parts)
    //   G(i,i) = 1/3 sum_{j != i} G(i,j)             (each element adds c_i to three
    //                                                 off-diagonal entries and the diagonal)
    // and the row moved into CSR order for the write-out (over the slots' edge
    // vectors and velocities, which are no longer needed)
    [[maybe_unused]] float dlo = 0.f;  // mixed64: the error term of the diagonal's leading part dhi
    [[maybe_unused]] float dhi = 0.f;
    const int len = !fits || row.dp == DIAG_LONG ? 0 : row.re - row.rs;
    const int zl = fits && dense && row.dp == DIAG_LONG ? row.re - row.rs : 0;  // a long row's entries in the staging
    // the lane's slots, in pairs from both ends of the row: in a natural node
    // order these lie on opposite sides of the node and their G cancel, so the
    // lanes' sums stay small (rms error of G(i,i) in float of a 36^3 box 1.6e-7 of
    // its size; every second slot to one lane 2.5e-7, one lane's slots in order
    // 2.1e-7).  Mixed64's time step has one sum, and that compensated.
    auto each_slot = [&](auto&& use) {
      int s = h, last = fits ? ns - 1 : -1;
      if constexpr (H > 1 && !(MODE == STEP && P == NSI_MIXED_F32_ACC64)) {
        const int paired = (last + 1) / (2 * H) * H;
        for (; s < paired; s += H) {
          use(s);
          use(last - s);
        }
        last -= paired;
      }
#pragma unroll 2
      for (; s <= last; s += H) use(s);
    };
    if constexpr (MODE == ASSEMBLE) {
      using S = Slots<P, ASSEMBLE>;
      Acc<P> ra;
      ra.zero();
      T4<T>* stage = reinterpret_cast<T4<T>*>(smem);
      // the planes' sums of the lane's slots and their entries
      auto each = [&](auto&& use) {
        each_slot([&](int s) {
          typename S::V v = slots(0).load(s * RW + t);
#pragma unroll
          for (int p = 1; p < H; ++p) v = S::sum(v, slots(p).load(s * RW + t));
          use(v, lb + slot_pos(s, row.dp));
        });
      };
      if constexpr (P == NSI_FP64) {
        double gx = 0.0, gy = 0.0, gz = 0.0;
        each([&](const typename S::V& v, int e) {
          ra.add(v.x.x);
          gx += v.x.y;
          gy += v.y.x;
          gz += v.y.y;
          stage[e] = T4<T>{v.x.x, v.x.y, v.y.x, v.y.y};
        });
#pragma unroll
        for (int off = RW; off < 32; off <<= 1) {
          merge_lanes<P>(ra, off);
          gx += __shfl_xor_sync(FULL, gx, off);
          gy += __shfl_xor_sync(FULL, gy, off);
          gz += __shfl_xor_sync(FULL, gz, off);
        }
        if (h == 0 && len > 0)
          stage[lb + row.dp] = T4<T>{fma(kmass, detsum.v, -ra.v), gx * (1.0 / 3.0), gy * (1.0 / 3.0), gz * (1.0 / 3.0)};
      } else {
        float2 g = make_float2(0.f, 0.f);
        float gz = 0.f;
        each([&](const typename S::V& v, int e) {
          ra.add(v.r.y);
          g = add2(g, v.g);
          gz += v.r.x;
          stage[e] = T4<T>{v.r.y, v.g.x, v.g.y, v.r.x};
        });
#pragma unroll
        for (int off = RW; off < 32; off <<= 1) {
          merge_lanes<P>(ra, off);
          g.x += __shfl_xor_sync(FULL, g.x, off);
          g.y += __shfl_xor_sync(FULL, g.y, off);
          gz += __shfl_xor_sync(FULL, gz, off);
        }
        float ad;
        if constexpr (P == NSI_MIXED_F32_ACC64) {
          Acc<P> d = scaled<P>(detsum, kmass);
          d.add(-ra.hi);
          d.lo -= ra.lo;
          dhi = ad = d.hi;
          dlo = d.lo;
        } else {
          ad = fmaf(kmass, detsum.v, -ra.v);
        }
        if (h == 0 && len > 0)
          stage[lb + row.dp] = T4<T>{ad, g.x * (1.0f / 3.0f), g.y * (1.0f / 3.0f), gz * (1.0f / 3.0f)};
      }
      for (int q = h; q < zl; q += H) stage[lb + q] = T4<T>{T(0), T(0), T(0), T(0)};  // a long row, computed later
    } else if constexpr (MODE == STEP) {
      using S = Slots<P, STEP>;
      Acc<P> ra;
      ra.zero();
      T* stage = reinterpret_cast<T*>(smem);
      each_slot([&](int s) {
        const int k = s * RW + t;
        T v = slots(0).load(k);
#pragma unroll
        for (int p = 1; p < H; ++p) v += slots(p).load(k);
        ra.add(v);
        stage[lb + slot_pos(s, row.dp)] = v;
      });
#pragma unroll
      for (int off = RW; off < 32; off <<= 1) merge_lanes<P>(ra, off);
      T ad;
      if constexpr (P == NSI_MIXED_F32_ACC64) {
        dhi = ad = -ra.hi;
        dlo = -ra.lo;
      } else {
        ad = -ra.v;
      }
      if (h == 0 && len > 0) stage[lb + row.dp] = ad;
      for (int q = h; q < zl; q += H) stage[lb + q] = T(0);  // a long row: A_static kept, C added later
    }
    // lumped RHS: (sum_e rho |T_e| / (4 dt)) u^n_i, spread over the row's lanes
    if (valid) {
      Out* Rh = static_cast<Out*>(o.rhs);
      const T unk[3] = {mul_rn(kmass, un.x), mul_rn(kmass, un.y), mul_rn(kmass, un.z)};
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k % H == h) store_acc(Rh + k * m.n + i, scaled<P>(detsum, unk[k]));
      if constexpr (MODE == NODAL) {
        if (h == 0) store_acc(static_cast<Out*>(o.dt_rho) + i, scaled<P>(detsum, kmass));
        if (h == H - 1) {
          T kmr;
          if constexpr (sizeof(T) == 8) kmr = o.kmr;
          else kmr = o.kmrf;
          store_acc(static_cast<Out*>(o.mass_rho) + i, scaled<P>(detsum, kmr));
        }
      }
    }
    cp_async_wait_all();
    __syncwarp();
    // the next group's records, in flight during the write-out
    Recs v{};
    if (more) {
      load_recs(v, src.item(atn), rown, basen, endn, (int64_t)(gn - src.item(atn).group0) * RW + t, h, true);
    }

    // 3. the group's contiguous slice of the outputs
    refresh();
    if constexpr (MODE == ASSEMBLE) {
      const T4<T>* stage = reinterpret_cast<const T4<T>*>(smem);
      Out* A = static_cast<Out*>(o.A) + base;
      Out *G = static_cast<Out*>(o.G) + base, *G1 = G + m.nnz, *G2 = G1 + m.nnz;
      // (plain stores: streaming ones took mixed64 275 against 270 us at 100^3 in
      // random order and 232 against 221 in natural, mixed32 236 against 226)
      auto write = [&](auto&& put) {
#pragma unroll 1
        for (int r = 0; r < (dense ? 1 : RW); ++r) {
          int n = fits ? Ld : 0, to = 0, from = 0;
          if (!dense) n = __shfl_sync(FULL, len, r), to = __shfl_sync(FULL, gb, r), from = r * (lay.W + 1);
#pragma unroll 1
          for (int k = lane; k < n; k += 32) put(to + k, stage[from + k]);
        }
      };
      if constexpr (P == NSI_MIXED_F32_ACC64) {
        // converted to double exactly, A by the FP64 pipe's conversion and G from
        // the bits (all four either way cost 2% more: the pipe's rate, or the
        // instructions), then every diagonal by the double nearest its
        // compensated pair
        write([&](int k, const T4<T>& v) {
          A[k] = (double)v.x;
          G[k] = float_double(v.y);
          G1[k] = float_double(v.z);
          G2[k] = float_double(v.w);
        });
        __syncwarp();
        if (fits && h == 0 && len > 0)
          A[gb + row.dp] = nonfinite_bits(dhi) ? nonfinite_double(dhi) : pair_double(dhi, dlo);
      } else {
        write([&](int k, const T4<T>& v) {
          A[k] = v.x;
          G[k] = v.y;
          G1[k] = v.z;
          G2[k] = v.w;
        });
      }
    } else if constexpr (MODE == STEP) {
      const T* stage = reinterpret_cast<const T*>(smem);
      const Out* As = static_cast<const Out*>(o.A_static) + base;
      Out* A = static_cast<Out*>(o.A) + base;
      // C(u) of entry k in the output type (mixed64: by the FP64 pipe's
      // conversion, 80.5 us for an 81x70x66 time step against 87.7 from the bits)
      auto value = [&](int k) { return (Out)stage[k]; };
      if (fits) {
#pragma unroll
        for (int c = 0; c < NS; ++c)
          if (lane + 32 * c < Ld) A[lane + 32 * c] = as[c] + value(lane + 32 * c);
        for (int k = lane + 32 * NS; k < Ld; k += 32) A[k] = As[k] + value(k);
      }
      if (fits && !dense) {  // (a row has no more entries than the warp has lanes)
#pragma unroll 1
        for (int r = 0; r < RW; ++r) {
          const int n = __shfl_sync(FULL, len, r), k = __shfl_sync(FULL, gb, r) + lane;
          if (lane < n) A[k] = As[k] + value(r * (lay.W + 1) + lane);
        }
      }
      if constexpr (P == NSI_MIXED_F32_ACC64) {  // the diagonal's sum is a compensated pair
        __syncwarp();
        if (fits && h == 0 && ns > 0)
          A[gb + row.dp] = sd + (nonfinite_bits(dhi) ? nonfinite_double(dhi) : pair_double(dhi, dlo));
      }
    }
    if (!more) return;
    __syncwarp();  // the next group reuses the staging
    refresh();
    put(v, src.item(atn), rown, (int64_t)(gn - src.item(atn).group0) * RW + t);
    g = gn;
    at = atn;
    row = rown;
    wb = wbn;
    we = wen;
    base = basen;
    end = endn;
  }
}


// where a group's mesh comes from: the one mesh of a launch, or a batch's
template <int MODE>
struct OneMesh {
  const WalkItem<MODE>& one;
  __device__ __forceinline__ int find(int) const { return 0; }
  __device__ __forceinline__ const WalkItem<MODE>& item(int) const { return one; }
};

template <int P, int H, int MODE, bool DEBUG, bool LONG>
__global__ void __launch_bounds__(32 * MAX_WARPS, P == NSI_FP64 ? 2 : 4)
    gather_persistent_kernel(const __grid_constant__ WalkItem<MODE> item, GroupLay lay, int g0, int g_end) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int warps = blockDim.x >> 5, w = threadIdx.x >> 5;
  group_loop<P, H, MODE, DEBUG, H == 4, LONG>(OneMesh<MODE>{item}, g0 + (int)blockIdx.x * warps + w,
                                              (int)gridDim.x * warps, g_end, smem_raw + w * lay.total, lay);
}

// ------------------------------------------------ badly shaped elements ---
// Rows listed at create (mixed modes: the rows of the nodes of an element with
// |d1||d2||d3| > EXACT_RATIO |det|) are recomputed after the assembly in double
// from the handle's coordinates (leading + residual float parts) and the given
// velocities, and their entries overwritten: a float determinant of such an
// element would carry about that ratio times the float rounding of its edge
// vectors.  The lanes of a warp walk 32 / H listed rows as in the group loop
// (the walk bytes read from memory, the entries written row by row): the FP64
// pipe, the bound here, issues a warp's instruction at the same cost whether or
// not its lanes are active, so rows side by side fill it best (a 14x40x70 pipe,
// 14,905 of its 39,831 rows listed: 66 us, of which the pipe is busy 45).
// MODE 0: A, G and rhs; 1: rhs only (the time
// step: the convection does not involve the determinant); 2: rhs, dt_rho and
// mass_rho.
template <int P, int H, int MODE>
__global__ void __launch_bounds__(32) exact_rows_kernel(WalkMesh m, FieldView f, RowOut o, GroupLay lay,
                                                        const int32_t* __restrict__ rows, int64_t count) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using Out = typename Prec<P>::Out;
  constexpr int RW = 32 / H, WMODE = MODE == 0 ? ASSEMBLE : NODAL;
  using S = Slots<NSI_FP64, WMODE>;
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, t = lane & (RW - 1), h = lane / RW;
  const int64_t r = (int64_t)blockIdx.x * RW + t;
  unsigned char* smem = smem_raw;
  const bool valid = r < count;
  const int64_t i = valid ? rows[r] : 0;
  const int32_t rs = m.row_ptr[i];
  const int ns = valid ? m.row_ptr[i + 1] - rs - 1 : 0, dp = m.diag_pos[i];
  auto coord = [&](int64_t j) {
    const float4 a = __ldg(m.xyz_hi + j), b = __ldg(m.xyz_lo + j);
    return V3<double>{(double)a.x + (double)b.x, (double)a.y + (double)b.y, (double)a.z + (double)b.z};
  };
  auto slots = [&](int p) { return S(smem + lay.acc + p * lay.plane, lay.N); };
  T4<double>* nb0 = reinterpret_cast<T4<double>*>(smem) + t;
  T2<double>* nb1 = reinterpret_cast<T2<double>*>(smem + lay.nb1) + t;
  const V3<double> xi = coord(i);
  V3<double> u2i{0.0, 0.0, 0.0};
  if constexpr (MODE == 0) {
    const V3<float> ui = load_vec<float>(f.u, i);
    u2i = V3<double>{2.0 * f.kc * ui.x, 2.0 * f.kc * ui.y, 2.0 * f.kc * ui.z};
  }
  for (int s = h; s < ns; s += H) {
    const int64_t j = m.col_idx[rs + slot_pos(s, dp)];
    const V3<double> d = sub(coord(j), xi);
    if constexpr (MODE == 0) {
      const V3<float> u = load_vec<float>(f.u, j);
      nb0[s * RW] = T4<double>{d.x, d.y, d.z, f.kc * u.x};
      nb1[s * RW] = T2<double>{f.kc * u.y, f.kc * u.z};
      for (int p = 0; p < H; ++p) slots(p).store(s * RW + t, S::zero_value());
    } else {
      nb0[s * RW] = T4<double>{d.x, d.y, d.z, 0.0};
    }
  }
  __syncwarp();
  Acc<NSI_FP64> det;
  det.zero();
  if (ns > 0) {
    const uint8_t* st = m.walk + m.walk_ptr[i];
    int b = H;
    for (int k = 0; k < h; ++k) b += st[k];
    S acc = slots(h);
    if constexpr (MODE == 0) {
      acc.a0 += t;
      acc.a1 += t;
    }
    walk_lane<NSI_FP64, RW, WMODE>(st + b, st[h], nb0, nb1, acc, u2i, f.kc, f.kmu, det);
  }
  __syncwarp();
  wait_for_previous();  // (the rows' first values come from an earlier launch)
#pragma unroll
  for (int off = RW; off < 32; off <<= 1) det.v += __shfl_xor_sync(FULL, det.v, off);
  if constexpr (MODE == 0) {
    Out* A = static_cast<Out*>(o.A) + rs;
    Out* G = static_cast<Out*>(o.G) + rs;
    double ra = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    for (int s = h; s < ns; s += H) {
      typename S::V v = slots(0).load(s * RW + t);
#pragma unroll
      for (int p = 1; p < H; ++p) v = S::sum(v, slots(p).load(s * RW + t));
      ra += v.x.x;
      gx += v.x.y;
      gy += v.y.x;
      gz += v.y.y;
      const int q = slot_pos(s, dp);
      A[q] = (Out)v.x.x;
      G[q] = (Out)v.x.y;
      G[m.nnz + q] = (Out)v.y.x;
      G[2 * m.nnz + q] = (Out)v.y.y;
    }
#pragma unroll
    for (int off = RW; off < 32; off <<= 1) {
      ra += __shfl_xor_sync(FULL, ra, off);
      gx += __shfl_xor_sync(FULL, gx, off);
      gy += __shfl_xor_sync(FULL, gy, off);
      gz += __shfl_xor_sync(FULL, gz, off);
    }
    if (h == 0 && ns > 0) {  // the diagonal from the partition of unity, as in the group loop
      A[dp] = (Out)(f.kmass * det.v - ra);
      G[dp] = (Out)(gx / 3.0);
      G[m.nnz + dp] = (Out)(gy / 3.0);
      G[2 * m.nnz + dp] = (Out)(gz / 3.0);
    }
  }
  if (valid && h == 0) {
    const V3<float> un = load_vec<float>(f.un, i);
    const double mass = f.kmass * det.v;
    Out* Rh = static_cast<Out*>(o.rhs);
    Rh[i] = (Out)(mass * un.x);
    Rh[m.n + i] = (Out)(mass * un.y);
    Rh[2 * m.n + i] = (Out)(mass * un.z);
    if constexpr (MODE == 2) {
      static_cast<Out*>(o.dt_rho)[i] = (Out)mass;
      static_cast<Out*>(o.mass_rho)[i] = (Out)(o.kmr * det.v);
    }
  }
}

// ------------------------------------------------------ batched kernel ---
// The meshes with one lane per row first, then those with two, then those with
// four: a warp takes its share of the first's groups, then of the next's, so
// that every mesh is assembled as by its own launch.
constexpr int KINDS = 3;
__host__ __device__ constexpr int kind_lanes(int kind) { return 1 << kind; }
struct BatchArgs {
  int32_t count[KINDS];  // meshes
  int32_t total[KINDS];  // row groups
  WalkItem<ASSEMBLE> item[NSI_MAX_BATCH];
};
struct BatchLays {
  GroupLay kind[KINDS];
  int stride;  // bytes of a warp's shared memory
};
static_assert(sizeof(BatchArgs) + sizeof(BatchLays) <= 32764, "kernel parameters");

struct BatchMesh {
  const BatchArgs& args;
  int first, count;
  // the mesh of group g: the last item with group0 <= g
  __device__ __forceinline__ int find(int g) const {
    int lo = first, hi = first + count - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (args.item[mid].group0 <= g) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  }
  __device__ __forceinline__ const WalkItem<ASSEMBLE>& item(int k) const { return args.item[k]; }
};

template <int P, bool LONG>
__global__ void __launch_bounds__(32 * MAX_WARPS, P == NSI_FP64 ? 2 : 4)
    batched_kernel(const __grid_constant__ BatchArgs args, const __grid_constant__ BatchLays lays) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int warps = blockDim.x >> 5, w = threadIdx.x >> 5;
  const int all = (int)gridDim.x * warps;
  unsigned char* smem = smem_raw + w * lays.stride;
  int me = (int)blockIdx.x * warps + w;
  // (the warps with one group less of a kind begin the next kind's)
  auto next = [&](int kind) {
    __syncwarp();
    me -= args.total[kind] % all;
    if (me < 0) me += all;
  };
  if constexpr (P == NSI_FP64) {
    group_loop<P, 1, ASSEMBLE, false, false, LONG>(BatchMesh{args, 0, args.count[0]}, me, all, args.total[0], smem,
                                             lays.kind[0]);
    next(0);
  }
  group_loop<P, 2, ASSEMBLE, false, false, LONG>(BatchMesh{args, args.count[0], args.count[1]}, me, all, args.total[1], smem,
                                           lays.kind[1]);
  next(1);
  group_loop<P, 4, ASSEMBLE, false, false, LONG>(BatchMesh{args, args.count[0] + args.count[1], args.count[2]}, me, all,
                                           args.total[2], smem, lays.kind[2]);
}

template <int P>
__global__ void __launch_bounds__(256) pack_kernel(WalkMesh m, FieldView f) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < m.n) pack_node<P>(m, f, m.rec, i);
}

// the node records of every mesh of a batch in one launch: a block packs the
// 128 rows of consecutive groups of one kind
template <int P>
__global__ void __launch_bounds__(128) batched_pack_kernel(const __grid_constant__ BatchArgs args) {
  int block = (int)blockIdx.x, kind = 0, first = 0;
  for (; kind < KINDS - 1; ++kind) {
    const int groups = 4 * kind_lanes(kind), blocks = (args.total[kind] + groups - 1) / groups;
    if (block < blocks) break;
    block -= blocks;
    first += args.count[kind];
  }
  const int rw = 32 / kind_lanes(kind);
  const int g = block * (128 / rw) + (int)threadIdx.x / rw;
  if (g >= args.total[kind]) return;
  const BatchMesh src{args, first, args.count[kind]};
  const WalkItem<ASSEMBLE>& it = src.item(src.find(g));
  const int64_t i = (int64_t)(g - it.group0) * rw + threadIdx.x % rw;
  if (i < it.m.n) pack_node<P>(it.m, it.f, it.m.rec, i);
}

// ----------------------------------------------------------- launchers ---
WalkMesh walk_mesh(const NsiHandle* h, void* rec) {
  WalkMesh m;
  m.n = h->n;
  m.nnz = h->nnz;
  m.row_ptr = h->row_ptr;
  m.col_idx = h->col_idx;
  m.walk_ptr = h->walk_ptr;
  m.walk = h->walk;
  m.diag_pos = h->diag_pos;
  m.xyz64 = h->xyz64;
  m.xyz_hi = h->xyz_hi;
  m.xyz_lo = h->xyz_lo;
  m.rec = rec ? rec : h->rec;
  m.err = h->err;
  return m;
}

template <typename K>
nsi_status allow_smem(K kernel, std::once_flag& once, cudaError_t& err) {
  std::call_once(once, [&] { err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX); });
  return err == cudaSuccess ? NSI_OK : cuda_fail(err, "cudaFuncSetAttribute(row gather)");
}

// blocks of a persistent launch: as many as are resident at once, no more
// than the groups need.  `resident` keeps the first number for a launch shape
// (0: not asked for yet; the device's answer takes longer than a small launch).
template <typename K>
nsi_status resident_grid(K kernel, int warps, size_t smem, int64_t groups, std::atomic<int>* resident, int64_t* grid) {
  int at_once = resident ? resident->load(std::memory_order_relaxed) : 0;
  if (at_once == 0) {
    int per_sm = 0, sms = 0, dev = 0;
    NSI_CUDA(cudaGetDevice(&dev));
    NSI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    NSI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * warps, smem));
    at_once = std::max(1, per_sm) * sms;
    if (resident) resident->store(at_once, std::memory_order_relaxed);
  }
  *grid = std::max<int64_t>(1, std::min<int64_t>((groups + warps - 1) / warps, at_once));
  return NSI_OK;
}

template <int P, int H, int MODE, bool DEBUG, bool LONG>
nsi_status run_groups(NsiHandle* h, const WalkItem<MODE>& item, int64_t row0, int64_t row1, cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  const auto kernel = gather_persistent_kernel<P, H, MODE, DEBUG, LONG>;
  nsi_status st = allow_smem(kernel, once, err);
  if (st) return st;
  constexpr int RW = 32 / H;
  const GatherPlan& pl = h->plan;
  const GatherSmem lay = gather_smem(P, MODE, H, pl.w, pl.max_block_steps);
  const size_t smem = lay.total() * pl.warps;
  const int64_t g0 = row0 / RW, g1 = (row1 + RW - 1) / RW;
  int64_t grid = 0;
  if ((st = resident_grid(kernel, pl.warps, smem, g1 - g0, &h->resident[MODE][pl.warps - 1], &grid))) return st;
  if (h->ev_start) NSI_CUDA(cudaEventRecord(h->ev_start, s));
  if constexpr (H == 4)
    kernel<<<grid, 32 * pl.warps, smem, s>>>(item, GroupLay(lay), (int)g0, (int)g1);
  else
    NSI_CUDA(launch_early(kernel, grid, 32 * pl.warps, smem, s, item, GroupLay(lay), (int)g0, (int)g1));
  if (h->ev_stop) NSI_CUDA(cudaEventRecord(h->ev_stop, s));
  return check_launch("gather_persistent_kernel");
}

template <int P, int H, int MODE>
nsi_status run_rows(NsiHandle* h, const WalkItem<MODE>& item, int64_t row0, int64_t row1, cudaStream_t s) {
  return h->debug             ? run_groups<P, H, MODE, true, true>(h, item, row0, row1, s)
         : h->plan.long_group ? run_groups<P, H, MODE, false, true>(h, item, row0, row1, s)
                              : run_groups<P, H, MODE, false, false>(h, item, row0, row1, s);
}

template <int P, int MODE>
nsi_status run_lanes(NsiHandle* h, const WalkItem<MODE>& item, int64_t row0, int64_t row1, cudaStream_t s) {
  switch (h->nsub) {
    case 1:
      if constexpr (P == NSI_FP64) return run_rows<P, 1, MODE>(h, item, row0, row1, s);
      return fail(NSI_ERR_UNSUPPORTED, "one lane per row in FP64 only");
    case 2: return run_rows<P, 2, MODE>(h, item, row0, row1, s);
    default: return run_rows<P, 4, MODE>(h, item, row0, row1, s);
  }
}

template <int P, int H>
nsi_status exact_rows_h(NsiHandle* h, const FieldView& f, int mode, const RowOut& o, cudaStream_t s) {
  const auto kernel = mode == 0   ? exact_rows_kernel<P, H, 0>
                      : mode == 1 ? exact_rows_kernel<P, H, 1>
                                  : exact_rows_kernel<P, H, 2>;
  static std::once_flag once[3];
  static cudaError_t err[3] = {};
  nsi_status st = allow_smem(kernel, once[mode], err[mode]);
  if (st) return st;
  const int64_t warps = (h->exact_rows * H + 31) / 32;
  const GatherSmem lay = gather_smem(NSI_FP64, mode == 0 ? ASSEMBLE : NODAL, H, h->exact_slots, 0);
  NSI_CUDA(launch_early(kernel, warps, 32, lay.total(), s, walk_mesh(h, nullptr), f, o, GroupLay(lay),
                        (const int32_t*)h->exact_list, h->exact_rows));
  return check_launch("exact_rows_kernel");
}

}  // namespace

template <int P>
nsi_status launch_pack(NsiHandle* h, const FieldView& f, void* rec, cudaStream_t s) {
  pack_kernel<P><<<(h->n + 255) / 256, 256, 0, s>>>(walk_mesh(h, rec), f);
  return check_launch("pack_kernel");
}

template <int P>
nsi_status launch_gather(NsiHandle* h, const FieldView& f, const OutView& o, int64_t row0, int64_t row1, void* rec,
                         cudaStream_t s) {
  const WalkItem<ASSEMBLE> item{walk_mesh(h, rec), f, {o.A, o.G, o.rhs}, 0};
  return run_lanes<P, ASSEMBLE>(h, item, row0, row1, s);
}

template <int P>
nsi_status launch_step(NsiHandle* h, const FieldView& f, const StepView& o, bool nodal, cudaStream_t s) {
  if (nodal) {
    const WalkItem<NODAL> item{walk_mesh(h, nullptr), f, {o.rhs, o.dt_rho, o.mass_rho, o.kmr, o.kmrf}, 0};
    return run_lanes<P, NODAL>(h, item, 0, h->n, s);
  }
  const WalkItem<STEP> item{walk_mesh(h, nullptr), f, {o.A, o.rhs, o.A_static}, 0};
  return run_lanes<P, STEP>(h, item, 0, h->n, s);
}

template <int P>
nsi_status launch_batched(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int count,
                          cudaStream_t s) {
  static BatchArgs args;  // host staging of the by-value kernel argument
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  int warps = MAX_WARPS, item = 0;
  int64_t all = 0, pack_blocks = 0;
  size_t bytes = 0;
  BatchLays lays;
  bool long_group = false;
  for (int kind = 0; kind < KINDS; ++kind) {
    const int H = kind_lanes(kind), rw = 32 / H;
    int W = group_slots(P, H, 1), S = 0;
    int64_t groups = 0;
    args.count[kind] = 0;
    for (int k = 0; k < count; ++k) {
      const NsiHandle* h = hs[k];
      if (h->nsub != H) continue;
      const GatherPlan& pl = h->plan;
      warps = std::min(warps, pl.warps);
      long_group |= pl.long_group;
      W = std::max(W, pl.w);
      S = std::max(S, pl.max_block_steps);
      args.item[item++] = WalkItem<ASSEMBLE>{walk_mesh(h, nullptr), fields_of(&fs[k]),
                                             {os[k].A_val, os[k].G_val, os[k].rhs}, (int)groups};
      ++args.count[kind];
      groups += (h->n + rw - 1) / rw;
      if (groups > INT32_MAX / 2) return fail(NSI_ERR_UNSUPPORTED, "too many rows in a batch");
    }
    args.total[kind] = (int)groups;
    all += groups;
    pack_blocks += (groups + 4 * H - 1) / (4 * H);
    const GatherSmem lay = gather_smem(P, ASSEMBLE, H, W, S);
    if (!lay.group_fits())  // (each mesh's fits, and so do the maxima of W and L)
      return fail(NSI_ERR_UNSUPPORTED, "batched meshes need more shared memory than a group has");
    if (args.count[kind]) bytes = std::max(bytes, lay.total());
    lays.kind[kind] = GroupLay(lay);
  }
  if (all == 0) return NSI_OK;
  while (warps > 1 && bytes * warps > SMEM_MAX) --warps;
  if (bytes > SMEM_MAX) return fail(NSI_ERR_UNSUPPORTED, "batched meshes need more shared memory than a block has");
  lays.stride = (int)bytes;
  const auto kernel = long_group ? batched_kernel<P, true> : batched_kernel<P, false>;
  static std::once_flag once[2];
  static cudaError_t err[2] = {};
  nsi_status st = allow_smem(kernel, once[long_group], err[long_group]);
  if (st) return st;
  batched_pack_kernel<P><<<pack_blocks, 128, 0, s>>>(args);
  if ((st = check_launch("batched_pack_kernel"))) return st;
  int64_t grid = 0;
  if ((st = resident_grid(kernel, warps, bytes * warps, all, nullptr, &grid))) return st;
  NSI_CUDA(launch_early(kernel, grid, 32 * warps, bytes * warps, s, args, lays));
  return check_launch("batched_kernel");
}

template <int P>
nsi_status launch_exact_rows(NsiHandle* h, const FieldView& f, int mode, const RowOut& o, cudaStream_t s) {
  return h->nsub == 2 ? exact_rows_h<P, 2>(h, f, mode, o, s) : exact_rows_h<P, 4>(h, f, mode, o, s);
}
template nsi_status launch_exact_rows<NSI_MIXED_F32_ACC64>(NsiHandle*, const FieldView&, int, const RowOut&,
                                                            cudaStream_t);
template nsi_status launch_exact_rows<NSI_MIXED_F32_ACC32>(NsiHandle*, const FieldView&, int, const RowOut&,
                                                            cudaStream_t);

#define NSI_INSTANTIATE(P)                                                                                          \
  template nsi_status launch_pack<P>(NsiHandle*, const FieldView&, void*, cudaStream_t);                            \
  template nsi_status launch_gather<P>(NsiHandle*, const FieldView&, const OutView&, int64_t, int64_t, void*,       \
                                       cudaStream_t);                                                               \
  template nsi_status launch_step<P>(NsiHandle*, const FieldView&, const StepView&, bool, cudaStream_t);            \
  template nsi_status launch_batched<P>(NsiHandle* const*, const NsiFields*, const NsiOutputs*, int, cudaStream_t);
NSI_INSTANTIATE(NSI_FP64)
NSI_INSTANTIATE(NSI_MIXED_F32_ACC64)
NSI_INSTANTIATE(NSI_MIXED_F32_ACC32)
#undef NSI_INSTANTIATE

int gather_kernel_regs(int precision) {
  cudaFuncAttributes a{};
  cudaError_t e;
  if (precision == NSI_FP64) e = cudaFuncGetAttributes(&a, gather_persistent_kernel<NSI_FP64, 2, ASSEMBLE, false, false>);
  else if (precision == NSI_MIXED_F32_ACC64)
    e = cudaFuncGetAttributes(&a, gather_persistent_kernel<NSI_MIXED_F32_ACC64, 2, ASSEMBLE, false, false>);
  else e = cudaFuncGetAttributes(&a, gather_persistent_kernel<NSI_MIXED_F32_ACC32, 2, ASSEMBLE, false, false>);
  return e == cudaSuccess ? a.numRegs : 96;
}

}  // namespace nsi
