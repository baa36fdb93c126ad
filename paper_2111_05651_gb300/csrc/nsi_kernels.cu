// Device kernels and the per-call entry points of libnsi_assemble.
//
//   elem_kernel     one element per thread (calculate_transients ...
//                   perform_assembly_in_global_system of Listing 1 fused),
//                   scatter by global atomics or, colour by colour, by plain
//                   read-add-write (deterministic)
//   fan_kernel      one CSR entry per thread, walking the ring of elements
//                   around its edge (autotuning candidate)
//   vjp_kernel      adjoint of R(u, mu) = A(u) u - b, element per thread
//   residual_kernel R(u, mu) without the matrix (both with an exact
//                   companion for badly shaped elements in double)
//   rows64_kernel   rows without a walk (more than 32 entries, for instance)
//                   in double, one block per row
//   stab_star_kernel  the stabilised velocity block (3x3 per CSR entry): one
//                   warp per row or pair of rows, each element evaluated
//                   once per row, entry sums from shared memory
//   stab_rows_kernel  the stabilised block of listed rows, one thread per
//                   row in double
//   gather_values_kernel, add_values_kernel  pack / add the interface-row
//                   values of the element-partition exchange
//
// The row gather, the time step and the batched launch are in nsi_gather.cu.
// Formulas: see the element-arithmetic comment in nsi_internal.cuh.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <vector>

#include "nsi_device.cuh"

namespace nsi {

__device__ __forceinline__ float fma_of(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_of(double a, double b, double c) { return fma(a, b, c); }

// ------------------------------------------------ element-centric kernel ---
template <typename T, typename Out>
__device__ __forceinline__ void add_out(Out* p, T v, bool atomic);

template <>
__device__ __forceinline__ void add_out<double, double>(double* p, double v, bool atomic) {
  if (atomic) atomicAdd(p, v);
  else *p += v;
}
template <>
__device__ __forceinline__ void add_out<float, float>(float* p, float v, bool atomic) {
  if (atomic) atomicAdd(p, v);
  else *p += v;
}
// an element value in the output type (float -> double exactly)
template <typename T, typename Out>
__device__ __forceinline__ Out to_out(T v) {
  if constexpr (sizeof(T) == sizeof(Out)) return v;
  else return __longlong_as_double(f32_to_f64_bits(v));
}
template <>
__device__ __forceinline__ void add_out<float, double>(double* p, float v, bool atomic) {
  double d = __longlong_as_double(f32_to_f64_bits(v));
  if (atomic) atomicAdd(p, d);  // the add itself happens in the L2 atomic unit
  else *p += d;
}

// Warp-aggregated global add: the lanes of a warp whose `key` (the output
// position) is equal form a group (__match_any_sync); the group's lowest lane
// collects the others' values by shuffles, in lane order, and issues one
// atomic add per value, value k to dst[k] (the same address in every lane of
// a group: it is a function of the key).  Every lane of the warp takes part
// (a lane with nothing to add passes a key of its own and valid = false).
template <int V, typename Out>
__device__ __forceinline__ void warp_aggregated_add(Out* const (&dst)[V], int64_t key, const Out (&val)[V],
                                                    bool valid) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned peers = __match_any_sync(0xffffffffu, key);
  Out sum[V];
#pragma unroll
  for (int k = 0; k < V; ++k) sum[k] = val[k];
  unsigned others = peers & (peers - 1u);  // the group's lanes after its leader
  while (__any_sync(0xffffffffu, others != 0u)) {
    const int src = others ? __ffs(others) - 1 : (int)lane;
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const Out v = __shfl_sync(0xffffffffu, val[k], src);
      if (others) sum[k] += v;
    }
    others &= others - 1u;
  }
  if (valid && lane == (unsigned)(__ffs(peers) - 1)) {
#pragma unroll
    for (int k = 0; k < V; ++k) atomicAdd(dst[k], sum[k]);
  }
}

// One element per thread (the Listing 1 subroutines fused).  Each of the 16
// (row, column) entries of the element is located in the CSR pattern through
// the element-position map (or, for rows longer than 32 entries, a scan of
// the row), and its A value and three G values are added:
//   ATOMIC: by global atomic adds, one per value, or with AGG by
//           warp-aggregated atomics (the elements of a warp are consecutive
//           in the mesh's order, so neighbouring elements share entries;
//           every group of lanes adding to one entry issues one atomic per
//           value) -- the scatter's order is not deterministic;
//   otherwise (one colour of a colouring: no two elements of the launch share
//           a node) by plain read-add-write, deterministic.
// In mixed64 the float element values are converted to double exactly
// before they are summed (the accumulation is in double).
template <int P, bool ATOMIC, bool DEBUG, bool AGG = false>
__global__ void __launch_bounds__(256) elem_kernel(MeshView m, FieldView f, OutView o,
                                                   const int32_t* __restrict__ elems, int64_t count,
                                                   const unsigned long long* __restrict__ elem_pos) {
  using T = typename Prec<P>::T;
  using Out = typename Prec<P>::Out;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool valid = t < count;
  if (!ATOMIC && !valid) return;  // (the atomic path keeps whole warps for the aggregation)
  const int64_t e = valid ? (elems ? (int64_t)elems[t] : t) : 0;
  const int4 q = valid ? m.lnods[e] : make_int4(0, 0, 0, 0);
  const int v[4] = {q.x, q.y, q.z, q.w};
  if (DEBUG && valid) {
    for (int a = 0; a < 4; ++a)
      if (v[a] < 0 || v[a] >= m.n) {
        atomicOr(m.err, ERR_BAD_INDEX);
        valid = false;
      }
    if (!valid) {
      if (!ATOMIC) return;
    }
  }
  const int vv[4] = {valid ? v[0] : 0, valid ? v[1] : 0, valid ? v[2] : 0, valid ? v[3] : 0};
  // gather (calculate_transients)
  NodeX<P> X[4];
  V3<T> u[4], un[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    X[a].load(m, vv[a]);
    u[a] = load_vec<T>(f.u, vv[a]);
    un[a] = load_vec<T>(f.un, vv[a]);
  }
  // Jacobian columns, cofactors, det (calculate_cartesian_derivatives)
  const V3<T> d1 = X[1].minus(X[0]), d2 = X[2].minus(X[0]), d3 = X[3].minus(X[0]);
  V3<T> c[4];
  c[1] = cross(d2, d3);
  c[2] = cross(d3, d1);
  c[3] = cross(d1, d2);
  const T det = dot(d1, c[1]);
  c[0] = {-(c[1].x + c[2].x + c[3].x), -(c[1].y + c[2].y + c[3].y), -(c[1].z + c[2].z + c[3].z)};
  // Gauss-point velocity moments and element matrices
  const V3<T> S = add(add(u[0], u[1]), add(u[2], u[3]));
  const T kc = kc_of<T>(f);
  const T kv = kmu_of<T>(f) * rcp(valid ? det : T(1));
  const T km = det * kmass_of<T>(f);
  const T kg = (T)(-1.0 / 24.0);
  Out* A = static_cast<Out*>(o.A);
  Out* G = static_cast<Out*>(o.G);
  Out* R = static_cast<Out*>(o.rhs);
  // perform_assembly_in_global_system: the 16 positions of the element's entries
  int pos[4][4];
  if (elem_pos) {
    const unsigned long long w = valid ? elem_pos[e] : 0ull;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int rs = m.row_ptr[vv[a]];
#pragma unroll
      for (int b = 0; b < 4; ++b)
        pos[a][b] = rs + (b == a ? (int)m.diag_pos[vv[a]]
                                 : (int)((w >> (ELEM_POS_BITS * elem_pos_slot(a, b))) & 31ull));
    }
  } else {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int r = vv[a];
      const int rs = m.row_ptr[r], re = m.row_ptr[r + 1];
#pragma unroll
      for (int b = 0; b < 4; ++b) pos[a][b] = -1;
      for (int s2 = rs; s2 < re; ++s2) {
        const int cidx = m.col_idx[s2];
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (cidx == vv[b]) pos[a][b] = s2;
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const V3<T> va = add(S, u[a]);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      bool ok = valid;
      if (DEBUG && ok && pos[a][b] < 0) {
        atomicOr(m.err, ERR_NOT_IN_PATTERN);
        ok = false;
      }
      T Aab = kc * dot(va, c[b]) + kv * dot(c[a], c[b]);
      if (a == b) Aab += km;
      const T g3[3] = {kg * c[a].x, kg * c[a].y, kg * c[a].z};
      if constexpr (ATOMIC) {
        Out vals[4];
        vals[0] = to_out<T, Out>(Aab);
#pragma unroll
        for (int d = 0; d < 3; ++d) vals[d + 1] = to_out<T, Out>(g3[d]);
        const int64_t key = ok ? (int64_t)pos[a][b] : -1 - (int64_t)(threadIdx.x & 31u);
        const int64_t pk = ok ? key : 0;
        Out* const dst[4] = {A + pk, G + pk, G + m.nnz + pk, G + 2 * m.nnz + pk};
        if constexpr (AGG) {
          warp_aggregated_add<4, Out>(dst, key, vals, ok);
        } else if (ok) {
#pragma unroll
          for (int k = 0; k < 4; ++k) atomicAdd(dst[k], vals[k]);
        }
      } else if (ok) {
        add_out<T, Out>(A + pos[a][b], Aab, false);
#pragma unroll
        for (int d = 0; d < 3; ++d) add_out<T, Out>(G + d * m.nnz + pos[a][b], g3[d], false);
      }
    }
    const T r3[3] = {km * un[a].x, km * un[a].y, km * un[a].z};
    if constexpr (ATOMIC) {
      Out rv[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) rv[k] = to_out<T, Out>(r3[k]);
      const int64_t key = valid ? (int64_t)vv[a] : -1 - (int64_t)(threadIdx.x & 31u);
      Out* const dst[3] = {R + vv[a], R + m.n + vv[a], R + 2 * m.n + vv[a]};
      if constexpr (AGG) {
        warp_aggregated_add<3, Out>(dst, key, rv, valid);
      } else if (valid) {
#pragma unroll
        for (int k = 0; k < 3; ++k) atomicAdd(dst[k], rv[k]);
      }
    } else if (valid) {
#pragma unroll
      for (int k = 0; k < 3; ++k) add_out<T, Out>(R + k * m.n + vv[a], r3[k], false);
    }
  }
}

// the element's coordinates, velocities and weights in double (the handle's
// copy of the coordinates: double, or the float hi + lo pair)
template <int P>
__device__ __forceinline__ V3<double> coord64(const MeshView& m, int64_t j) {
  if constexpr (P == NSI_FP64) {
    const D4 x = m.xyz64[j];
    return V3<double>{x.x, x.y, x.z};
  } else {
    const float4 h = m.xyz_hi[j], l = m.xyz_lo[j];
    return V3<double>{(double)h.x + (double)l.x, (double)h.y + (double)l.y, (double)h.z + (double)l.z};
  }
}
template <typename T>
__device__ __forceinline__ V3<double> vec64(const void* const* comp, int64_t j) {
  const V3<T> v = load_vec<T>(comp, j);
  return V3<double>{(double)v.x, (double)v.y, (double)v.z};
}

// ------------------------------------------------- rows without a walk ---
// Listed rows computed in double, one block per row: the rows the row gather
// leaves out (more than 32 entries, whose row positions do not fit the walk's
// five bits, or a star the walk encoder could not cover) and, of the rows of
// badly shaped elements, those without a walk.  In chunks of a block's threads
// every thread evaluates one element of the row (the row's node i first, the
// others in an even order, so that det > 0; its nodes' row positions by binary
// search) into shared memory and marks it in its entries' bit masks, then every
// entry's thread adds, in element order, the contributions w . c_j and
// -c_i / 24 of its marked elements; rows of more entries than threads take the
// elements again for every tile of entries.  The
// diagonal follows from the partition of unity as in the row gather,
// A(i,i) = lumped mass - sum_{j != i} A(i,j) and G(i,i) = 1/3 sum_{j != i}
// G(i,j).  MODE 0: A, G and rhs; 1: the time step, A = A_static + C(u) (A may
// alias A_static: each entry is read before it is written, by its thread) and
// rhs, or with no A (rows of badly shaped elements: the convection does not
// involve the determinant) rhs alone; 2: rhs, dt_rho and mass_rho.
// The rows are few and their serial work is what counts: the assembly of a
// pipe with 71 of them (the axis: 83 entries, 240 elements) takes 106 us with
// 256 threads a block, 111 with 128, 138 with 64; 14 us more with the entries
// scanning all elements instead of their marked ones; with one thread per row
// (and one per row of a badly shaped element) it took 7.2 ms.
constexpr int ROW_THREADS = 256;
template <int P, int MODE>
__global__ void __launch_bounds__(ROW_THREADS) rows64_kernel(MeshView m, FieldView f, RowOut o,
                                                             const int32_t* __restrict__ rows,
                                                             const int32_t* __restrict__ ptr,
                                                             const uint32_t* __restrict__ inc) {
  using Out = typename Prec<P>::Out;
  constexpr int B = ROW_THREADS;
  __shared__ double ea[B][3], ec[B][3], red[5][B / 32];
  __shared__ int ep[B][3];
  __shared__ unsigned mask[B][B / 32];  // per entry of the tile: the chunk's elements that hold it
  __shared__ int32_t near[4 * B];       // the row's columns, or the first of them
  const int tid = threadIdx.x;
  const int64_t r = blockIdx.x, i = rows[r];
  const int32_t rs = m.row_ptr[i], len = m.row_ptr[i + 1] - rs;
  const int32_t* cols = m.col_idx + rs;
  const int32_t t0 = ptr[r], nel = ptr[r + 1] - t0;
  auto vel = [&](const void* const* comp, int64_t j) { return vec64<typename Prec<P>::T>(comp, j); };
  // even permutations of (0,1,2,3) that bring vertex a to the front
  const int EVEN[4][3] = {{1, 2, 3}, {0, 3, 2}, {3, 0, 1}, {2, 1, 0}};
  const V3<double> xi = coord64<P>(m, i), ui = vel(f.u, i);
  // of this thread: the determinants of its elements, its entries' sums for the diagonal
  double det = 0.0, sa = 0.0, sg[3] = {0.0, 0.0, 0.0};
  const bool entries = MODE == 0 || (MODE == 1 && o.A);
  if (entries)
    for (int q = tid; q < min(len, 4 * B); q += B) near[q] = cols[q];
  // position of column j in the row (columns ascending)
  auto position = [&](int32_t j) {
    int lo = 0, hi = len - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((mid < 4 * B ? near[mid] : cols[mid]) < j) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  for (int q0 = 0; q0 == 0 || (entries && q0 < len); q0 += B) {
    const int q = q0 + tid;
    const bool mine = entries && q < len && cols[q] != i;
    double a = 0.0, g[3] = {0.0, 0.0, 0.0};
    for (int c0 = 0; c0 < nel; c0 += B) {
      __syncthreads();  // the previous chunk is used up
      if (entries) {
        for (int w = 0; w < B / 32; ++w) mask[tid][w] = 0u;
        __syncthreads();
      }
      if (c0 + tid < nel) {
        const uint32_t w = inc[t0 + c0 + tid];
        const int4 v4 = m.lnods[w >> 2];
        const int v[4] = {v4.x, v4.y, v4.z, v4.w};
        int nb[3];
        V3<double> d[3], us{2.0 * ui.x, 2.0 * ui.y, 2.0 * ui.z};
        for (int b = 0; b < 3; ++b) {
          nb[b] = v[EVEN[w & 3u][b]];
          d[b] = sub(coord64<P>(m, nb[b]), xi);
        }
        const V3<double> c[3] = {cross(d[1], d[2]), cross(d[2], d[0]), cross(d[0], d[1])};
        const double dt = dot(d[0], c[0]);
        if (q0 == 0) det += dt;
        if (entries) {
          const V3<double> ci{-(c[0].x + c[1].x + c[2].x), -(c[0].y + c[1].y + c[2].y), -(c[0].z + c[1].z + c[2].z)};
          for (int b = 0; b < 3; ++b) us = add(us, vel(f.u, nb[b]));
          const double kv = MODE == 0 ? f.kmu * rcp_fast(dt) : 0.0;
          const V3<double> w3{f.kc * us.x + kv * ci.x, f.kc * us.y + kv * ci.y, f.kc * us.z + kv * ci.z};
          for (int b = 0; b < 3; ++b) {
            ea[tid][b] = dot(w3, c[b]);
            ep[tid][b] = position(nb[b]);
            const int e = ep[tid][b] - q0;
            if (e >= 0 && e < B) atomicOr(&mask[e][tid >> 5], 1u << (tid & 31));
          }
          ec[tid][0] = ci.x;
          ec[tid][1] = ci.y;
          ec[tid][2] = ci.z;
        }
      }
      __syncthreads();
      if (mine) {
        for (int w = 0; w < B / 32; ++w)
          for (unsigned bits = mask[tid][w]; bits; bits &= bits - 1) {
            const int e = 32 * w + __ffs(bits) - 1;
            a += ea[e][ep[e][0] == q ? 0 : ep[e][1] == q ? 1 : 2];
            if constexpr (MODE == 0)
              for (int d = 0; d < 3; ++d) g[d] += ec[e][d];
          }
      }
    }
    wait_for_previous();  // (the rows' first values come from the launch before)
    if (mine) {
      sa += a;
      if constexpr (MODE == 0) {
        static_cast<Out*>(o.A)[rs + q] = (Out)a;
        for (int d = 0; d < 3; ++d) {
          static_cast<Out*>(o.G)[d * m.nnz + rs + q] = (Out)(-g[d] / 24.0);
          sg[d] += g[d];
        }
      } else if constexpr (MODE == 1) {
        static_cast<Out*>(o.A)[rs + q] = (Out)((double)static_cast<const Out*>(o.A_static)[rs + q] + a);
      }
    }
  }
  // the row's totals: a tree over each warp, then the warps in order
  double tot[5] = {det, sa, sg[0], sg[1], sg[2]};
  for (int k = 0; k < 5; ++k) {
    for (int off = 16; off > 0; off >>= 1) tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], off);
    if ((tid & 31) == 0) red[k][tid >> 5] = tot[k];
  }
  __syncthreads();
  if (tid != 0) return;
  for (int k = 0; k < 5; ++k) {
    tot[k] = 0.0;
    for (int w = 0; w < B / 32; ++w) tot[k] += red[k][w];
  }
  if (entries && len > 0) {
    const int lo = position((int32_t)i);
    Out* A = static_cast<Out*>(o.A) + rs + lo;
    if constexpr (MODE == 0) {
      *A = (Out)(f.kmass * tot[0] - tot[1]);
      for (int d = 0; d < 3; ++d) static_cast<Out*>(o.G)[d * m.nnz + rs + lo] = (Out)(-tot[2 + d] / 72.0);
    } else {
      *A = (Out)((double)static_cast<const Out*>(o.A_static)[rs + lo] - tot[1]);
    }
  }
  const V3<double> un = vel(f.un, i);
  const double mass = f.kmass * tot[0];
  Out* Rh = static_cast<Out*>(o.rhs);
  Rh[i] = (Out)(mass * un.x);
  Rh[m.n + i] = (Out)(mass * un.y);
  Rh[2 * m.n + i] = (Out)(mass * un.z);
  if constexpr (MODE == 2) {
    static_cast<Out*>(o.dt_rho)[i] = (Out)mass;
    static_cast<Out*>(o.mass_rho)[i] = (Out)(o.kmr * tot[0]);
  }
}

// asynchronous global -> shared copies (cp.async): many gathers in flight per
// thread without holding registers
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ------------------------------------------------------ edge-fan kernel ---
// One thread per CSR entry (i, j) of a block of whole rows.  An off-diagonal
// entry walks the ring of nodes k_0 .. k_{r-1} around the edge (i, j): the
// elements containing the edge are (i, j, k_m, k_{m+1}), positively oriented.
// With i as the origin and q_m = d_j x d_{k_m}, such an element has
//   c_j = d_{k_m} x d_{k_{m+1}},  c_i = -(c_j + q_m - q_{m+1}),  det = d_j . c_j
// (c_{k_m} = -q_{m+1} and c_{k_{m+1}} = q_m come for free from the ring), and
// adds w . c_j to A(i, j), c_i to the pressure-gradient sum and det to the
// lumped mass sum, with w = rho/120 (2 u_i + u_j + u_{k_m} + u_{k_{m+1}}) +
// mu/(6 det) c_i.  All sums stay in registers.  The diagonal entry receives
// the row totals through a tree reduction in shared memory:
//   A(i,i) = M_i - sum_{j != i} A(i,j), G(i,i) = 1/3 sum_{j != i} G(i,j),
//   M_i = rho/(24 dt) * 1/3 sum_{j != i} sum_fan det
// (every element of the star appears in the fans of its three other nodes).
// Every thread then writes its own entry: the block's slice of A and G goes
// out coalesced.

// shared-memory layout of a fan block (T entries)
template <int P>
struct FanSmem {
  using T = typename Prec<P>::T;
  static constexpr size_t rec() { return 0; }                                        // T4 [T] x 2
  static constexpr size_t rp(int Tn) { return 2 * sizeof(T4<T>) * (size_t)Tn; }      // int32 [T + 1]
  static constexpr size_t red(int Tn) { return rp(Tn) + (((size_t)4 * (Tn + 1) + 15) & ~size_t(15)); }
  static constexpr size_t total(int Tn) { return red(Tn) + 5 * sizeof(Acc<P>) * (size_t)Tn; }
};

template <int P>
__device__ __forceinline__ void acc_merge(Acc<P>& a, const Acc<P>& b) {
  if constexpr (P == NSI_MIXED_F32_ACC64) {
    a.add(b.hi);
    a.lo += b.lo;
  } else {
    a.v += b.v;
  }
}

// x / 3 of an accumulator (compensated for the pair)
template <int P>
__device__ __forceinline__ Acc<P> acc_third(const Acc<P>& a) {
  Acc<P> r;
  if constexpr (P == NSI_MIXED_F32_ACC64) {
    const float q = a.hi * (1.0f / 3.0f);
    r.hi = q;
    r.lo = fmaf(a.hi, 1.0f / 3.0f, -q) + a.lo * (1.0f / 3.0f);
  } else {
    r.v = a.v * (typename Prec<P>::T(1) / typename Prec<P>::T(3));
  }
  return r;
}

// c * (a), product error kept for the pair
template <int P>
__device__ __forceinline__ Acc<P> acc_scale(const Acc<P>& a, typename Prec<P>::T c) {
  Acc<P> r;
  if constexpr (P == NSI_MIXED_F32_ACC64) {
    const float p = c * a.hi;
    r.hi = p;
    r.lo = fmaf(c, a.hi, -p) + c * a.lo;
  } else {
    r.v = c * a.v;
  }
  return r;
}

// One CSR entry of a fan block (blocks of whole rows, one thread per entry):
// its row within the block, the row's start and length in the block, the
// diagonal's position, the fan word, and (node i the row's node, j the
// column's) the edge vector d_j = x_j - x_i and the velocities u_j, u_i.
template <typename T>
struct FanEntry {
  int64_t R0;
  int32_t base;
  int nr, L, row, a, len, dp;
  uint32_t w;
  V3<T> dj, uj, ui;
};

// Steps 1-2 of a fan block: the row starts of the block, this entry's
// neighbour record (calculate_transients), its row and edge vector; then
// every entry's record in shared memory is replaced by (edge vector from its
// row's node, velocity).  Returns false (block-uniform) when DEBUG finds the
// block larger than the kernel's.
template <int P, bool DEBUG>
__device__ __forceinline__ bool fan_entry(const MeshView& m, int64_t blk, T4<typename Prec<P>::T>* rec0,
                                          T4<typename Prec<P>::T>* rec1, int32_t* rp,
                                          FanEntry<typename Prec<P>::T>& e) {
  using T = typename Prec<P>::T;
  constexpr int TB = FAN_BLOCK;
  const int k = threadIdx.x;
  e.R0 = m.fan_blk[blk];
  const int64_t R1 = m.fan_blk[blk + 1];
  e.nr = (int)(R1 - e.R0);
  e.base = m.row_ptr[e.R0];
  e.L = m.row_ptr[R1] - e.base;
  if (DEBUG && (e.L > TB || e.nr > TB)) {
    if (k == 0) atomicOr(m.err, ERR_STAR);
    return false;
  }
  for (int r = k; r <= e.nr; r += TB) rp[r] = m.row_ptr[e.R0 + r] - e.base;
  e.w = 0;
  if (k < e.L) {
    const int j = m.col_idx[e.base + k];
    e.w = m.fan[e.base + k];
    if (!DEBUG || (j >= 0 && j < m.n)) {
      const unsigned char* r = static_cast<const unsigned char*>(m.rec) + (size_t)j * (2 * sizeof(T4<T>));
      if constexpr (P == NSI_FP64) {
        cp_async16(&rec0[k], r);
        cp_async16(reinterpret_cast<char*>(&rec0[k]) + 16, r + 16);
        cp_async16(&rec1[k], r + 32);
        cp_async16(reinterpret_cast<char*>(&rec1[k]) + 16, r + 48);
      } else {
        cp_async16(&rec0[k], r);
        cp_async16(&rec1[k], r + 16);
      }
    } else {
      atomicOr(m.err, ERR_BAD_INDEX);
    }
  }
  cp_async_wait_all();
  __syncthreads();

  e.row = e.a = e.len = e.dp = 0;
  e.dj = e.uj = e.ui = V3<T>{T(0), T(0), T(0)};
  if (k < e.L) {
    int lo = 0, hi = e.nr - 1;  // last row whose start is <= k
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (rp[mid] <= k) lo = mid;
      else hi = mid - 1;
    }
    e.row = lo;
    e.a = rp[e.row];
    e.len = rp[e.row + 1] - e.a;
    e.dp = m.diag_pos[e.R0 + e.row];
    const T4<T> h = rec0[k], s = rec1[k];
    const T4<T> hd = rec0[e.a + e.dp], sd = rec1[e.a + e.dp];
    if constexpr (P == NSI_FP64) {
      e.dj = {h.x - hd.x, h.y - hd.y, h.z - hd.z};
      e.uj = {s.x, s.y, s.z};
      e.ui = {sd.x, sd.y, sd.z};
    } else {
      const V3<float> lj = record_lo(s.z, s.w), li = record_lo(sd.z, sd.w);
      e.dj = add(sub(V3<float>{h.x, h.y, h.z}, V3<float>{hd.x, hd.y, hd.z}), sub(lj, li));
      e.uj = {h.w, s.x, s.y};
      e.ui = {hd.w, sd.x, sd.y};
    }
  }
  __syncthreads();
  if (k < e.L) {
    rec0[k] = T4<T>{e.dj.x, e.dj.y, e.dj.z, T(0)};
    rec1[k] = T4<T>{e.uj.x, e.uj.y, e.uj.z, T(0)};
  }
  __syncthreads();
  return true;
}

template <int P, bool DEBUG>
__device__ __forceinline__ void fan_block(const MeshView& m, const FieldView& f, const OutView& o, int64_t blk,
                                          unsigned char* smem) {
  using T = typename Prec<P>::T;
  using Out = typename Prec<P>::Out;
  constexpr int TB = FAN_BLOCK;
  T4<T>* rec0 = reinterpret_cast<T4<T>*>(smem + FanSmem<P>::rec());
  T4<T>* rec1 = rec0 + TB;
  int32_t* rp = reinterpret_cast<int32_t*>(smem + FanSmem<P>::rp(TB));
  Acc<P>* red = reinterpret_cast<Acc<P>*>(smem + FanSmem<P>::red(TB));  // 5 arrays of TB
  const int k = threadIdx.x;
  FanEntry<T> fe;
  if (!fan_entry<P, DEBUG>(m, blk, rec0, rec1, rp, fe)) return;
  const int64_t R0 = fe.R0;
  const int nr = fe.nr, L = fe.L, row = fe.row, a = fe.a, len = fe.len, dp = fe.dp;
  const int32_t base = fe.base;
  const uint32_t w = fe.w;
  const V3<T> dj = fe.dj, uj = fe.uj, ui = fe.ui;
  const T kc = kc_of<T>(f), kmu = kmu_of<T>(f), kmass = kmass_of<T>(f);
  const T kg = (T)(-1.0 / 24.0);

  // 3. the fan of an off-diagonal entry, summed in registers
  Acc<P> sA, sGx, sGy, sGz, sD;
  sA.zero(); sGx.zero(); sGy.zero(); sGz.zero(); sD.zero();
  const int nring = (w >> 24) & 7;
  if (k < L && nring > 0) {
    const bool closed = (w >> 27) & 1;
    const int nel = closed ? nring : nring - 1;
    const V3<T> uij{ui.x + ui.x + uj.x, ui.y + ui.y + uj.y, ui.z + ui.z + uj.z};  // 2 u_i + u_j
    auto node = [&](int mpos, V3<T>& d, V3<T>& u) {
      const int pos = (w >> (4 * mpos)) & 15;
      if (DEBUG && pos >= len) atomicOr(m.err, ERR_STAR);
      const T4<T> x = rec0[a + pos], y = rec1[a + pos];
      d = {x.x, x.y, x.z};
      u = {y.x, y.y, y.z};
    };
    V3<T> d0, u0;
    node(0, d0, u0);
    V3<T> q0 = cross(dj, d0);
    const V3<T> dfirst = d0, ufirst = u0, qfirst = q0;
    for (int e = 0; e < nel; ++e) {
      V3<T> d1, u1, q1;
      if (e + 1 < nring) {
        node(e + 1, d1, u1);
        q1 = cross(dj, d1);
      } else {  // closing element of an interior ring
        d1 = dfirst;
        u1 = ufirst;
        q1 = qfirst;
      }
      const V3<T> cj = cross(d0, d1);
      const T det = dot(dj, cj);
      const V3<T> ci{-(cj.x + q0.x - q1.x), -(cj.y + q0.y - q1.y), -(cj.z + q0.z - q1.z)};
      const T kv = kmu * rcp_fast(det);
      const V3<T> w3{kc * (uij.x + u0.x + u1.x) + kv * ci.x, kc * (uij.y + u0.y + u1.y) + kv * ci.y,
                     kc * (uij.z + u0.z + u1.z) + kv * ci.z};
      sA.add(dot(w3, cj));
      sGx.add(ci.x);
      sGy.add(ci.y);
      sGz.add(ci.z);
      sD.add(det);
      d0 = d1;
      u0 = u1;
      q0 = q1;
    }
  }

  // 4. row totals for the diagonal: tree reduction over each row's entries
  Acc<P>* rA = red;
  Acc<P>* rGx = red + TB;
  Acc<P>* rGy = red + 2 * TB;
  Acc<P>* rGz = red + 3 * TB;
  Acc<P>* rD = red + 4 * TB;
  if (k < L) {
    rA[k] = sA;
    rGx[k] = sGx;
    rGy[k] = sGy;
    rGz[k] = sGz;
    rD[k] = sD;
  }
  __syncthreads();
#pragma unroll
  for (int st = 1; st < FAN_MAX_ROW; st <<= 1) {
    if (k < L && ((k - a) & (2 * st - 1)) == 0 && k - a + st < len) {
      acc_merge<P>(rA[k], rA[k + st]);
      acc_merge<P>(rGx[k], rGx[k + st]);
      acc_merge<P>(rGy[k], rGy[k + st]);
      acc_merge<P>(rGz[k], rGz[k + st]);
      acc_merge<P>(rD[k], rD[k + st]);
    }
    __syncthreads();
  }

  // 5. this entry's outputs (coalesced across the block), the diagonal's and the RHS
  Out* A = static_cast<Out*>(o.A);
  Out* G = static_cast<Out*>(o.G);
  Out* Rh = static_cast<Out*>(o.rhs);
  if (k < L) {
    const int64_t g = (int64_t)base + k;
    if (k == a + dp) {
      const Acc<P> d3 = acc_third<P>(rD[a]);
      const Acc<P> mass = acc_scale<P>(d3, kmass);
      Acc<P> add_ = mass;
      if constexpr (P == NSI_MIXED_F32_ACC64) {
        add_.add(-rA[a].hi);
        add_.lo -= rA[a].lo;
      } else {
        add_.v = mass.v - rA[a].v;
      }
      store_acc(A + g, add_);
      store_acc(G + g, acc_scale<P>(acc_third<P>(rGx[a]), kg));
      store_acc(G + m.nnz + g, acc_scale<P>(acc_third<P>(rGy[a]), kg));
      store_acc(G + 2 * m.nnz + g, acc_scale<P>(acc_third<P>(rGz[a]), kg));
      const int64_t i = R0 + row;
      const V3<T> un = load_vec<T>(f.un, i);
      store_acc(Rh + i, acc_scale<P>(mass, un.x));
      store_acc(Rh + m.n + i, acc_scale<P>(mass, un.y));
      store_acc(Rh + 2 * m.n + i, acc_scale<P>(mass, un.z));
    } else {
      store_acc(A + g, sA);
      store_acc(G + g, acc_scale<P>(sGx, kg));
      store_acc(G + m.nnz + g, acc_scale<P>(sGy, kg));
      store_acc(G + 2 * m.nnz + g, acc_scale<P>(sGz, kg));
    }
  }
  // rows without entries (nodes in no element): zero right-hand side
  for (int r = k; r < nr; r += TB) {
    if (rp[r + 1] == rp[r]) {
      Acc<P> z;
      z.zero();
      store_acc(Rh + R0 + r, z);
      store_acc(Rh + m.n + R0 + r, z);
      store_acc(Rh + 2 * m.n + R0 + r, z);
    }
  }
}

template <int P, bool DEBUG>
__global__ void __launch_bounds__(FAN_BLOCK) fan_kernel(MeshView m, FieldView f, OutView o) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fan_block<P, DEBUG>(m, f, o, blockIdx.x, smem_raw);
}

// --------------------------------------------- stabilised velocity block ---
// The paper's 12x12 element matrix (Section II-A: every pair of dimensions of
// two nodes coupled, equal dimensions receiving the scalar part) assembled on
// the CSR pattern as one 3x3 block per entry, Auu[(3 a + b) nnz + p] the
// (a, b) entry of the block of entry p = (i, j):
//   Auu(i,j)[a][b] = delta_ab (A(i,j) + S(i,j)) + K(i,j)[a][b]
// with A the Galerkin operator and the implicit terms of Codina's algebraic
// subgrid scales (Comput. Methods Appl. Mech. Engrg. 191 (2002) 4295-4321,
// linear elements, c1 = 4, c2 = 2):
//   tau1 = (4 mu / h^2 + 2 rho |ubar| / h)^-1,  tau2 = h^2 / (4 tau1),
//   S(i,j)       += tau1 rho^2 int (u . grad N_i)(u . grad N_j)
//   K(i,j)[a][b] += mu int d_b N_i d_a N_j + tau2 int d_a N_i d_b N_j
// per element, h = (6 |T|)^(1/3) = det^(1/3), ubar the mean of the element's
// four node velocities.  With the cofactors c_n = det grad N_n, the sum us of
// the four velocities and s = |us| (so 2 rho |ubar| h = rho s h / 2, and the
// moments int lam_m lam_n = |T| (1 + delta_mn) / 20 of the linear velocity):
//   S += rho^2 / (120 h (4 mu + rho s h / 2)) [(us . c_i)(us . c_j) + sum_n (u_n . c_i)(u_n . c_j)]
//   K[a][b] += kv c_j[a] c_i[b] + kd c_i[a] c_j[b],
//   kv = mu / (6 det),  kd = tau2 / (6 det) = kv + rho s h / (48 det).
// Every term vanishes on a constant column field (sum_n c_n = 0), so, as for
// A, the diagonal block is the lumped mass times I minus the sum of the row's
// off-diagonal blocks.
struct StabConst {
  double ks, k4mu, krh, kr48;  // rho^2 / 120, 4 mu, rho / 2, rho / 48
  double kml;                  // what rho / (24 dt) lacks in FieldView::kmass
  float ksf, k4muf, krhf, kr48f, kmlf;
};

static StabConst stab_const(const NsiFields* f) {
  StabConst c;
  c.ks = f->rho * f->rho / 120.0;
  c.k4mu = 4.0 * f->mu;
  c.krh = f->rho / 2.0;
  c.kr48 = f->rho / 48.0;
  const double k = f->rho / (24.0 * f->dt), d = 24.0 * f->dt;
  c.kml = (std::fma(-k, d, f->rho) - k * std::fma(24.0, f->dt, -d)) / d;
  if (!std::isfinite(c.kml)) c.kml = 0.0;
  c.kmlf = (float)(k - (double)(float)k);
  if (!std::isfinite(c.kmlf)) c.kmlf = 0.0f;
  c.ksf = (float)c.ks;
  c.k4muf = (float)c.k4mu;
  c.krhf = (float)c.krh;
  c.kr48f = (float)c.kr48;
  return c;
}

template <typename T>
struct StabK {
  T ks, k4mu, krh, kr48, kml;
};
template <typename T>
__device__ __forceinline__ StabK<T> stab_k(const StabConst& c) {
  if constexpr (sizeof(T) == 8) return StabK<T>{c.ks, c.k4mu, c.krh, c.kr48, c.kml};
  else return StabK<T>{c.ksf, c.k4muf, c.krhf, c.kr48f, c.kmlf};
}
__device__ __forceinline__ float cbrt_of(float x) { return cbrtf(x); }
__device__ __forceinline__ double cbrt_of(double x) { return cbrt(x); }
__device__ __forceinline__ float sqrt_of(float x) { return sqrtf(x); }
__device__ __forceinline__ double sqrt_of(double x) { return sqrt(x); }
// One element's stabilisation terms for the entry (row node, column node):
// ci, cj the two nodes' cofactors, det, and the element's four node
// velocities (any order).  K is added to; S is returned.
template <typename T>
__device__ __forceinline__ T stab_terms(const V3<T>& ci, const V3<T>& cj, T det, const V3<T>& ua, const V3<T>& ub,
                                        const V3<T>& uc, const V3<T>& ud, const StabK<T>& k, T kmu, T (&K)[9]) {
  const V3<T> us = add(add(ua, ub), add(uc, ud));
  const T h = cbrt_of(det);
  const T sh = sqrt_of(dot(us, us)) * h;  // s h
  const T rdet = rcp_fast(det);
  T mm = dot(us, ci) * dot(us, cj);
  mm = fma_of(dot(ua, ci), dot(ua, cj), mm);
  mm = fma_of(dot(ub, ci), dot(ub, cj), mm);
  mm = fma_of(dot(uc, ci), dot(uc, cj), mm);
  mm = fma_of(dot(ud, ci), dot(ud, cj), mm);
  const T kv = kmu * rdet;
  const T kd = fma_of(k.kr48 * sh, rdet, kv);
  const T r[3] = {ci.x, ci.y, ci.z}, c[3] = {cj.x, cj.y, cj.z};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) K[3 * a + b] = fma_of(kv * c[a], r[b], fma_of(kd * r[a], c[b], K[3 * a + b]));
  return k.ks * mm * rcp_fast(h * fma_of(k.krh, sh, k.k4mu));
}

// Lengths of Codina's tau for one element: h = det^(1/3) and s h with s the
// norm of the four velocities' sum.  Float: h from the exp2/log2 estimate and
// one Newton step for the cube root (h <- (2 h + det / h^2) / 3), s as
// s2 rsqrt(s2) (0 for s2 = 0); double: cbrt and sqrt.
__device__ __forceinline__ void tau_lengths(float det, float s2, float& h, float& sh) {
  const float h0 = exp2f(__log2f(det) * (1.0f / 3.0f));
  h = fmaf(h0, 2.0f / 3.0f, det * __fdividef(1.0f / 3.0f, h0 * h0));
  sh = (s2 > 0.0f ? s2 * rsqrtf(s2) : 0.0f) * h;
}
__device__ __forceinline__ void tau_lengths(double det, double s2, double& h, double& sh) {
  h = cbrt(det);
  sh = sqrt(s2) * h;
}

// Shared memory of one warp of the stabilised row kernel: entry records (edge
// vector from the row's node and u_x in a T4, u_y and u_z in a T2), then element
// records for a chunk of 64 elements, field by field: (c_i, mu/(6 det)),
// (c_1, A+S to node 1), (c_2, ..), (c_3, ..), tau2/(6 det); then per entry three
// 64-bit masks of the chunk's elements holding the entry as their first, second
// or third node.  The entries' reads of the element records are scattered and
// are what the kernel's shared memory is busy with most, so they are two T4 and
// one T per element and entry, and det stays with the lane that evaluated it.
template <int P>
struct StarSmem {
  using T = typename Prec<P>::T;
  static constexpr int CHUNK = 64;
  static constexpr size_t ent() { return 0; }
  static constexpr size_t el() { return sizeof(T) * 6 * 32; }
  static constexpr size_t kd() { return el() + sizeof(T4<T>) * 4 * CHUNK; }
  static constexpr size_t mask() { return kd() + sizeof(T) * CHUNK; }
  static constexpr size_t bytes() { return mask() + sizeof(unsigned) * 6 * 32; }
};
constexpr int STAR_WARPS = 4;  // warps (tasks) per block
// sum of x[0], x[ST], ..., x[(N - 1) ST] in pairs, neighbours first
template <int N, int ST, typename T>
__device__ __forceinline__ T pair_sum(const T* x) {
  if constexpr (N == 1) return x[0];
  else return pair_sum<N / 2, ST>(x) + pair_sum<N / 2, ST>(x + N / 2 * ST);
}

// The stabilised block by rows, one warp per task (one row of up to 32
// entries, or two consecutive rows of up to 16 on the two half-warps).
//  1. Each entry lane loads its column's node record; the edge vector from the
//     row's node (the diagonal lane's record, by shuffles) and the velocity go
//     to shared memory.
//  2. In chunks of 64 elements (two per lane), each lane takes elements of the
//     task's stars (node i first, the others in a positively oriented order,
//     from the star word): cofactors, det, c_i, w = rho/120 (2 u_i + u_1 +
//     u_2 + u_3) + mu/(6 det) c_i, Codina's tau from h = det^(1/3) and the
//     velocity sum, the SUPG vector v = fs [(us . c_i) us + sum_n (u_n . c_i) u_n],
//     and the contributions (w + v) . c_k to its three entries; its record
//     goes to shared memory and its bit into those entries' masks.
//  3. Each off-diagonal entry lane adds, in element order, the records of its
//     masked elements: A + S, K += kv c_k x c_i + kd c_i x c_k and G's c_i sum.
//  4. The row's lanes 0-13 add up one value each over the row's entries, in
//     shared memory; the diagonal block is the lumped mass times I minus the
//     off-diagonal blocks' sum.
//  5. Every lane writes its own entry (the row's slice of each output array
//     is contiguous); the diagonal's twelve values and the right-hand side are
//     written by the row's lanes 0-14, one each.
// Each element is evaluated once per row of its star (four times per tet).
// Long rows (more than 32 entries, or a star the row-gather encoder could
// not cover) are single-row tasks this kernel skips.
// No unit is saturated: issue 67%, shared memory's data path 66%, the integer
// pipe 43% busy at six blocks per SM (registers; five 233 us per call of a
// 64x57x60 box in mixed64, seven 206, six 205), and the largest stall is the
// wait for a task's descriptor, columns and records.  With the totals by shuffles of
// every lane, the diagonal's values by its own lane and det in the records the
// call took 222 us, and the kernel at 100^3 944 instead of 890.
template <int P, bool DEBUG>
__global__ void __launch_bounds__(32 * STAR_WARPS, P == NSI_FP64 ? 1 : 6) stab_star_kernel(
    MeshView m, FieldView f, StabConst sc, const int4* __restrict__ tasks, int64_t ntasks,
    const uint16_t* __restrict__ star_word, void* Auu, void* Gv, void* rhs) {
  extern __shared__ __align__(128) unsigned char smem[];
  using T = typename Prec<P>::T;
  using Out = typename Prec<P>::Out;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int CH = StarSmem<P>::CHUNK;
  const int lane = threadIdx.x & 31;
  const int64_t task = (int64_t)blockIdx.x * STAR_WARPS + (threadIdx.x >> 5);
  if (task >= ntasks) return;  // warp-uniform
  unsigned char* ws = smem + (threadIdx.x >> 5) * StarSmem<P>::bytes();
  T4<T>* er = reinterpret_cast<T4<T>*>(ws + StarSmem<P>::ent());
  T2<T>* eu = reinterpret_cast<T2<T>*>(er + 32);
  T4<T>* el = reinterpret_cast<T4<T>*>(ws + StarSmem<P>::el());
  T* ekd = reinterpret_cast<T*>(ws + StarSmem<P>::kd());
  unsigned* mk = reinterpret_cast<unsigned*>(ws + StarSmem<P>::mask());  // [3 nodes][2 words][32 lanes]

  // the task's rows, CSR and star bounds and diagonal positions in one
  // 32-byte descriptor; long rows are left to the per-row kernel
  const int4 ta = tasks[2 * task], tb = tasks[2 * task + 1];
  if ((tb.w >> 24) & 1) return;  // warp-uniform
  const int nrow = (tb.w >> 16) & 3;  // 1 or 2
  const int64_t s0 = tb.x, s1 = tb.y, s2 = tb.z;
  const int nel = (int)(s2 - s0);
  // the first chunk's star words, loaded ahead of the rows' records
  unsigned wpre[2];
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) wpre[hf] = hf * 32 + lane < nel ? star_word[s0 + hf * 32 + lane] : 0u;
  const int width = nrow == 2 ? 16 : 32;
  const int seg = nrow == 2 ? lane >> 4 : 0;
  const int q = lane - seg * width;  // this lane's position in its row
  const int64_t i = (int64_t)ta.x + seg;
  const int32_t rs = seg ? ta.z : ta.y, len = (seg || nrow == 1 ? ta.w : ta.z) - rs;
  const int dp = seg ? (tb.w >> 8) & 255 : tb.w & 255;
  if (DEBUG && __any_sync(FULL, len > width || (len > 0 && dp >= len))) {  // warp-uniform
    if (lane == 0) atomicOr(m.err, ERR_STAR);
    return;
  }
  const bool has = q < len;
  const T kc = kc_of<T>(f), kmu = kmu_of<T>(f), kmass = kmass_of<T>(f);
  const StabK<T> sk = stab_k<T>(sc);
  const T kg = (T)(-1.0 / 24.0);

  // 1. entry records
  {
    const int j = has ? m.col_idx[rs + q] : 0;
    wait_for_previous();
    if (DEBUG && has && (j < 0 || j >= m.n)) atomicOr(m.err, ERR_BAD_INDEX);
    const int dl = seg * width + (len > 0 ? dp : 0);  // the diagonal's lane
    V3<T> d, u;
    if constexpr (P == NSI_FP64) {
      V3<double> x{0.0, 0.0, 0.0}, v{0.0, 0.0, 0.0};
      if (has && (!DEBUG || (j >= 0 && j < m.n))) {
        const double* r = static_cast<const double*>(m.rec) + 8 * (int64_t)j;
        load_record<true>(r, x.x, x.y, x.z);
        load_record<true>(r + 4, v.x, v.y, v.z);
      }
      const double xi = __shfl_sync(FULL, x.x, dl), yi = __shfl_sync(FULL, x.y, dl), zi = __shfl_sync(FULL, x.z, dl);
      d = {x.x - xi, x.y - yi, x.z - zi};
      u = v;
    } else {
      uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
      // (one 256-bit load instead of two 128-bit ones: 0.944 against 0.954 ms
      // mixed64, 0.733 against 0.755 mixed32)
      if (has && (!DEBUG || (j >= 0 && j < m.n)))
        load_record<true>(static_cast<const unsigned*>(m.rec) + 8 * (int64_t)j, a, b);
      const V3<float> hj{__uint_as_float(a.x), __uint_as_float(a.y), __uint_as_float(a.z)};
      const V3<float> lj = record_lo(__uint_as_float(b.z), __uint_as_float(b.w));
      const V3<float> hi{__shfl_sync(FULL, hj.x, dl), __shfl_sync(FULL, hj.y, dl), __shfl_sync(FULL, hj.z, dl)};
      const V3<float> li{__shfl_sync(FULL, lj.x, dl), __shfl_sync(FULL, lj.y, dl), __shfl_sync(FULL, lj.z, dl)};
      d = add(sub(hj, hi), sub(lj, li));
      u = {__uint_as_float(a.w), __uint_as_float(b.x), __uint_as_float(b.y)};
    }
    er[lane] = T4<T>{d.x, d.y, d.z, u.x};
    eu[lane] = T2<T>{u.y, u.z};
  }
  __syncwarp();

  // 2-3. elements in chunks of 64, then the entries' sums
  const int dp0 = __shfl_sync(FULL, dp, 0), dp1 = __shfl_sync(FULL, dp, 16);
  const int len0 = __shfl_sync(FULL, len, 0), len1 = __shfl_sync(FULL, len, 16);
  // an entry's sums (the few elements of its edge) in plain T; the row
  // totals below are compensated in mixed64
  T sA = T(0), dA = T(0), dB = T(0);  // dA, dB: det of this lane's elements of the task's rows
  T K[9], G[3] = {T(0), T(0), T(0)};
#pragma unroll
  for (int c = 0; c < 9; ++c) K[c] = T(0);
  for (int c0 = 0; c0 < nel; c0 += CH) {
#pragma unroll
    for (int w = 0; w < 6; ++w) mk[w * 32 + lane] = 0u;
    __syncwarp();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int slot = half * 32 + lane;
      const int t = c0 + slot;
      if (t < nel) {
        const int es = (nrow == 2 && s0 + t >= s1) ? 1 : 0;  // the element's row
        const int eb = es * width;
        const int edp = es ? dp1 : dp0;
        const unsigned w = c0 == 0 ? wpre[half] : star_word[s0 + t];
        const int pa = w & 31, pb = (w >> 5) & 31, pc = (w >> 10) & 31;
        const int elen = es ? len1 : len0;
        if (DEBUG && (pa >= elen || pb >= elen || pc >= elen || elen > width)) {
          atomicOr(m.err, ERR_STAR);  // the element is left out
          continue;
        }
        V3<T> d1, d2, d3, di, u1, u2, u3, ui;
        auto rd = [&](int l, V3<T>& d, V3<T>& u) {
          const T4<T> a = er[l];
          const T2<T> b = eu[l];
          d = {a.x, a.y, a.z};
          u = {a.w, b.x, b.y};
        };
        rd(eb + pa, d1, u1);
        rd(eb + pb, d2, u2);
        rd(eb + pc, d3, u3);
        rd(eb + edp, di, ui);
        const V3<T> c1 = cross(d2, d3), c2 = cross(d3, d1), c3 = cross(d1, d2);
        const T det = dot(d1, c1);
        const V3<T> ci{-(c1.x + c2.x + c3.x), -(c1.y + c2.y + c3.y), -(c1.z + c2.z + c3.z)};
        const T rdet = rcp_fast(det);
        const T kv = kmu * rdet;
        const V3<T> us = add(add(ui, u1), add(u2, u3));
        T h, sh;
        tau_lengths(det, dot(us, us), h, sh);
        const T fs = sk.ks * rcp_fast(h * fma_of(sk.krh, sh, sk.k4mu));
        const T kd = fma_of(sk.kr48 * sh, rdet, kv);
        const T as = fs * dot(us, ci), ai = fs * dot(ui, ci), a1 = fs * dot(u1, ci), a2 = fs * dot(u2, ci),
                a3 = fs * dot(u3, ci);
        // w + v: Galerkin convection and viscosity plus the SUPG vector
        V3<T> wv;
        wv.x = kc * (ui.x + us.x) + kv * ci.x + (as * us.x + ai * ui.x + a1 * u1.x + a2 * u2.x + a3 * u3.x);
        wv.y = kc * (ui.y + us.y) + kv * ci.y + (as * us.y + ai * ui.y + a1 * u1.y + a2 * u2.y + a3 * u3.y);
        wv.z = kc * (ui.z + us.z) + kv * ci.z + (as * us.z + ai * ui.z + a1 * u1.z + a2 * u2.z + a3 * u3.z);
        T4<T>* r = el + slot;
        r[0] = T4<T>{ci.x, ci.y, ci.z, kv};
        r[CH] = T4<T>{c1.x, c1.y, c1.z, dot(wv, c1)};
        r[2 * CH] = T4<T>{c2.x, c2.y, c2.z, dot(wv, c2)};
        r[3 * CH] = T4<T>{c3.x, c3.y, c3.z, dot(wv, c3)};
        ekd[slot] = kd;
        if (es) dB += det;
        else dA += det;
        const unsigned bit = 1u << lane;
        atomicOr(&mk[(0 * 2 + half) * 32 + eb + pa], bit);
        atomicOr(&mk[(1 * 2 + half) * 32 + eb + pb], bit);
        atomicOr(&mk[(2 * 2 + half) * 32 + eb + pc], bit);
      }
    }
    __syncwarp();
    if (has && q != dp) {
      const unsigned long long m1 = mk[2 * 32 + lane] | ((unsigned long long)mk[3 * 32 + lane] << 32);
      const unsigned long long m2 = mk[4 * 32 + lane] | ((unsigned long long)mk[5 * 32 + lane] << 32);
      unsigned long long bits = mk[0 * 32 + lane] | ((unsigned long long)mk[1 * 32 + lane] << 32) | m1 | m2;
      while (bits) {
        const int e = __ffsll((long long)bits) - 1;
        bits &= bits - 1;
        const int k = ((m1 >> e) & 1ull) ? 2 : ((m2 >> e) & 1ull) ? 3 : 1;
        const T4<T> r0v = el[e], rk = el[k * CH + e];
        sA += rk.w;
        const T kv = r0v.w, kd = ekd[e];
        const T ri[3] = {r0v.x, r0v.y, r0v.z}, c[3] = {rk.x, rk.y, rk.z};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b2 = 0; b2 < 3; ++b2)
            K[3 * a + b2] = fma_of(kv * c[a], ri[b2], fma_of(kd * ri[a], c[b2], K[3 * a + b2]));
        G[0] += ri[0];
        G[1] += ri[1];
        G[2] += ri[2];
      }
    }
    __syncwarp();
  }

  // 4. row totals: every lane's sums (a lane without an off-diagonal entry has
  // zeros) to shared memory (the element records' space, free now), where the
  // row's lanes 0-13 each add one value up over the row's entries (mixed64:
  // compensated; else in pairs, neighbours first: one after the other the
  // diagonal's rounding in mixed32 is a sixth larger); A's and det's go to all of the row's
  // lanes
  constexpr int NV = 14, ST = 15;  // K, G, A + S, det; an odd stride: no bank conflicts
  T* red = reinterpret_cast<T*>(el);
#pragma unroll
  for (int c = 0; c < 9; ++c) red[lane * ST + c] = K[c];
#pragma unroll
  for (int c = 0; c < 3; ++c) red[lane * ST + 9 + c] = G[c];
  red[lane * ST + 12] = sA;
  {  // two rows of 16 lanes: a row's elements are on all 32
    const T a = dA + __shfl_xor_sync(FULL, dA, 16), b = dB + __shfl_xor_sync(FULL, dB, 16);
    red[lane * ST + 13] = nrow == 2 ? (seg ? b : a) : dA;
  }
  __syncwarp();
  Acc<P> tot;
  tot.zero();
  if (q < NV) {
    const T* x = red + seg * width * ST + q;
    if constexpr (P == NSI_MIXED_F32_ACC64) {
      for (int r = 0; r < width; ++r) tot.add(x[r * ST]);
    } else {
      tot.v = pair_sum<16, ST>(x);
      if (width == 32) tot.v += pair_sum<16, ST>(x + 16 * ST);
    }
  }
  auto from = [&](int l) {
    Acc<P> a;
    if constexpr (P == NSI_MIXED_F32_ACC64) {
      a.hi = __shfl_sync(FULL, tot.hi, seg * width + l);
      a.lo = __shfl_sync(FULL, tot.lo, seg * width + l);
    } else {
      a.v = __shfl_sync(FULL, tot.v, seg * width + l);
    }
    return a;
  };
  const Acc<P> tA = from(12), tD = from(13);

  // 5. write-out: every lane its own entry; then the row's lanes 0-11 the
  // components of the diagonal block and of the diagonal's G (the totals they
  // hold), lanes 12-14 the right-hand side: each one value, in one store
  Out* A = static_cast<Out*>(Auu);
  Out* Go = static_cast<Out*>(Gv);
  Out* Rh = static_cast<Out*>(rhs);
  if (has && q != dp) {
    const int64_t g = (int64_t)rs + q;
#pragma unroll
    for (int c = 0; c < 9; ++c) A[c * m.nnz + g] = (Out)(c % 4 == 0 ? sA + K[c] : K[c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) Go[c * m.nnz + g] = (Out)(G[c] * kg);
  }
  if (len > 0 && q < 15) {  // (a row's lanes number 16 or 32)
    // (the factor's own rounding would be the same in every row's mass; mixed32
    // keeps it, its values are rounded to float once more anyway)
    Acc<P> mass = acc_scale<P>(tD, kmass);
    if constexpr (P == NSI_MIXED_F32_ACC64) mass.lo = fmaf(sk.kml, tD.hi, mass.lo);
    else if constexpr (P == NSI_FP64) mass.v = fma(sk.kml, tD.v, mass.v);
    Acc<P> x;
    Out* at;
    if (q < 12) {  // A(i,i)[a][b] = delta_ab (lumped mass - sum of the row's A + S) - sum of K[a][b]; G(i,i) = G's / 3
      x = acc_scale<P>(tot, q < 9 ? T(-1) : kg / T(3));
      if (q < 9 && q % 4 == 0) {
        Acc<P> y = mass;
        if constexpr (P == NSI_MIXED_F32_ACC64) {
          y.add(-tA.hi);
          y.lo -= tA.lo;
          y.add(x.hi);
          y.lo += x.lo;
        } else {
          y.v = (mass.v - tA.v) + x.v;
        }
        x = y;
      }
      at = (q < 9 ? A + q * m.nnz : Go + (q - 9) * m.nnz) + rs + dp;
    } else {  // rhs[k][i] = lumped mass * u^n_k
      const T* un = static_cast<const T*>(q == 12 ? f.un[0] : q == 13 ? f.un[1] : f.un[2]);
      x = acc_scale<P>(mass, __ldg(un + i));
      at = Rh + (q - 12) * m.n + i;
    }
    store_acc(at, x);
  } else if (q == 0 && len == 0) {  // a node in no element: zero right-hand side
    Rh[i] = Out(0);
    Rh[m.n + i] = Out(0);
    Rh[2 * m.n + i] = Out(0);
  }
}

// The stabilised block of listed rows (or of every row when `rows` is null),
// one thread per row in double whatever the handle's precision: the mixed
// modes' rows touching badly shaped elements, and whole meshes without an
// edge-fan map.  Each off-diagonal entry (i, j) sums the row's elements that
// contain j (node i first, the others in an even order so that det > 0), the
// diagonal block follows from the row totals as in the fan kernel.
template <int P>
__global__ void __launch_bounds__(64) stab_rows_kernel(MeshView m, FieldView f, StabConst sc, void* Auu, void* Gv,
                                                       void* rhs, const int32_t* rows, const int32_t* ptr,
                                                       const uint32_t* inc, int64_t count) {
  using Out = typename Prec<P>::Out;
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= count) return;
  const int64_t i = rows ? rows[r] : r;
  const int32_t rs = m.row_ptr[i], len = m.row_ptr[i + 1] - rs;
  const int32_t* cols = m.col_idx + rs;
  auto coord = [&](int64_t j) {
    if constexpr (P == NSI_FP64) {
      const D4 x = m.xyz64[j];
      return V3<double>{x.x, x.y, x.z};
    } else {
      const float4 h = m.xyz_hi[j], l = m.xyz_lo[j];
      return V3<double>{(double)h.x + (double)l.x, (double)h.y + (double)l.y, (double)h.z + (double)l.z};
    }
  };
  auto vel = [&](const void* const* comp, int64_t j) {
    if constexpr (P == NSI_FP64) return load_vec<double>(comp, j);
    else {
      const V3<float> w = load_vec<float>(comp, j);
      return V3<double>{w.x, w.y, w.z};
    }
  };
  const int EVEN[4][3] = {{1, 2, 3}, {0, 3, 2}, {3, 0, 1}, {2, 1, 0}};
  const V3<double> xi = coord(i), ui = vel(f.u, i);
  const StabK<double> sk = stab_k<double>(sc);
  struct El {
    int v[3];
    V3<double> c[3], ci, u[3];
    double det;
  };
  auto element = [&](int32_t t) {
    El el;
    const int64_t e = inc[t] >> 2;
    const int a = (int)(inc[t] & 3u);
    const int4 v4 = m.lnods[e];
    const int v[4] = {v4.x, v4.y, v4.z, v4.w};
    V3<double> d[3];
    for (int b = 0; b < 3; ++b) {
      el.v[b] = v[EVEN[a][b]];
      d[b] = sub(coord(el.v[b]), xi);
      el.u[b] = vel(f.u, el.v[b]);
    }
    el.c[0] = cross(d[1], d[2]);
    el.c[1] = cross(d[2], d[0]);
    el.c[2] = cross(d[0], d[1]);
    el.det = dot(d[0], el.c[0]);
    el.ci = V3<double>{-(el.c[0].x + el.c[1].x + el.c[2].x), -(el.c[0].y + el.c[1].y + el.c[2].y),
                       -(el.c[0].z + el.c[1].z + el.c[2].z)};
    return el;
  };
  double detsum = 0.0;
  for (int32_t t = ptr[r]; t < ptr[r + 1]; ++t) detsum += element(t).det;
  Out* A = static_cast<Out*>(Auu) + rs;
  Out* G = static_cast<Out*>(Gv) + rs;
  double sa = 0.0, sK[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, sg[3] = {0.0, 0.0, 0.0};
  int dpos = -1;
  for (int q = 0; q < len; ++q) {
    const int32_t j = cols[q];
    if (j == i) {
      dpos = q;
      continue;
    }
    double a = 0.0, K[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, g[3] = {0.0, 0.0, 0.0};
    for (int32_t t = ptr[r]; t < ptr[r + 1]; ++t) {
      const int4 v4 = m.lnods[inc[t] >> 2];
      if (v4.x != j && v4.y != j && v4.z != j && v4.w != j) continue;
      const El el = element(t);
      const int b = el.v[0] == j ? 0 : el.v[1] == j ? 1 : 2;
      const double kv = f.kmu / el.det;
      const V3<double> us2{2.0 * ui.x + el.u[0].x + el.u[1].x + el.u[2].x,
                           2.0 * ui.y + el.u[0].y + el.u[1].y + el.u[2].y,
                           2.0 * ui.z + el.u[0].z + el.u[1].z + el.u[2].z};
      const V3<double> w{f.kc * us2.x + kv * el.ci.x, f.kc * us2.y + kv * el.ci.y, f.kc * us2.z + kv * el.ci.z};
      a += dot(w, el.c[b]);
      a += stab_terms<double>(el.ci, el.c[b], el.det, ui, el.u[0], el.u[1], el.u[2], sk, f.kmu, K);
      g[0] += el.ci.x;
      g[1] += el.ci.y;
      g[2] += el.ci.z;
    }
    sa += a;
    for (int c = 0; c < 9; ++c) {
      sK[c] += K[c];
      A[c * m.nnz + q] = (Out)((c % 4 == 0 ? a : 0.0) + K[c]);
    }
    for (int d = 0; d < 3; ++d) {
      G[d * m.nnz + q] = (Out)(-g[d] / 24.0);
      sg[d] += g[d];
    }
  }
  if (dpos >= 0) {
    const double dm = f.kmass * detsum - sa;
    for (int c = 0; c < 9; ++c) A[c * m.nnz + dpos] = (Out)((c % 4 == 0 ? dm : 0.0) - sK[c]);
    for (int d = 0; d < 3; ++d) G[d * m.nnz + dpos] = (Out)(-sg[d] / 72.0);
  }
  const V3<double> un = vel(f.un, i);
  Out* Rh = static_cast<Out*>(rhs);
  Rh[i] = (Out)(f.kmass * detsum * un.x);
  Rh[m.n + i] = (Out)(f.kmass * detsum * un.y);
  Rh[2 * m.n + i] = (Out)(f.kmass * detsum * un.z);
}

// --------------------------------------------- batched edge-fan kernel ---
struct BatchItem {
  MeshView m;
  FieldView f;
  OutView o;
  int64_t block0;  // first global fan block of this mesh
};
struct BatchArgs {
  int32_t count;
  int64_t total_blocks;
  BatchItem item[NSI_MAX_BATCH];
};

// many meshes, edge-fan variant: a persistent grid strides over the fan
// blocks of all meshes (item.block0 counts fan blocks here)
template <int P>
__global__ void __launch_bounds__(FAN_BLOCK) batched_fan_kernel(const __grid_constant__ BatchArgs args) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (int64_t b = blockIdx.x; b < args.total_blocks; b += gridDim.x) {
    int lo = 0, hi = args.count - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (args.item[mid].block0 <= b) lo = mid;
      else hi = mid - 1;
    }
    const BatchItem& it = args.item[lo];
    fan_block<P, false>(it.m, it.f, it.o, b - it.block0, smem_raw);
    __syncthreads();  // the next block reuses the shared records
  }
}

// ----------------------------------------------------------- VJP kernel ---
// One element's adjoint terms in arithmetic C (edge vectors d1, d2, d3 from
// node 0; velocities u and adjoint weights w of the 4 nodes):
//   g[m] = sum_a w_a A_e[a][m] + rho/120 sum_k (W_k + w_{m,k}) Gu[k]
//   returned: 1/(6 det) sum_{a,k} w_{a,k} c_a . Gu[k]   (the grad_mu term)
// with W = sum_a w_a and Gu[k][l] = sum_b u_{b,k} c_b[l] = det du^k/dx_l.
// The viscosity gradient is one sum of terms of both signs over all elements,
// so a term's rounding shows in it multiplied by the sum's cancellation: the
// terms keep this form.  (With 3x3 moments, Q = sum_a w_a c_a^T and the term Q . Gu,
// an FP64 call took 300 operations per element instead of 380, and grad_mu of
// cancelling weights moved by 1e-14 and more.)
template <typename C>
__device__ __forceinline__ C vjp_element(const V3<C>& d1, const V3<C>& d2, const V3<C>& d3, const V3<C> (&u)[4],
                                         const V3<C> (&w)[4], C kc, C kmu, C kmass, V3<C> (&g)[4]) {
  V3<C> c[4];
  c[1] = cross(d2, d3);
  c[2] = cross(d3, d1);
  c[3] = cross(d1, d2);
  const C det = dot(d1, c[1]);
  c[0] = {-(c[1].x + c[2].x + c[3].x), -(c[1].y + c[2].y + c[3].y), -(c[1].z + c[2].z + c[3].z)};
  const V3<C> S = add(add(u[0], u[1]), add(u[2], u[3]));
  const V3<C> Ws = add(add(w[0], w[1]), add(w[2], w[3]));
  const C kv = kmu * rcp(det);
  const C km = det * kmass;
  V3<C> Gu[3];
  const C uk[4][3] = {{u[0].x, u[0].y, u[0].z}, {u[1].x, u[1].y, u[1].z}, {u[2].x, u[2].y, u[2].z},
                      {u[3].x, u[3].y, u[3].z}};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    Gu[k] = {C(0), C(0), C(0)};
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      Gu[k].x += uk[b][k] * c[b].x;
      Gu[k].y += uk[b][k] * c[b].y;
      Gu[k].z += uk[b][k] * c[b].z;
    }
  }
#pragma unroll
  for (int mm = 0; mm < 4; ++mm) {
    V3<C> acc = {C(0), C(0), C(0)};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      C Aam = kc * dot(add(S, u[a]), c[mm]) + kv * dot(c[a], c[mm]);
      if (a == mm) Aam += km;
      acc.x += w[a].x * Aam;
      acc.y += w[a].y * Aam;
      acc.z += w[a].z * Aam;
    }
    const C wk[3] = {Ws.x + w[mm].x, Ws.y + w[mm].y, Ws.z + w[mm].z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      acc.x += kc * wk[k] * Gu[k].x;
      acc.y += kc * wk[k] * Gu[k].y;
      acc.z += kc * wk[k] * Gu[k].z;
    }
    g[mm] = acc;
  }
  C s = C(0);
#pragma unroll
  for (int a = 0; a < 4; ++a) s += w[a].x * dot(c[a], Gu[0]) + w[a].y * dot(c[a], Gu[1]) + w[a].z * dot(c[a], Gu[2]);
  return s * (C)(1.0 / 6.0) * rcp(det);
}

// true if element e is marked in the bit mask of badly shaped elements
__device__ __forceinline__ bool marked(const uint32_t* __restrict__ mask, int64_t e) {
  return mask && ((mask[e >> 5] >> (e & 31)) & 1u);
}

// The adjoint, one element per thread, in the handle's arithmetic; the
// elements marked in `skip` (badly shaped, mixed modes) are left to
// vjp_exact_kernel.  grad_mu's block sums are added by atomics, in FP64 one for
// every cluster of VJP_CLUSTER blocks: an addition rounds at the size of the
// running sum, which weights of both signs let wander far from the result (on
// the worst of 12 random 30x28x33 boxes repeats of one call differ by 1.4e-14
// with an addition per block, by 5.5e-15 with one per four).  Four blocks cost
// nothing there (148 us) and 1.5% at 750,000 tets (564 us); eight cost 6% at
// both, as a cluster begins when all its blocks fit.
constexpr int VJP_CLUSTER = 4;
// A block's first arrival only says that it has begun; it may end after its
// last one (a wait is for the threads that have not ended).
__device__ __forceinline__ void cluster_begun() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
template <int P>
__global__ void __launch_bounds__(256) vjp_kernel(MeshView m, FieldView f, const void* __restrict__ wv, void* gu,
                                                  double* gmu, const uint32_t* __restrict__ skip) {
  using T = typename Prec<P>::T;
  __shared__ T red[32];
  [[maybe_unused]] __shared__ double part[VJP_CLUSTER];
  [[maybe_unused]] const int rank = (int)blockIdx.x % VJP_CLUSTER;
  if constexpr (P == NSI_FP64) cluster_begun();
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  T my_mu = T(0);
  if (e < m.E && !marked(skip, e)) {
    const int4 q = m.lnods[e];
    const int v[4] = {q.x, q.y, q.z, q.w};
    const T* W = static_cast<const T*>(wv);
    NodeX<P> X[4];
    V3<T> u[4], w[4], g[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      X[a].load(m, v[a]);
      u[a] = load_vec<T>(f.u, v[a]);
      w[a] = {W[v[a]], W[m.n + v[a]], W[2 * m.n + v[a]]};
    }
    my_mu = vjp_element(X[1].minus(X[0]), X[2].minus(X[0]), X[3].minus(X[0]), u, w, kc_of<T>(f), kmu_of<T>(f),
                           kmass_of<T>(f), g);
    T* gp = static_cast<T*>(gu);
#pragma unroll
    for (int mm = 0; mm < 4; ++mm) {
      atomicAdd(gp + v[mm], g[mm].x);
      atomicAdd(gp + m.n + v[mm], g[mm].y);
      atomicAdd(gp + 2 * m.n + v[mm], g[mm].z);
    }
  }
  // block reduction of the viscosity sensitivity
  for (int off = 16; off > 0; off >>= 1) my_mu += __shfl_down_sync(0xffffffffu, my_mu, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = my_mu;
  __syncthreads();
  T s = T(0);
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : T(0);
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  }
  if constexpr (sizeof(T) == 4) {
    if (threadIdx.x == 0) atomicAdd(gmu, __longlong_as_double(f32_to_f64_bits(s)));
  } else {
    // the cluster's block sums, by its first block in rank order, the rounding
    // errors kept
    cluster_wait();  // the first block has begun
    if (threadIdx.x == 0) *cooperative_groups::this_cluster().map_shared_rank(&part[rank], 0) = s;
    __syncwarp();
    cluster_arrive();
    if (rank != 0) return;
    cluster_wait();
    if (threadIdx.x == 0) {
      double hi = 0.0, lo = 0.0;
      for (int k = 0; k < VJP_CLUSTER; ++k) {
        const double t = hi + part[k], c = t - hi;
        lo += (hi - (t - c)) + (part[k] - c);
        hi = t;
      }
      atomicAdd(gmu, hi + lo);
    }
  }
}

// the badly shaped elements of the mixed modes in double (their determinant
// in float would carry about their shape ratio times the float rounding)
template <int P>
__global__ void __launch_bounds__(64) vjp_exact_kernel(MeshView m, FieldView f, const void* __restrict__ wv, void* gu,
                                                        double* gmu, const int32_t* __restrict__ list, int64_t count) {
  using T = typename Prec<P>::T;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count) return;
  const int64_t e = list[t];
  const int4 q = m.lnods[e];
  const int v[4] = {q.x, q.y, q.z, q.w};
  const void* wc[3] = {static_cast<const T*>(wv), static_cast<const T*>(wv) + m.n, static_cast<const T*>(wv) + 2 * m.n};
  V3<double> X[4], u[4], w[4], g[4];
  for (int a = 0; a < 4; ++a) {
    X[a] = coord64<P>(m, v[a]);
    u[a] = vec64<T>(f.u, v[a]);
    w[a] = vec64<T>(wc, v[a]);
  }
  const double mu = vjp_element(sub(X[1], X[0]), sub(X[2], X[0]), sub(X[3], X[0]), u, w, f.kc, f.kmu, f.kmass, g);
  T* gp = static_cast<T*>(gu);
  for (int mm = 0; mm < 4; ++mm) {
    atomicAdd(gp + v[mm], (T)g[mm].x);
    atomicAdd(gp + m.n + v[mm], (T)g[mm].y);
    atomicAdd(gp + 2 * m.n + v[mm], (T)g[mm].z);
  }
  atomicAdd(gmu, mu);
}


// ----------------------------------------------------- residual kernel ---
// reciprocal of a determinant: IEEE in float; double by rcp_fast (its error is
// below the double's rounding, and the FP64 pipe bounds the FP64 kernels)
__device__ __forceinline__ float rcp_det(float x) { return rcp(x); }
__device__ __forceinline__ double rcp_det(double x) { return rcp_fast(x); }

// m[k] = sum_b v_{b,k} c_b over the element's nodes: v = u gives det grad u_k
// (by the differences to node 0, of as many operations, R was up to 7% further
// from 64 bits on coarse meshes)
template <typename C>
__device__ __forceinline__ V3<C> moment(C v0, C v1, C v2, C v3, const V3<C> (&c)[4]) {
  return {fma_of(v3, c[3].x, fma_of(v2, c[2].x, fma_of(v1, c[1].x, v0 * c[0].x))),
          fma_of(v3, c[3].y, fma_of(v2, c[2].y, fma_of(v1, c[1].y, v0 * c[0].y))),
          fma_of(v3, c[3].z, fma_of(v2, c[2].z, fma_of(v1, c[1].z, v0 * c[0].z)))};
}
template <typename C>
__device__ __forceinline__ void moments(const V3<C> (&v)[4], const V3<C> (&c)[4], V3<C> (&m)[3]) {
  m[0] = moment(v[0].x, v[1].x, v[2].x, v[3].x, c);
  m[1] = moment(v[0].y, v[1].y, v[2].y, v[3].y, c);
  m[2] = moment(v[0].z, v[1].z, v[2].z, v[3].z, c);
}
template <typename C>
__device__ __forceinline__ V3<C> axpy(C a, const V3<C>& x, const V3<C>& y) {
  return {fma_of(a, x.x, y.x), fma_of(a, x.y, y.y), fma_of(a, x.z, y.z)};
}

// R[k][v_a] += sum_b A_e[a][b] u_b[k] - rho |T_e| / (4 dt) u^n_a[k]: the
// residual of the assembled system without forming A (element per thread).  The
// sum over b is a product with Gu[k] = sum_b u_{b,k} c_b:
//   (rho/120 (S + u_a) + mu/(6 det) c_a) . Gu[k],  S = sum_b u_b.  (150 operations per
// element instead of 250 with every entry: 166,320 tets in FP64 93 -> 62 us.)
// un: nullptr where u^n is u (the lumped terms cancel).
template <typename C>
__device__ __forceinline__ void residual_element(const V3<C>& d1, const V3<C>& d2, const V3<C>& d3,
                                                 const V3<C> (&u)[4], const V3<C>* un, C kc, C kmu, C kmass,
                                                 V3<C> (&r)[4]) {
  V3<C> c[4];
  c[1] = cross(d2, d3);
  c[2] = cross(d3, d1);
  c[3] = cross(d1, d2);
  const C det = dot(d1, c[1]);
  c[0] = {-(c[1].x + c[2].x + c[3].x), -(c[1].y + c[2].y + c[3].y), -(c[1].z + c[2].z + c[3].z)};
  const V3<C> S = add(add(u[0], u[1]), add(u[2], u[3]));
  const C kv = kmu * rcp_det(det);
  const C km = det * kmass;
  const V3<C> kS = {kc * S.x, kc * S.y, kc * S.z};
  V3<C> Gu[3];
  moments(u, c, Gu);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const V3<C> E = axpy(kv, c[a], axpy(kc, u[a], kS));
    r[a] = {dot(E, Gu[0]), dot(E, Gu[1]), dot(E, Gu[2])};
    if (un) r[a] = axpy(km, sub(u[a], un[a]), r[a]);
  }
}

template <int P>
__global__ void __launch_bounds__(256) residual_kernel(MeshView m, FieldView f, void* rout,
                                                       const uint32_t* __restrict__ skip) {
  using T = typename Prec<P>::T;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.E || marked(skip, e)) return;
  const int4 q = m.lnods[e];
  const int v[4] = {q.x, q.y, q.z, q.w};
  NodeX<P> X[4];
  V3<T> u[4], un[4], r[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    X[a].load(m, v[a]);
    u[a] = load_vec<T>(f.u, v[a]);
  }
  const bool moving = f.un[0] != f.u[0] || f.un[1] != f.u[1] || f.un[2] != f.u[2];  // launch-uniform
  if (moving) {
#pragma unroll
    for (int a = 0; a < 4; ++a) un[a] = load_vec<T>(f.un, v[a]);
  }
  const V3<T> d1 = X[1].minus(X[0]), d2 = X[2].minus(X[0]), d3 = X[3].minus(X[0]);
  if (moving) residual_element<T>(d1, d2, d3, u, un, kc_of<T>(f), kmu_of<T>(f), kmass_of<T>(f), r);
  else residual_element<T>(d1, d2, d3, u, nullptr, kc_of<T>(f), kmu_of<T>(f), kmass_of<T>(f), r);
  T* R = static_cast<T*>(rout);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    atomicAdd(R + v[a], r[a].x);
    atomicAdd(R + m.n + v[a], r[a].y);
    atomicAdd(R + 2 * m.n + v[a], r[a].z);
  }
}

template <int P>
__global__ void __launch_bounds__(64) residual_exact_kernel(MeshView m, FieldView f, void* rout,
                                                             const int32_t* __restrict__ list, int64_t count) {
  using T = typename Prec<P>::T;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count) return;
  const int64_t e = list[t];
  const int4 q = m.lnods[e];
  const int v[4] = {q.x, q.y, q.z, q.w};
  V3<double> X[4], u[4], un[4], r[4];
  for (int a = 0; a < 4; ++a) {
    X[a] = coord64<P>(m, v[a]);
    u[a] = vec64<T>(f.u, v[a]);
    un[a] = vec64<T>(f.un, v[a]);
  }
  residual_element<double>(sub(X[1], X[0]), sub(X[2], X[0]), sub(X[3], X[0]), u, un, f.kc, f.kmu, f.kmass, r);
  T* R = static_cast<T*>(rout);
  for (int a = 0; a < 4; ++a) {
    atomicAdd(R + v[a], (T)r[a].x);
    atomicAdd(R + m.n + v[a], (T)r[a].y);
    atomicAdd(R + 2 * m.n + v[a], (T)r[a].z);
  }
}

// --------------------------------------------- partition exchange ---
// The interface-row sum of a mesh split over ranks (disjoint element sets):
// values of chosen entries packed into an exchange buffer, and received
// values added into the owner's rows.
constexpr int XCH_MAX_COMP = 4;
struct CompPtrs {
  void* p[XCH_MAX_COMP];
};
// dst[k][c] = comp[c][idx[k]] (dst row-major [count][ncomp])
template <typename V>
__global__ void __launch_bounds__(256) gather_values_kernel(CompPtrs src, int ncomp, const int32_t* __restrict__ idx,
                                                            int64_t count, V* __restrict__ dst) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int32_t i = idx[k];
  for (int c = 0; c < ncomp; ++c) dst[k * ncomp + c] = static_cast<const V*>(src.p[c])[i];
}
// comp[c][idx[k]] += src[k][c]; the positions of one call are distinct
template <typename V>
__global__ void __launch_bounds__(256) add_values_kernel(CompPtrs dst, int ncomp, const int32_t* __restrict__ idx,
                                                         int64_t count, const V* __restrict__ src) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int32_t i = idx[k];
  for (int c = 0; c < ncomp; ++c) static_cast<V*>(dst.p[c])[i] += src[k * ncomp + c];
}

// ----------------------------------------------------------- launchers ---
template <int P>
static nsi_status zero_outputs(const NsiHandle* h, const OutView& o, cudaStream_t s) {
  using Out = typename Prec<P>::Out;
  NSI_CUDA(cudaMemsetAsync(o.A, 0, sizeof(Out) * h->nnz, s));
  NSI_CUDA(cudaMemsetAsync(o.G, 0, sizeof(Out) * 3 * h->nnz, s));
  NSI_CUDA(cudaMemsetAsync(o.rhs, 0, sizeof(Out) * 3 * h->n, s));
  return NSI_OK;
}

// listed rows by one block each
template <int P>
static nsi_status launch_rows64(NsiHandle* h, const FieldView& f, int mode, const RowOut& o, const int32_t* rows,
                                const int32_t* ptr, const uint32_t* inc, int64_t count, cudaStream_t s) {
  const auto kernel = mode == 0 ? rows64_kernel<P, 0> : mode == 1 ? rows64_kernel<P, 1> : rows64_kernel<P, 2>;
  NSI_CUDA(launch_early(kernel, count, ROW_THREADS, 0, s, view_of(h), f, o, rows, ptr, inc));
  return check_launch("rows64_kernel");
}

// After an assembly, time step or nodal outputs: the long rows (after a row
// gather), and in a mixed mode the rows listed at create for badly shaped
// elements, recomputed in double (nothing if there are none; the time step's A
// does not depend on the determinant and stays).  (Run side by side, the few
// rows of the first kind wait for the FP64 pipe that the others fill: a pipe's
// assembly 121 us, one after the other 112.)
template <int P>
static nsi_status fix_rows(NsiHandle* h, const FieldView& f, int mode, const RowOut& out, bool gathered,
                           cudaStream_t s) {
  nsi_status st = NSI_OK;
  if (gathered && h->long_rows > 0)
    st = launch_rows64<P>(h, f, mode, out, h->long_list, h->long_ptr, h->long_inc, h->long_rows, s);
  if constexpr (P != NSI_FP64) {
    RowOut o = out;
    if (mode == 1) o.A = nullptr;
    if (!st && h->exact_rest > 0)
      st = launch_rows64<P>(h, f, mode, o, h->exact_list + h->exact_rows, h->exact_ptr + h->exact_rows, h->exact_inc,
                            h->exact_rest, s);
    if (!st && h->exact_rows > 0) st = launch_exact_rows<P>(h, f, mode, o, s);
  }
  return st;
}

// `rec` (nullptr: the handle's buffer) receives the row gather's per-call
// node records
template <int P>
static nsi_status assemble_core_p(NsiHandle* h, const FieldView& f, const OutView& o, int mode, cudaStream_t s,
                                  void* rec = nullptr) {
  MeshView m = view_of(h);
  if (rec) m.rec = rec;
  const int blk = 256;
  if (mode == NSI_SCATTER_ATOMIC) {
    nsi_status st = zero_outputs<P>(h, o, s);
    if (st) return st;
    if (h->E == 0) return NSI_OK;
    const int64_t grid = (h->E + blk - 1) / blk;
    if (h->ev_start) NSI_CUDA(cudaEventRecord(h->ev_start, s));
    // one atomic per value by default; the warp-aggregated variant issues 38%
    // fewer L2 reductions but about twice the instructions, slower on GB300
    // (100^3 cube: 2.19 against 2.60 ms mixed64, 1.81 against 1.89 mixed32,
    // 3.05 against 4.20 FP64); nsi_set_launch or the autotuner may select it
    if (h->atomic_agg) {
      if (h->debug) elem_kernel<P, true, true, true><<<grid, blk, 0, s>>>(m, f, o, nullptr, h->E, h->elem_pos);
      else elem_kernel<P, true, false, true><<<grid, blk, 0, s>>>(m, f, o, nullptr, h->E, h->elem_pos);
    } else {
      if (h->debug) elem_kernel<P, true, true><<<grid, blk, 0, s>>>(m, f, o, nullptr, h->E, h->elem_pos);
      else elem_kernel<P, true, false><<<grid, blk, 0, s>>>(m, f, o, nullptr, h->E, h->elem_pos);
    }
    if (h->ev_stop) NSI_CUDA(cudaEventRecord(h->ev_stop, s));
    return check_launch("elem_kernel (atomic)");
  }
  if (mode == NSI_SCATTER_COLOR) {
    nsi_status st = zero_outputs<P>(h, o, s);
    if (st) return st;
    if (h->ev_start) NSI_CUDA(cudaEventRecord(h->ev_start, s));
    for (int c = 0; c < h->n_colors; ++c) {
      const int64_t off = h->color_off[c], cnt = h->color_off[c + 1] - off;
      if (cnt == 0) continue;
      const int64_t grid = (cnt + blk - 1) / blk;
      if (h->debug) elem_kernel<P, false, true><<<grid, blk, 0, s>>>(m, f, o, h->color_elems + off, cnt, h->elem_pos);
      else elem_kernel<P, false, false><<<grid, blk, 0, s>>>(m, f, o, h->color_elems + off, cnt, h->elem_pos);
      nsi_status st2 = check_launch("elem_kernel (colour)");
      if (st2) return st2;
    }
    if (h->ev_stop) NSI_CUDA(cudaEventRecord(h->ev_stop, s));
    return NSI_OK;
  }
  // row gather
  if (!h->gather_ok) return fail(NSI_ERR_UNSUPPORTED, "row-gather mode not available for this mesh");
  nsi_status st = h->use_fan || h->packs() ? launch_pack<P>(h, f, rec, s) : NSI_OK;
  if (st) return st;
  if (h->use_fan) {
    const size_t fsm = FanSmem<P>::total(FAN_BLOCK);
    if (h->ev_start) NSI_CUDA(cudaEventRecord(h->ev_start, s));
    if (h->debug) fan_kernel<P, true><<<h->fan_blocks, FAN_BLOCK, fsm, s>>>(m, f, o);
    else fan_kernel<P, false><<<h->fan_blocks, FAN_BLOCK, fsm, s>>>(m, f, o);
    if (h->ev_stop) NSI_CUDA(cudaEventRecord(h->ev_stop, s));
    return check_launch("fan_kernel");
  }
  return launch_gather<P>(h, f, o, 0, h->n, rec, s);
}

template <int P>
static nsi_status assemble_p(NsiHandle* h, const FieldView& f, const OutView& o, int mode, cudaStream_t s) {
  nsi_status st = assemble_core_p<P>(h, f, o, mode, s);
  if (st) return st;
  const RowOut ro{nullptr, o.A, o.G, o.rhs, nullptr, nullptr, 0.0};
  return fix_rows<P>(h, f, 0, ro, mode == NSI_SCATTER_GATHER, s);
}

static nsi_status check_call(const NsiHandle* h, const NsiFields* f, const NsiOutputs* o) {
  if (!h || !f || !o) return fail(NSI_ERR_INVALID_ARG, "handle, fields or outputs is NULL");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if ((h->nnz > 0 && (!o->A_val || !o->G_val)) || !o->rhs)
    return fail(NSI_ERR_INVALID_ARG, "output pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  return NSI_OK;
}

static int resolve_mode(const NsiHandle* h, int mode) {
  if (mode == NSI_SCATTER_AUTO) mode = h->scatter;
  if (mode == NSI_SCATTER_AUTO) mode = h->gather_ok ? NSI_SCATTER_GATHER : NSI_SCATTER_ATOMIC;
  return mode;
}

static nsi_status assemble_dispatch(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, int mode,
                                    cudaStream_t s) {
  nsi_status st = check_call(h, f, o);
  if (st) return st;
  if (mode < NSI_SCATTER_AUTO || mode > NSI_SCATTER_GATHER) return fail(NSI_ERR_INVALID_ARG, "unknown scatter mode");
  mode = resolve_mode(h, mode);
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != h->device) return fail(NSI_ERR_INVALID_ARG, "current device differs from the handle's device");
  const FieldView fv = fields_of(f);
  const OutView ov{o->A_val, o->G_val, o->rhs};
  switch (h->precision) {
    case NSI_FP64: return assemble_p<NSI_FP64>(h, fv, ov, mode, s);
    case NSI_MIXED_F32_ACC64: return assemble_p<NSI_MIXED_F32_ACC64>(h, fv, ov, mode, s);
    default: return assemble_p<NSI_MIXED_F32_ACC32>(h, fv, ov, mode, s);
  }
}

// the time step and the nodal outputs: the node records, the row gather, then
// the rows that it leaves out
template <int P, bool NODAL>
static nsi_status step_p(NsiHandle* h, const FieldView& f, const StepView& o, cudaStream_t s) {
  nsi_status st = h->packs() ? launch_pack<P>(h, f, nullptr, s) : NSI_OK;
  if (!st) st = launch_step<P>(h, f, o, NODAL, s);
  if (st) return st;
  const RowOut ro{o.A_static, o.A, nullptr, o.rhs, o.dt_rho, o.mass_rho, o.kmr};
  return fix_rows<P>(h, f, NODAL ? 2 : 1, ro, true, s);
}

static nsi_status step_dispatch(NsiHandle* h, const NsiFields* f, const StepView& o, bool nodal, cudaStream_t s) {
  if (!h->gather_ok || h->n == 0)
    return h->n == 0 ? NSI_OK : fail(NSI_ERR_UNSUPPORTED, "the time-step kernels need the row-gather map");
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != h->device) return fail(NSI_ERR_INVALID_ARG, "current device differs from the handle's device");
  const FieldView fv = fields_of(f);
  switch (h->precision) {
    case NSI_FP64:
      return nodal ? step_p<NSI_FP64, true>(h, fv, o, s) : step_p<NSI_FP64, false>(h, fv, o, s);
    case NSI_MIXED_F32_ACC64:
      return nodal ? step_p<NSI_MIXED_F32_ACC64, true>(h, fv, o, s) : step_p<NSI_MIXED_F32_ACC64, false>(h, fv, o, s);
    default:
      return nodal ? step_p<NSI_MIXED_F32_ACC32, true>(h, fv, o, s) : step_p<NSI_MIXED_F32_ACC32, false>(h, fv, o, s);
  }
}

template <int P>
static nsi_status batched_core_p(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int count,
                                 cudaStream_t s);

template <int P>
static nsi_status batched_p(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int count,
                            cudaStream_t s) {
  nsi_status st = batched_core_p<P>(hs, fs, os, count, s);
  for (int k = 0; k < count && !st; ++k) {
    const RowOut ro{nullptr, os[k].A_val, os[k].G_val, os[k].rhs, nullptr, nullptr, 0.0};
    st = fix_rows<P>(hs[k], fields_of(&fs[k]), 0, ro, true, s);
  }
  return st;
}

template <int P>
static nsi_status batched_core_p(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int count,
                                 cudaStream_t s) {
  bool all_fan = true;
  for (int k = 0; k < count; ++k) all_fan &= hs[k]->use_fan;
  if (!all_fan) return launch_batched<P>(hs, fs, os, count, s);
  static BatchArgs args;  // host staging of the by-value kernel argument
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  args.count = count;
  int64_t fblocks = 0;
  for (int k = 0; k < count; ++k) {
    args.item[k].m = view_of(hs[k]);
    args.item[k].f = fields_of(&fs[k]);
    args.item[k].o = OutView{os[k].A_val, os[k].G_val, os[k].rhs};
    args.item[k].block0 = fblocks;
    fblocks += hs[k]->fan_blocks;
  }
  args.total_blocks = fblocks;
  if (fblocks == 0) return NSI_OK;
  for (int k = 0; k < count; ++k) {
    nsi_status st = launch_pack<P>(hs[k], args.item[k].f, nullptr, s);
    if (st) return st;
  }
  const size_t fsm = FanSmem<P>::total(FAN_BLOCK);
  int per_sm = 0, sms = 0, dev = 0;
  NSI_CUDA(cudaGetDevice(&dev));
  NSI_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  NSI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batched_fan_kernel<P>, FAN_BLOCK, fsm));
  const int64_t grid = std::min<int64_t>(fblocks, (int64_t)std::max(1, per_sm) * sms);
  batched_fan_kernel<P><<<grid, FAN_BLOCK, fsm, s>>>(args);
  return check_launch("batched_fan_kernel");
}

template <int P>
static nsi_status vjp_p(NsiHandle* h, const FieldView& f, const void* w, void* gu, double* gmu, cudaStream_t s) {
  using T = typename Prec<P>::T;
  NSI_CUDA(cudaMemsetAsync(gu, 0, sizeof(T) * 3 * h->n, s));
  NSI_CUDA(cudaMemsetAsync(gmu, 0, sizeof(double), s));
  if (h->E == 0) return NSI_OK;
  const int blk = 256;
  const int64_t grid = (h->E + blk - 1) / blk;
  if constexpr (P == NSI_FP64) {
    cudaLaunchAttribute cl;
    cl.id = cudaLaunchAttributeClusterDimension;
    cl.val.clusterDim.x = VJP_CLUSTER;
    cl.val.clusterDim.y = cl.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((grid + VJP_CLUSTER - 1) / VJP_CLUSTER * VJP_CLUSTER));
    cfg.blockDim = dim3(blk);
    cfg.stream = s;
    cfg.attrs = &cl;
    cfg.numAttrs = 1;
    NSI_CUDA(cudaLaunchKernelEx(&cfg, vjp_kernel<P>, view_of(h), f, w, gu, gmu, (const uint32_t*)h->bad_mask));
  } else {
    vjp_kernel<P><<<grid, blk, 0, s>>>(view_of(h), f, w, gu, gmu, h->bad_mask);
  }
  nsi_status st = check_launch("vjp_kernel");
  if (st || h->n_bad == 0) return st;
  vjp_exact_kernel<P><<<(h->n_bad + 63) / 64, 64, 0, s>>>(view_of(h), f, w, gu, gmu, h->bad_list, h->n_bad);
  return check_launch("vjp_exact_kernel");
}


template <int P>
static nsi_status residual_p(NsiHandle* h, const FieldView& f, void* r, cudaStream_t s) {
  using T = typename Prec<P>::T;
  NSI_CUDA(cudaMemsetAsync(r, 0, sizeof(T) * 3 * h->n, s));
  if (h->E == 0) return NSI_OK;
  const int blk = 256;
  residual_kernel<P><<<(h->E + blk - 1) / blk, blk, 0, s>>>(view_of(h), f, r, h->bad_mask);
  nsi_status st = check_launch("residual_kernel");
  if (st || h->n_bad == 0) return st;
  residual_exact_kernel<P><<<(h->n_bad + 63) / 64, 64, 0, s>>>(view_of(h), f, r, h->bad_list, h->n_bad);
  return check_launch("residual_exact_kernel");
}

// ------------------------------------------------ allocation-free variant ---
// Scratch of nsi_assemble_noalloc: room for the per-call node records of one
// mesh (32 bytes per node in the mixed modes, 64 in FP64).  It lives in the
// library's own device image, so every GPU that loads the library holds these
// 16 MiB until the process exits, and no call ever allocates it.
constexpr size_t NOALLOC_SCRATCH_BYTES = size_t(16) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

// Device address of the scratch for the current device.  In host code the
// array's name is only a host-side stand-in, so the address is looked up once
// per device, with that device current, and cached.
static nsi_status noalloc_scratch(int dev, void** out) {
  constexpr int MAX_DEV = 64;
  static std::mutex mu;
  static void* addr[MAX_DEV] = {};
  if (dev < 0 || dev >= MAX_DEV) return fail(NSI_ERR_UNSUPPORTED, "device ordinal beyond 63");
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    NSI_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    addr[dev] = p;
  }
  *out = addr[dev];
  return NSI_OK;
}

// the row gather of nsi_assemble (the same kernels and launch choice: star or
// edge-fan kernel, persistent grid, debug checks) with the node records in
// the static scratch, then the double-precision rows of badly shaped elements
template <int P>
static nsi_status assemble_noalloc_p(NsiHandle* h, const FieldView& f, const OutView& o, void* scratch,
                                     cudaStream_t s) {
  nsi_status st = assemble_core_p<P>(h, f, o, NSI_SCATTER_GATHER, s, scratch);
  if (st) return st;
  const RowOut ro{nullptr, o.A, o.G, o.rhs, nullptr, nullptr, 0.0};
  return fix_rows<P>(h, f, 0, ro, true, s);
}

}  // namespace nsi

using namespace nsi;

// Host-buffer call in the row-gather mode: the blocks of rows are assembled
// in chunks, and each finished chunk's slices of A, G and rhs go to the host
// on the handle's copy stream while the next chunk is assembled (the copies
// are the larger part of such a call).
template <int P>
static nsi_status host_chunked_p(NsiHandle* h, const NsiFields* fd, const NsiOutputs* od, const NsiOutputs* o,
                                 cudaStream_t s) {
  using Out = typename Prec<P>::Out;
  constexpr int C = (int)(sizeof(h->chunk_ev) / sizeof(h->chunk_ev[0]));
  if (!h->copy_stream) NSI_CUDA(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
  for (cudaEvent_t& e : h->chunk_ev)
    if (!e) NSI_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  const FieldView fv = fields_of(fd);
  const OutView ov{od->A_val, od->G_val, od->rhs};
  const int R = 32;
  nsi_status st = h->packs() ? launch_pack<P>(h, fv, nullptr, s) : NSI_OK;
  if (st) return st;
  const int64_t nb = (h->n + R - 1) / R;
  const int chunks = (int)std::min<int64_t>(C, nb);
  const Out* dA = static_cast<const Out*>(od->A_val);
  const Out* dG = static_cast<const Out*>(od->G_val);
  const Out* dR = static_cast<const Out*>(od->rhs);
  Out* hA = static_cast<Out*>(o->A_val);
  Out* hG = static_cast<Out*>(o->G_val);
  Out* hR = static_cast<Out*>(o->rhs);
  // the link, not the kernel, bounds the call: a small first chunk starts the
  // copies early, later chunks grow (the kernel runs ahead of the copies)
  static_assert(C == 8, "chunk fractions are listed for 8 chunks");
  const double frac[C + 1] = {0.0, 1.0 / 64, 1.0 / 16, 3.0 / 16, 5.0 / 16, 0.5, 11.0 / 16, 27.0 / 32, 1.0};
  auto bound = [&](int c) {
    return chunks == C ? (int64_t)((double)nb * frac[c]) : nb * c / chunks;
  };
  for (int c = 0; c < chunks; ++c) {
    const int64_t b0 = bound(c), b1 = c + 1 == chunks ? nb : bound(c + 1);
    if (b1 <= b0) continue;
    const int64_t r0 = b0 * R, r1 = std::min<int64_t>(h->n, b1 * R);
    st = launch_gather<P>(h, fv, ov, r0, r1, nullptr, s);
    if (st) return st;
    NSI_CUDA(cudaEventRecord(h->chunk_ev[c], s));
    NSI_CUDA(cudaStreamWaitEvent(h->copy_stream, h->chunk_ev[c], 0));
    const int64_t e0 = h->row_ptr_host[r0], e1 = h->row_ptr_host[r1];
    const size_t eb = sizeof(Out) * (size_t)(e1 - e0), rb = sizeof(Out) * (size_t)(r1 - r0);
    // A's slice, then the three components of G and of rhs (equal slices at a
    // fixed pitch) as one 2D copy each
    NSI_CUDA(cudaMemcpyAsync(hA + e0, dA + e0, eb, cudaMemcpyDeviceToHost, h->copy_stream));
    const size_t gp = sizeof(Out) * (size_t)h->nnz, rp = sizeof(Out) * (size_t)h->n;
    NSI_CUDA(cudaMemcpy2DAsync(hG + e0, gp, dG + e0, gp, eb, 3, cudaMemcpyDeviceToHost, h->copy_stream));
    NSI_CUDA(cudaMemcpy2DAsync(hR + r0, rp, dR + r0, rp, rb, 3, cudaMemcpyDeviceToHost, h->copy_stream));
  }
  NSI_CUDA(cudaStreamSynchronize(h->copy_stream));
  NSI_CUDA(cudaStreamSynchronize(s));
  return NSI_OK;
}

template <int P, bool DEBUG>
static nsi_status set_star_smem() {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  std::call_once(once, [] {
    err = cudaFuncSetAttribute(stab_star_kernel<P, DEBUG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(StarSmem<P>::bytes() * STAR_WARPS));
  });
  if (err != cudaSuccess) return cuda_fail(err, "cudaFuncSetAttribute(stabilised row kernel smem)");
  return NSI_OK;
}

// the stabilised velocity block: pack, the row kernel over every task, then
// the long rows and (mixed modes) the rows touching badly shaped elements by
// the per-row double kernel
template <int P>
static nsi_status stabilized_p(NsiHandle* h, const FieldView& f, const StabConst& sc, void* Auu, void* G, void* rhs,
                               cudaStream_t s) {
  if (h->n == 0) return NSI_OK;
  if (!h->gather_ok || !h->star_task)
    return fail(NSI_ERR_UNSUPPORTED, "the stabilised block needs the row maps (more than 2^31 node-element incidences)");
  nsi_status st = h->debug ? set_star_smem<P, true>() : set_star_smem<P, false>();
  if (st) return st;
  MeshView m = view_of(h);
  if ((st = launch_pack<P>(h, f, nullptr, s))) return st;
  const size_t smem = StarSmem<P>::bytes() * STAR_WARPS;
  const int64_t grid = (h->n_star_tasks + STAR_WARPS - 1) / STAR_WARPS;
  if (h->ev_start) NSI_CUDA(cudaEventRecord(h->ev_start, s));
  const auto kernel = h->debug ? stab_star_kernel<P, true> : stab_star_kernel<P, false>;
  NSI_CUDA(launch_early(kernel, grid, 32 * STAR_WARPS, smem, s, m, f, sc, (const int4*)h->star_task, h->n_star_tasks,
                        (const uint16_t*)h->star_word, Auu, G, rhs));
  if (h->ev_stop) NSI_CUDA(cudaEventRecord(h->ev_stop, s));
  st = check_launch("stab_star_kernel");
  if (st) return st;
  if (h->long_rows > 0) {
    stab_rows_kernel<P><<<(h->long_rows + 63) / 64, 64, 0, s>>>(m, f, sc, Auu, G, rhs, h->long_list, h->long_ptr,
                                                                 h->long_inc, h->long_rows);
    if ((st = check_launch("stab_rows_kernel (long rows)"))) return st;
  }
  const int64_t exact = h->exact_rows + h->exact_rest;
  if (P == NSI_FP64 || exact == 0) return NSI_OK;
  stab_rows_kernel<P><<<(exact + 63) / 64, 64, 0, s>>>(m, f, sc, Auu, G, rhs, h->exact_list, h->exact_ptr,
                                                       h->exact_inc, exact);
  return check_launch("stab_rows_kernel (exact rows)");
}

extern "C" {

nsi_status nsi_assemble(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, void* stream) {
  return assemble_dispatch(h, f, o, NSI_SCATTER_AUTO, static_cast<cudaStream_t>(stream));
}

nsi_status nsi_assemble_mode(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, int32_t scatter, void* stream) {
  return assemble_dispatch(h, f, o, scatter, static_cast<cudaStream_t>(stream));
}

nsi_status nsi_assemble_batched(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int32_t count,
                                void* stream) {
  if (count < 0 || count > NSI_MAX_BATCH) return fail(NSI_ERR_INVALID_ARG, "count must be in [0, NSI_MAX_BATCH]");
  if (count == 0) return NSI_OK;
  if (!hs || !fs || !os) return fail(NSI_ERR_INVALID_ARG, "batch array is NULL");
  const int prec = hs[0] ? hs[0]->precision : -1;
  for (int k = 0; k < count; ++k) {
    nsi_status st = check_call(hs[k], &fs[k], &os[k]);
    if (st) return st;
    if (hs[k]->precision != prec) return fail(NSI_ERR_INVALID_ARG, "batched handles must share one precision");
    if (!hs[k]->gather_ok) return fail(NSI_ERR_UNSUPPORTED, "batched assembly needs the row-gather mode");
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (prec) {
    case NSI_FP64: return batched_p<NSI_FP64>(hs, fs, os, count, s);
    case NSI_MIXED_F32_ACC64: return batched_p<NSI_MIXED_F32_ACC64>(hs, fs, os, count, s);
    default: return batched_p<NSI_MIXED_F32_ACC32>(hs, fs, os, count, s);
  }
}

nsi_status nsi_assemble_convective(NsiHandle* h, const NsiFields* f, const void* A_static, void* A_val, void* rhs,
                                   void* stream) {
  if (!h || !f || !rhs || (h->nnz > 0 && (!A_static || !A_val))) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  const StepView o{A_static, A_val, rhs, nullptr, nullptr, 0.0, 0.0f};
  return step_dispatch(h, f, o, false, static_cast<cudaStream_t>(stream));
}

nsi_status nsi_assemble_stabilized(NsiHandle* h, const NsiFields* f, void* Auu, void* G_val, void* rhs,
                                   void* stream) {
  if (!h || !f || !rhs || (h->nnz > 0 && (!Auu || !G_val))) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  if (!(f->mu > 0.0) || !std::isfinite(f->mu))
    return fail(NSI_ERR_INVALID_ARG, "mu must be finite and > 0 (tau1 of an element at rest is h^2 / (4 mu))");
  if (!(f->rho >= 0.0) || !std::isfinite(f->rho)) return fail(NSI_ERR_INVALID_ARG, "rho must be finite and >= 0");
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev != h->device) return fail(NSI_ERR_INVALID_ARG, "current device differs from the handle's device");
  const FieldView fv = fields_of(f);
  const StabConst sc = stab_const(f);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (h->precision) {
    case NSI_FP64: return stabilized_p<NSI_FP64>(h, fv, sc, Auu, G_val, rhs, s);
    case NSI_MIXED_F32_ACC64: return stabilized_p<NSI_MIXED_F32_ACC64>(h, fv, sc, Auu, G_val, rhs, s);
    default: return stabilized_p<NSI_MIXED_F32_ACC32>(h, fv, sc, Auu, G_val, rhs, s);
  }
}

nsi_status nsi_assemble_nodal(NsiHandle* h, const NsiFields* f, void* rhs, void* dt_rho, void* mass_rho, void* stream) {
  if (!h || !f || !rhs || !dt_rho || !mass_rho) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  const double kmr = f->rho / 24.0;
  const StepView o{nullptr, nullptr, rhs, dt_rho, mass_rho, kmr, (float)kmr};
  return step_dispatch(h, f, o, true, static_cast<cudaStream_t>(stream));
}

nsi_status nsi_assemble_vjp(NsiHandle* h, const NsiFields* f, const void* w, void* grad_u, double* grad_mu,
                            void* stream) {
  if (!h || !f || !w || !grad_u || !grad_mu) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  const FieldView fv = fields_of(f);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (h->precision) {
    case NSI_FP64: return vjp_p<NSI_FP64>(h, fv, w, grad_u, grad_mu, s);
    default: return vjp_p<NSI_MIXED_F32_ACC32>(h, fv, w, grad_u, grad_mu, s);
  }
}

nsi_status nsi_residual(NsiHandle* h, const NsiFields* f, void* r, void* stream) {
  if (!h || !f || !r) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (!f->u[k]) return fail(NSI_ERR_INVALID_ARG, "velocity component pointer is NULL");
  if (!(f->dt > 0.0)) return fail(NSI_ERR_INVALID_ARG, "dt must be > 0");
  const FieldView fv = fields_of(f);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (h->precision == NSI_FP64) return residual_p<NSI_FP64>(h, fv, r, s);
  return residual_p<NSI_MIXED_F32_ACC32>(h, fv, r, s);
}

static nsi_status values_args(void* const* comp, int32_t ncomp, const int32_t* idx, int64_t count, const void* buf,
                              int32_t value_bytes, CompPtrs& cp) {
  if (count < 0) return fail(NSI_ERR_INVALID_ARG, "count < 0");
  if (ncomp < 1 || ncomp > XCH_MAX_COMP) return fail(NSI_ERR_INVALID_ARG, "ncomp must be in [1, 4]");
  if (value_bytes != 4 && value_bytes != 8) return fail(NSI_ERR_INVALID_ARG, "value_bytes must be 4 or 8");
  if (count > 0 && (!comp || !idx || !buf)) return fail(NSI_ERR_INVALID_ARG, "NULL argument");
  for (int c = 0; c < XCH_MAX_COMP; ++c) cp.p[c] = nullptr;
  for (int c = 0; c < ncomp && count > 0; ++c) {
    if (!comp[c]) return fail(NSI_ERR_INVALID_ARG, "NULL component pointer");
    cp.p[c] = comp[c];
  }
  return NSI_OK;
}

nsi_status nsi_gather_values(const void* const* src, int32_t ncomp, const int32_t* idx, int64_t count, void* dst,
                             int32_t value_bytes, void* stream) {
  CompPtrs cp;
  nsi_status st = values_args(const_cast<void* const*>(src), ncomp, idx, count, dst, value_bytes, cp);
  if (st || count == 0) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t grid = (count + 255) / 256;
  if (value_bytes == 8) gather_values_kernel<double><<<grid, 256, 0, s>>>(cp, ncomp, idx, count, static_cast<double*>(dst));
  else gather_values_kernel<float><<<grid, 256, 0, s>>>(cp, ncomp, idx, count, static_cast<float*>(dst));
  return check_launch("gather_values_kernel");
}

nsi_status nsi_add_values(void* const* dst, int32_t ncomp, const int32_t* idx, int64_t count, const void* src,
                          int32_t value_bytes, void* stream) {
  CompPtrs cp;
  nsi_status st = values_args(dst, ncomp, idx, count, src, value_bytes, cp);
  if (st || count == 0) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t grid = (count + 255) / 256;
  if (value_bytes == 8) add_values_kernel<double><<<grid, 256, 0, s>>>(cp, ncomp, idx, count, static_cast<const double*>(src));
  else add_values_kernel<float><<<grid, 256, 0, s>>>(cp, ncomp, idx, count, static_cast<const float*>(src));
  return check_launch("add_values_kernel");
}

nsi_status nsi_assemble_noalloc(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, void* stream) {
  nsi_status st = check_call(h, f, o);
  if (st) return st;
  if (!h->gather_ok) return fail(NSI_ERR_UNSUPPORTED, "the allocation-free call needs the row-gather mode");
  const size_t rec = h->precision == NSI_FP64 ? 64 : 32;
  if ((size_t)h->n * rec > NOALLOC_SCRATCH_BYTES) {
    char buf[200];
    snprintf(buf, sizeof buf,
             "mesh too large for the allocation-free call: %lld nodes need %zu bytes of scratch, the static "
             "scratch holds %zu (%zu nodes at %zu bytes each)",
             (long long)h->n, (size_t)h->n * rec, NOALLOC_SCRATCH_BYTES, NOALLOC_SCRATCH_BYTES / rec, rec);
    return fail(NSI_ERR_UNSUPPORTED, buf);
  }
  int dev = 0;
  NSI_CUDA(cudaGetDevice(&dev));
  if (dev != h->device) return fail(NSI_ERR_INVALID_ARG, "current device differs from the handle's device");
  void* scratch = nullptr;
  st = noalloc_scratch(dev, &scratch);
  if (st) return st;
  const FieldView fv = fields_of(f);
  const OutView ov{o->A_val, o->G_val, o->rhs};
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (h->precision) {
    case NSI_FP64: return assemble_noalloc_p<NSI_FP64>(h, fv, ov, scratch, s);
    case NSI_MIXED_F32_ACC64: return assemble_noalloc_p<NSI_MIXED_F32_ACC64>(h, fv, ov, scratch, s);
    default: return assemble_noalloc_p<NSI_MIXED_F32_ACC32>(h, fv, ov, scratch, s);
  }
}

nsi_status nsi_autotune(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, int32_t reps, void* stream,
                        int32_t* chosen_scatter, int32_t* chosen_rows) {
  nsi_status st = check_call(h, f, o);
  if (st) return st;
  if (reps < 1 || reps > 1000) return fail(NSI_ERR_INVALID_ARG, "reps must be in [1, 1000]");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaEvent_t e0, e1;
  NSI_CUDA(cudaEventCreate(&e0));
  NSI_CUDA(cudaEventCreate(&e1));
  struct Cand {
    int scatter, plan;  // plan: index into h->plans (star kernel), -2: edge-fan kernel,
                        // -3: warp-aggregated atomics, -1: n/a
  };
  std::vector<Cand> cands;
  if (h->fan_ok) cands.push_back({NSI_SCATTER_GATHER, -2});
  if (h->gather_ok)
    for (int k = 0; k < h->n_plans; ++k) cands.push_back({NSI_SCATTER_GATHER, k});
  cands.push_back({NSI_SCATTER_COLOR, -1});
  cands.push_back({NSI_SCATTER_ATOMIC, -1});
  cands.push_back({NSI_SCATTER_ATOMIC, -3});
  const GatherPlan saved = h->plan;
  const bool saved_fan = h->use_fan, saved_agg = h->atomic_agg;
  float best = 1e30f;
  Cand pick{h->scatter, saved_fan ? -2 : -1};
  cudaEvent_t ev0 = h->ev_start, ev1 = h->ev_stop;
  h->ev_start = h->ev_stop = nullptr;
  for (const Cand& c : cands) {
    h->use_fan = c.plan == -2;
    h->atomic_agg = c.plan == -3;
    if (c.plan >= 0) h->plan = h->plans[c.plan];
    st = assemble_dispatch(h, f, o, c.scatter, s);  // warm-up
    if (st) break;
    cudaEventRecord(e0, s);
    for (int r = 0; r < reps && !st; ++r) st = assemble_dispatch(h, f, o, c.scatter, s);
    cudaEventRecord(e1, s);
    if (st) break;
    cudaError_t ce = cudaEventSynchronize(e1);
    if (ce != cudaSuccess) {
      st = cuda_fail(ce, "cudaEventSynchronize in autotune");
      break;
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best) {
      best = ms;
      pick = c;
    }
  }
  h->ev_start = ev0;
  h->ev_stop = ev1;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  h->plan = pick.plan >= 0 ? h->plans[pick.plan] : saved;
  h->use_fan = pick.scatter == NSI_SCATTER_GATHER ? pick.plan == -2 : saved_fan;
  h->atomic_agg = pick.scatter == NSI_SCATTER_ATOMIC ? pick.plan == -3 : saved_agg;
  if (st) return st;
  h->scatter = pick.scatter;
  if (chosen_scatter) *chosen_scatter = pick.scatter;
  if (chosen_rows)
    *chosen_rows = pick.scatter == NSI_SCATTER_GATHER ? (h->use_fan ? -1 : h->plan.rows_per_block)
                   : pick.scatter == NSI_SCATTER_ATOMIC ? (h->atomic_agg ? 1 : 2)
                                                        : 0;
  return NSI_OK;
}

nsi_status nsi_assemble_host(NsiHandle* h, const NsiFields* f, const NsiOutputs* o, void* stream) {
  nsi_status st = check_call(h, f, o);
  if (st) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t tsz = h->precision == NSI_FP64 ? 8 : 4;
  const size_t osz = h->precision == NSI_MIXED_F32_ACC32 ? 4 : 8;
  const bool sep_un = f->u_n[0] || f->u_n[1] || f->u_n[2];
  const size_t u_bytes = tsz * h->n * (sep_un ? 6 : 3);
  const size_t o_bytes = osz * (4 * h->nnz + 3 * h->n);
  const size_t need = ((u_bytes + 255) / 256) * 256 + o_bytes;
  if (h->stage_bytes < need) {
    cudaFree(h->stage);
    h->stage = nullptr;
    h->stage_bytes = 0;
    NSI_CUDA(cudaMalloc(&h->stage, need));
    h->stage_bytes = need;
  }
  char* base = static_cast<char*>(h->stage);
  NsiFields fd = *f;
  for (int k = 0; k < 3; ++k) {
    void* dst = base + k * tsz * h->n;
    NSI_CUDA(cudaMemcpyAsync(dst, f->u[k], tsz * h->n, cudaMemcpyHostToDevice, s));
    fd.u[k] = dst;
    fd.u_n[k] = nullptr;
  }
  if (sep_un) {
    for (int k = 0; k < 3; ++k) {
      void* dst = base + (3 + k) * tsz * h->n;
      const void* src = f->u_n[k] ? f->u_n[k] : f->u[k];
      NSI_CUDA(cudaMemcpyAsync(dst, src, tsz * h->n, cudaMemcpyHostToDevice, s));
      fd.u_n[k] = dst;
    }
  }
  char* ob = base + ((u_bytes + 255) / 256) * 256;
  NsiOutputs od{ob, ob + osz * h->nnz, ob + osz * 4 * h->nnz};
  if (resolve_mode(h, NSI_SCATTER_AUTO) == NSI_SCATTER_GATHER && !h->use_fan && h->n > 0 && h->exact_rows + h->exact_rest == 0 &&
      h->long_rows == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != h->device) return fail(NSI_ERR_INVALID_ARG, "current device differs from the handle's device");
    switch (h->precision) {
      case NSI_FP64: return host_chunked_p<NSI_FP64>(h, &fd, &od, o, s);
      case NSI_MIXED_F32_ACC64: return host_chunked_p<NSI_MIXED_F32_ACC64>(h, &fd, &od, o, s);
      default: return host_chunked_p<NSI_MIXED_F32_ACC32>(h, &fd, &od, o, s);
    }
  }
  st = assemble_dispatch(h, &fd, &od, NSI_SCATTER_AUTO, s);
  if (st) return st;
  NSI_CUDA(cudaMemcpyAsync(o->A_val, od.A_val, osz * h->nnz, cudaMemcpyDeviceToHost, s));
  NSI_CUDA(cudaMemcpyAsync(o->G_val, od.G_val, osz * 3 * h->nnz, cudaMemcpyDeviceToHost, s));
  NSI_CUDA(cudaMemcpyAsync(o->rhs, od.rhs, osz * 3 * h->n, cudaMemcpyDeviceToHost, s));
  NSI_CUDA(cudaStreamSynchronize(s));
  return NSI_OK;
}

}  // extern "C"
