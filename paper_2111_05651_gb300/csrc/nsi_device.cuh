// Device code shared by the kernel files: the views of a mesh, its fields and
// outputs that the kernels take, precision traits, per-call node records,
// accumulators and the float -> double conversions of the write-outs.
#pragma once

#include "nsi_internal.cuh"

namespace nsi {

// ------------------------------------------------------------ views ------
struct MeshView {
  int64_t n, E, nnz;
  const int32_t* __restrict__ row_ptr;
  const int32_t* __restrict__ col_idx;
  const int4* __restrict__ lnods;
  const uint8_t* __restrict__ diag_pos;
  const D4* __restrict__ xyz64;
  const float4* __restrict__ xyz_hi;
  const float4* __restrict__ xyz_lo;
  const void* rec;  // (written by the packing, which an early launch may overlap)
  const uint32_t* __restrict__ fan;
  const int32_t* __restrict__ fan_blk;
  unsigned* err;
};

// Physical constants of the element formulas, precomputed on the host in
// double (the float copies are rounded once): rho/120 (convection), mu/6
// (viscous) and rho/(24 dt) (lumped mass).
struct FieldView {
  const void* u[3];
  const void* un[3];
  double kc, kmu, kmass;
  float kcf, kmuf, kmassf;
};

template <typename T>
__device__ __forceinline__ T kc_of(const FieldView& f) {
  if constexpr (sizeof(T) == 8) return f.kc;
  else return f.kcf;
}
template <typename T>
__device__ __forceinline__ T kmu_of(const FieldView& f) {
  if constexpr (sizeof(T) == 8) return f.kmu;
  else return f.kmuf;
}
template <typename T>
__device__ __forceinline__ T kmass_of(const FieldView& f) {
  if constexpr (sizeof(T) == 8) return f.kmass;
  else return f.kmassf;
}

struct OutView {
  void* A;
  void* G;
  void* rhs;
};

// outputs of the time step and the nodal kernels; kmr = rho/24 (the density
// mass per det)
struct StepView {
  const void* A_static;
  void* A;
  void* rhs;
  void* dt_rho;
  void* mass_rho;
  double kmr;
  float kmrf;
};

inline MeshView view_of(const NsiHandle* h) {
  MeshView m;
  m.n = h->n;
  m.E = h->E;
  m.nnz = h->nnz;
  m.row_ptr = h->row_ptr;
  m.col_idx = h->col_idx;
  m.lnods = h->lnods;
  m.diag_pos = h->diag_pos;
  m.xyz64 = h->xyz64;
  m.xyz_hi = h->xyz_hi;
  m.xyz_lo = h->xyz_lo;
  m.rec = h->rec;
  m.fan = h->fan;
  m.fan_blk = h->fan_blk;
  m.err = h->err;
  return m;
}

inline FieldView fields_of(const NsiFields* f) {
  FieldView v;
  for (int k = 0; k < 3; ++k) {
    v.u[k] = f->u[k];
    v.un[k] = f->u_n[k] ? f->u_n[k] : f->u[k];
  }
  v.kc = f->rho / 120.0;
  v.kmu = f->mu / 6.0;
  v.kmass = f->rho / (24.0 * f->dt);
  v.kcf = (float)v.kc;
  v.kmuf = (float)v.kmu;
  v.kmassf = (float)v.kmass;
  return v;
}

// outputs of the kernels that compute listed rows in double: A, G (assembly),
// A with A_static (time step), rhs, dt_rho and mass_rho (nodal outputs)
struct RowOut {
  const void* A_static;
  void *A, *G, *rhs, *dt_rho, *mass_rho;
  double kmr;
};

// precision traits: compute type T, output type Out
template <int P>
struct Prec;
template <>
struct Prec<NSI_FP64> {
  using T = double;
  using Out = double;
};
template <>
struct Prec<NSI_MIXED_F32_ACC64> {
  using T = float;
  using Out = double;
};
template <>
struct Prec<NSI_MIXED_F32_ACC32> {
  using T = float;
  using Out = float;
};

template <typename T>
__device__ __forceinline__ T rcp(T x);
template <>
__device__ __forceinline__ float rcp<float>(float x) {
  return __frcp_rn(x);
}
template <>
__device__ __forceinline__ double rcp<double>(double x) {
  return 1.0 / x;
}

// node coordinates: exact double, or a float hi/lo pair whose difference
// gives edge vectors to ~2^-48 relative before the float arithmetic starts
template <int P>
struct NodeX;
template <>
struct NodeX<NSI_FP64> {
  V3<double> x;
  __device__ __forceinline__ void load(const MeshView& m, int64_t v) {
    D4 p = m.xyz64[v];
    x = {p.x, p.y, p.z};
  }
  __device__ __forceinline__ V3<double> minus(const NodeX& o) const { return sub(x, o.x); }
};
template <int P>
struct NodeX {
  V3<float> hi, lo;
  __device__ __forceinline__ void load(const MeshView& m, int64_t v) {
    float4 a = __ldg(m.xyz_hi + v);
    float4 b = __ldg(m.xyz_lo + v);
    hi = {a.x, a.y, a.z};
    lo = {b.x, b.y, b.z};
  }
  __device__ __forceinline__ V3<float> minus(const NodeX& o) const { return add(sub(hi, o.hi), sub(lo, o.lo)); }
};

template <typename T>
__device__ __forceinline__ V3<T> load_vec(const void* const* comp, int64_t v) {
  return {__ldg(static_cast<const T*>(comp[0]) + v), __ldg(static_cast<const T*>(comp[1]) + v),
          __ldg(static_cast<const T*>(comp[2]) + v)};
}

// ---------------------------------------------------------- node records ---
// One record per node, rebuilt every call from the handle's coordinates and
// the caller's velocities, so that the row-gather kernel fetches a neighbour
// with one 32-byte (mixed) or 64-byte (FP64) request instead of five:
//   mixed: {hx, hy, hz, ux} {uy, uz, lo_xy, lo_z}, lo_* the top 16 bits of
//          the float low parts (coordinates kept to ~2^-32 relative)
//   FP64:  {x, y, z, 0} {ux, uy, uz, 0} as doubles
template <int P, typename Mesh>
__device__ __forceinline__ void pack_node(const Mesh& m, const FieldView& f, void* __restrict__ rec, int64_t i) {
  if constexpr (P == NSI_FP64) {
    const D4 x = m.xyz64[i];
    const V3<double> u = load_vec<double>(f.u, i);
    D4* r = static_cast<D4*>(rec) + 2 * i;
    r[0] = D4{x.x, x.y, x.z, 0.0};
    r[1] = D4{u.x, u.y, u.z, 0.0};
  } else {
    const float4 hi = __ldg(m.xyz_hi + i);
    const float4 lo = __ldg(m.xyz_lo + i);
    const V3<float> u = load_vec<float>(f.u, i);
    uint4* r = static_cast<uint4*>(rec) + 2 * i;
    r[0] = make_uint4(__float_as_uint(hi.x), __float_as_uint(hi.y), __float_as_uint(hi.z), __float_as_uint(u.x));
    r[1] = make_uint4(__float_as_uint(u.y), __float_as_uint(u.z),
                      (__float_as_uint(lo.x) >> 16) | (__float_as_uint(lo.y) & 0xffff0000u),
                      __float_as_uint(lo.z) & 0xffff0000u);
  }
}

__device__ __forceinline__ V3<float> record_lo(float w6, float w7) {
  const unsigned a = __float_as_uint(w6), b = __float_as_uint(w7);
  return {__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u), __uint_as_float(b & 0xffff0000u)};
}

// ------------------------------------------ accumulators, conversions ---
// Register accumulator of one output value: plain T, or a compensated float
// pair (TwoSum) for the mixed mode with double output.
template <int P>
struct Acc {
  using T = typename Prec<P>::T;
  T v;
  __device__ __forceinline__ void zero() { v = T(0); }
  __device__ __forceinline__ void add(T x) { v += x; }
};
template <>
struct Acc<NSI_MIXED_F32_ACC64> {
  float hi, lo;
  __device__ __forceinline__ void zero() { hi = lo = 0.0f; }
  __device__ __forceinline__ void add(float x) {
    float s, e;
    two_sum(hi, x, s, e);
    hi = s;
    lo += e;
  }
};

__device__ __forceinline__ void store_acc(double* p, const Acc<NSI_FP64>& a) { *p = a.v; }
__device__ __forceinline__ void store_acc(float* p, const Acc<NSI_MIXED_F32_ACC32>& a) { *p = a.v; }
// The double nearest hi + lo for a renormalised float pair (|lo| <= ulp(hi) /
// 2) with a finite hi, without branches: the double of |hi| from its bits, lo
// (with hi's sign taken out) added as an integer k of the double's units in
// the last place (|k| <= 2^28), hi's sign set last.  When |hi| is a power of
// two and the sum lies below it, k counts the half-size units of the binade
// below.  Zero gives zero; a tiny |hi| (below 2^-75, where the scale of k would
// leave the float range) is handled at 2^100 times its size, the exponent
// taken back in the result.  Infinite and NaN values are the callers' (a test
// for them here costs the write-out loop several percent).
__device__ __forceinline__ double normalised_pair_double(float hi, float lo) {
  const unsigned u0 = __float_as_uint(hi);
  const bool tiny = ((u0 >> 23) & 0xffu) < 52u;
  const float sc = tiny ? 0x1p100f : 1.0f;
  const float h2 = hi * sc, l2 = lo * sc;  // exact
  const unsigned uh = __float_as_uint(h2);
  const unsigned eh = (uh >> 23) & 0xffu;
  const float ls = __uint_as_float(__float_as_uint(l2) ^ (uh & 0x80000000u));
  const unsigned below = ((uh << 9) == 0u && ls < 0.0f) ? 1u : 0u;
  const int k = __float2int_rn(ls * __uint_as_float((306u + below - eh) << 23));
  const unsigned long long mag =
      ((unsigned long long)(uh & 0x7fffffffu) << 29) + ((tiny ? 796ull : 896ull) << 52);
  const unsigned long long r = (mag + (unsigned long long)(long long)k) | ((unsigned long long)(uh & 0x80000000u) << 32);
  return __longlong_as_double((u0 << 1) == 0u ? (long long)((unsigned long long)(u0 & 0x80000000u) << 32)
                                              : (long long)r);
}
// an infinite or NaN accumulator (hi) as a double of the same class
__device__ __forceinline__ double nonfinite_double(float hi) { return __longlong_as_double(f32_to_f64_bits(hi)); }
// true if the exponent bits of x are all ones (infinite or NaN)
__device__ __forceinline__ bool nonfinite_bits(float x) { return (__float_as_uint(x) | 0x807fffffu) == 0xffffffffu; }
// the double equal to a normal or zero float, from its bit pattern: the
// exponent rebiased (+896), the 23 mantissa bits moved to the top of the
// double's 52; the sign kept (an arithmetic shift leaves it in the top bit).  A
// subnormal float (below 2^-126 in magnitude) gives a subnormal double (below
// 2^-1022, no more than a signed zero); infinite and NaN floats are not handled
// (the values converted this way are the pressure-gradient sums, functions of
// the coordinates a handle validates, far inside the float range for any mesh
// whose float element arithmetic is meaningful).
__device__ __forceinline__ double float_double(float x) {
  const int u = __float_as_int(x);
  const int bias = fabsf(x) < 0x1p-126f ? 0 : (896 << 20);
  return __hiloint2double(((u >> 3) & (int)0x8fffffffu) + bias, u << 29);
}
// the double nearest hi + lo of a pair with a finite hi: renormalised first
// (Fast2Sum)
__device__ __forceinline__ double pair_double(float hi, float lo) {
  const float s = hi + lo;
  const float l = lo - (s - hi);
  return normalised_pair_double(s, l);
}
__device__ __forceinline__ void store_acc(double* p, const Acc<NSI_MIXED_F32_ACC64>& a) {
  *p = nonfinite_bits(a.hi) ? nonfinite_double(a.hi) : pair_double(a.hi, a.lo);
}

template <typename T>
struct alignas(4 * sizeof(T)) T4 {
  T x, y, z, w;
};
template <typename T>
struct alignas(2 * sizeof(T)) T2 {
  T x, y;
};

// reciprocal of det: the float path uses the fast approximate division
// (about 1 ulp); the double path refines the hardware's approximate double
// reciprocal r (rcp.approx.ftz.f64, relative error at most 2^-20 over 4 M
// normal inputs measured on GB300) once by the cubic iteration for 1/x,
// r (1 + e + e^2) with e = 1 - x r, whose relative error is e^3 (2^-60, below
// the double's rounding): three FMAs on GB300's slow FP64 pipe instead of the
// four of two Newton-Raphson steps.  det is a normal number here (the mesh is
// validated at create).
__device__ __forceinline__ float rcp_fast(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double rcp_fast(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  r = fma(r, fma(e, e, e), r);
  return r;
}

// Programmatic dependent launch: a kernel launched by launch_early may start
// as the blocks of the launch directly before it end, and calls
// wait_for_previous before it reads what that launch writes, or writes what it
// may write too; the wait ends when that launch, and so every one before it, is
// complete.  What that launch writes is not read-only for such a kernel's
// life: it is never read by .nc loads (or __ldg), and inline loads of it are
// volatile with a memory clobber, so that they stay after the wait.  Used by the
// kernels that read the packing's node records, which first fetch row bounds,
// column indices and walk bytes, and by those that overwrite listed rows.
// (Letting them start with the packing's first blocks
// takes the SMs from it: a batch of 16 meshes 90.1 us, without early launches
// 84.2, as it is 84.1; a 47x61x38 box in mixed32 33.0, 36.3, 33.1; a time step
// of 81x70x66 96.8, 94.6, 92.5.)
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// 32 bytes of a node record (32-byte aligned) by one 256-bit load.  CACHE:
// through L1 (the stabilised kernel, whose warps share neighbours), else past it.
template <bool CACHE>
__device__ __forceinline__ void load_record(const unsigned* r, uint4& a, uint4& b) {
  if constexpr (CACHE)
    asm volatile("ld.global.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(r)
                 : "memory");
  else
    asm volatile("ld.global.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
                 : "l"(r)
                 : "memory");
}
template <bool CACHE>
__device__ __forceinline__ void load_record(const double* r, double& x, double& y, double& z) {
  [[maybe_unused]] double pad;
  if constexpr (CACHE)
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(x), "=d"(y), "=d"(z), "=d"(pad) : "l"(r) : "memory");
  else
    asm volatile("ld.global.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(x), "=d"(y), "=d"(z), "=d"(pad)
                 : "l"(r)
                 : "memory");
}
template <typename... Params, typename... Args>
cudaError_t launch_early(void (*kernel)(Params...), int64_t grid, int block, size_t smem, cudaStream_t s,
                         const Args&... args) {
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

inline nsi_status check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, what);
  return NSI_OK;
}

// ------------------------------------------------- launchers (nsi_gather.cu) ---
// The call's node records (rec: where to, nullptr: the handle's buffer), read
// by the launches below.
template <int P>
nsi_status launch_pack(NsiHandle* h, const FieldView& f, void* rec, cudaStream_t s);
// A, G and rhs of rows [row0, row1) (row0 a multiple of 32, row1 too unless it
// is n)
template <int P>
nsi_status launch_gather(NsiHandle* h, const FieldView& f, const OutView& o, int64_t row0, int64_t row1, void* rec,
                         cudaStream_t s);
template <int P>
nsi_status launch_step(NsiHandle* h, const FieldView& f, const StepView& o, bool nodal, cudaStream_t s);
// the handle's rows of badly shaped elements that have a walk, in double (mixed
// modes), by mode: 0 the assembly, 1 the time step, 2 the nodal outputs
template <int P>
nsi_status launch_exact_rows(NsiHandle* h, const FieldView& f, int mode, const RowOut& o, cudaStream_t s);
template <int P>
nsi_status launch_batched(NsiHandle* const* hs, const NsiFields* fs, const NsiOutputs* os, int count, cudaStream_t s);

}  // namespace nsi
