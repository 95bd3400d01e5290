// Row units and their moves between the fields, the half spectra and the transform core, shared by the
// film (2D) and bulk (3D) kernels.
//
// A row unit is RU consecutive rows (4 in FP32, 2 in FP64): two rows per complex line, a + i b, one (FP64)
// or two (FP32) lines per element of the core.  The real fields of the workspace and the mask are kept by
// row units: for each x the unit's RU values lie together, 16 bytes, and their mask classes in one byte.
// A half spectrum (nx/2 + 1 x-wavenumbers) is S[kx][y] per (field and z): the values of a unit's rows at
// one kx are 32 contiguous bytes.
#pragma once
#include "mf_core.cuh"
#include "mf_rhs_common.cuh"

namespace mf {

// ------------------------------------------------------------------------------------------
// row units
// ------------------------------------------------------------------------------------------
// the RU rows of one element at one x: 16 bytes
template <typename T> struct alignas(16) Q { T v[Lane<T>::RU]; };
__device__ __forceinline__ Q<float> ld_q(const float* p) {
  Q<float> r;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]) : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ Q<double> ld_q(const double* p) {
  Q<double> r;
  asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(r.v[0]), "=d"(r.v[1]) : "l"(p) : "memory");
  return r;
}
// read-only for the whole launch (non-coherent path)
__device__ __forceinline__ Q<float> ldg_q(const float* p) {
  Q<float> r;
  asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]) : "l"(p));
  return r;
}
__device__ __forceinline__ Q<double> ldg_q(const double* p) {
  Q<double> r;
  asm("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(r.v[0]), "=d"(r.v[1]) : "l"(p));
  return r;
}
__device__ __forceinline__ void st_q(float* p, const Q<float>& q) { *(float4*)p = make_float4(q.v[0], q.v[1], q.v[2], q.v[3]); }
__device__ __forceinline__ void st_q(double* p, const Q<double>& q) { *(double2*)p = make_double2(q.v[0], q.v[1]); }
// element <-> rows: lines pack rows (0, 2) and (1, 3) in FP32, (0, 1) in FP64, as a + i b
__device__ __forceinline__ Q<float> to_q(const CV<F2>& e) {
  Q<float> q;
  upk(e.x, q.v[0], q.v[1]);
  upk(e.y, q.v[2], q.v[3]);
  return q;
}
__device__ __forceinline__ Q<double> to_q(const CV<double>& e) { return Q<double>{{e.x, e.y}}; }
__device__ __forceinline__ CV<F2> to_e(const Q<float>& q) { return {pk(q.v[0], q.v[1]), pk(q.v[2], q.v[3])}; }
__device__ __forceinline__ CV<double> to_e(const Q<double>& q) { return {q.v[0], q.v[1]}; }
// mask classes of a unit's rows, 2 bits each
__device__ __forceinline__ int ld_mask(const uint8_t* p) {
  unsigned m;
  asm("ld.global.nc.L1::no_allocate.u8 %0, [%1];" : "=r"(m) : "l"(p));
  return (int)m;
}
__device__ __forceinline__ int cls(int m, int r) { return (m >> (2 * r)) & 3; }

// 32 bytes of one half-spectrum column: the complex values of a unit's rows at one x-wavenumber
struct B32f { float a[8]; };
struct B32d { double a[4]; };
__device__ __forceinline__ B32f ld_b32(const C2<float>* p) {
  B32f r;
  asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(r.a[0]), "=f"(r.a[1]), "=f"(r.a[2]), "=f"(r.a[3]), "=f"(r.a[4]), "=f"(r.a[5]),
                 "=f"(r.a[6]), "=f"(r.a[7]) : "l"(p) : "memory");
  return r;
}
__device__ __forceinline__ B32d ld_b32(const C2<double>* p) {
  B32d r;
  asm volatile("ld.global.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(r.a[0]), "=d"(r.a[1]), "=d"(r.a[2]), "=d"(r.a[3]) : "l"(p) : "memory");
  return r;
}
// position k of the packed lines (a + i b per pair of rows) from the rows' half spectra A, B at k:
// A + i B; at nx - k: conj(A) + i conj(B); at k = 0 and nx/2 the imaginary parts are dropped
__device__ __forceinline__ CV<F2> pack_lo(const B32f& s) { return {pk(s.a[0] - s.a[5], s.a[2] - s.a[7]), pk(s.a[1] + s.a[4], s.a[3] + s.a[6])}; }
__device__ __forceinline__ CV<F2> pack_hi(const B32f& s) { return {pk(s.a[0] + s.a[5], s.a[2] + s.a[7]), pk(s.a[4] - s.a[1], s.a[6] - s.a[3])}; }
__device__ __forceinline__ CV<F2> pack_re(const B32f& s) { return {pk(s.a[0], s.a[2]), pk(s.a[4], s.a[6])}; }
__device__ __forceinline__ CV<double> pack_lo(const B32d& s) { return {s.a[0] - s.a[3], s.a[1] + s.a[2]}; }
__device__ __forceinline__ CV<double> pack_hi(const B32d& s) { return {s.a[0] + s.a[3], s.a[2] - s.a[1]}; }
__device__ __forceinline__ CV<double> pack_re(const B32d& s) { return {s.a[0], s.a[2]}; }
// twice the rows' half spectra at k from the packed lines' transforms at k and nx - k (the factor
// 1/2 is in the column passes' scale)
__device__ __forceinline__ void st_b32(C2<float>* p, const CV<F2>& zk, const CV<F2>& zm) {
  float r[8];
  upk(vadd(zk.x, zm.x), r[0], r[2]);
  upk(vsub(zk.y, zm.y), r[1], r[3]);
  upk(vadd(zk.y, zm.y), r[4], r[6]);
  upk(vsub(zm.x, zk.x), r[5], r[7]);
  asm volatile("st.global.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
               :: "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "l"(p) : "memory");
}
__device__ __forceinline__ void st_b32(C2<double>* p, const CV<double>& zk, const CV<double>& zm) {
  asm volatile("st.global.v4.f64 [%4], {%0, %1, %2, %3};"
               :: "d"(zk.x + zm.x), "d"(zk.y - zm.y), "d"(zk.y + zm.y), "d"(zm.x - zk.x), "l"(p) : "memory");
}
// one column element: the values of line kx (and, in FP32, of line kx + 1 at `stride`)
__device__ __forceinline__ CV<F2> ld_col(const C2<float>* p, int stride, bool two) {
  const C2<float> a = lds_c2(p);
  C2<float> b = {0.f, 0.f};
  if (two) b = lds_c2(p + stride);
  return {pk(a.x, b.x), pk(a.y, b.y)};
}
__device__ __forceinline__ CV<double> ld_col(const C2<double>* p, int, bool) {
  const C2<double> a = lds_c2(p);
  return {a.x, a.y};
}
__device__ __forceinline__ void st_col(C2<float>* p, int stride, bool two, const CV<F2>& e) {
  C2<float> a, b;
  upk(e.x, a.x, b.x);
  upk(e.y, a.y, b.y);
  p[0] = a;
  if (two) p[stride] = b;
}
__device__ __forceinline__ void st_col(C2<double>* p, int, bool, const CV<double>& e) { p[0] = C2<double>{e.x, e.y}; }

// FP64 state fields are row-major (the caller's layout)
__device__ __forceinline__ double ld_s(const double* p) {
  double v;
  asm volatile("ld.global.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}

struct NoLd {};

// Asynchronous copies global -> shared, 16 bytes each: issued without a register round trip, complete at
// cp_wait (this thread's copies; a barrier of the threads that read them makes them visible).
__device__ __forceinline__ void cp16(void* s, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"((unsigned)__cvta_generic_to_shared(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// The packed lines of a unit's rows from their half spectra at src + kx ny: a thread loads the half
// spectrum at its k < nx/2 once, keeps Z[k] and hands Z[nx - k] over through the shared buffer.
// ld(j, k) gives the 32 bytes at the thread's j-th k (j = E/2: k = nx/2, asked for by thread 0).
template <typename T, int E, class Ld>
__device__ __forceinline__ void row_gather_from(CV<typename Lane<T>::V> (&v)[E], const Team<T, E>& t, int nx, Ld ld) {
  const int q = t.step();
  t.sync();
#pragma unroll
  for (int j = 0; j < E / 2; ++j) {
    const int k = t.i + j * q;
    const auto s = ld(j, k);
    if (k == 0) {
      v[j] = pack_re(s);
    } else {
      v[j] = pack_lo(s);
      t.at(nx - k) = pack_hi(s);
    }
  }
  if (t.i == 0) t.at(nx >> 1) = pack_re(ld(E / 2, nx >> 1));
  t.sync();
#pragma unroll
  for (int j = E / 2; j < E; ++j) v[j] = t.at(t.i + j * q);
}
template <typename T, int E>
__device__ __forceinline__ void row_gather(CV<typename Lane<T>::V> (&v)[E], const Team<T, E>& t, const C2<T>* src, int nx, int ny) {
  row_gather_from(v, t, nx, [&](int, int k) { return ld_b32(src + k * ny); });
}
// The same from a copy in shared memory that row_stage issued for the group's 2^lgG neighbouring units:
// their 2^lgG x 32 contiguous bytes at each k < nx/2, one k after the other (stg), and at nx/2 (top).
// src: the spectra of the group's first unit.
template <typename T, int E>
__device__ __forceinline__ void row_stage(const Team<T, E>& t, int lgG, uint4* stg, uint4* top, const C2<T>* src, int nx, int ny) {
  const int g = (t.i << lgG) + t.u;                // thread of the group
  const int lgc = 1 + lgG;                         // 16-byte pieces per k
  const char* const base = (const char*)src;
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int e = g + (m << t.lgt), k = e >> lgc;
    cp16(stg + e, base + k * (ny * (int)sizeof(C2<T>)) + ((e & ((1 << lgc) - 1)) << 4));
  }
  for (int e = g; e < (1 << lgc); e += 1 << t.lgt)
    cp16(top + e, base + (nx >> 1) * (ny * (int)sizeof(C2<T>)) + (e << 4));
  cp_commit();
}
__device__ __forceinline__ B32f staged_b32(const uint4* a, const C2<float>*) {
  const float4 x = *(const float4*)a, y = *(const float4*)(a + 1);
  return B32f{{x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w}};
}
__device__ __forceinline__ B32d staged_b32(const uint4* a, const C2<double>*) {
  const double2 x = *(const double2*)a, y = *(const double2*)(a + 1);
  return B32d{{x.x, x.y, y.x, y.y}};
}
template <typename T, int E>
__device__ __forceinline__ void row_gather_staged(CV<typename Lane<T>::V> (&v)[E], const Team<T, E>& t, int lgG, const uint4* stg, const uint4* top, int nx) {
  cp_wait();                                       // (the gather's first barrier makes the copies visible)
  row_gather_from(v, t, nx, [&](int j, int k) {
    return staged_b32((j < E / 2 ? stg + (k << (1 + lgG)) : top) + 2 * t.u, (const C2<T>*)nullptr);
  });
}
// The reverse: (twice) the half spectra of a unit's rows from the packed lines' transform.
template <typename T, int E>
__device__ __forceinline__ void row_scatter(CV<typename Lane<T>::V> (&v)[E], const Team<T, E>& t, C2<T>* dst, int nx, int ny, bool mine) {
  const int q = t.step();
  t.sync();
#pragma unroll
  for (int j = E / 2; j < E; ++j) t.at(t.i + j * q) = v[j];
  t.sync();
#pragma unroll
  for (int j = 0; j < E / 2; ++j) {
    const int k = t.i + j * q;
    const CV<typename Lane<T>::V> zm = k == 0 ? v[j] : t.at(nx - k);
    if (mine) st_b32(dst + k * ny, v[j], zm);
  }
  if (t.i == 0 && mine) st_b32(dst + (nx >> 1) * ny, v[E / 2], v[E / 2]);
}

}  // namespace mf
