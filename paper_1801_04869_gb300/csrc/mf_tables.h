// Host-side tables and launch shapes: twiddles of the transform core, elements per thread, fields and
// masks by row units.
#pragma once
#include <algorithm>
#include <cmath>

#include "mf_common.cuh"

namespace mf {

// Values of type T set aside per point of an axis for its twiddle table, which holds fewer than L
// entries of 4 (single) or 2 (double) values
constexpr size_t TWIDDLE_VALUES = 4;

// Table of the transform core (mf_core.cuh) for length L and E = 2^e elements per thread, stage after
// stage: p = E, E^2, ...: w^(2^m), m < e, with w = exp(-2 pi i k / (E p)) for k < p; a last stage of
// radix 2^r < E holds m < r with w = exp(-2 pi i k / L) for k < L / E.  E = 8 adds w exp(-i pi/4), which a
// product in the kernel would round twice more (error of a 2048^2 FP32 right-hand side against 64 bits
// 6.9e-7 -> 4.7e-7, at the same 758 us).  A single-precision entry is
// stored twice over, (re, re, im, im), for the packed instructions.  Returns the number of values of
// type T written.
template <typename T>
inline size_t core_twiddles(int L, int E, T* out) {
  int lg = 0, e = 0;
  while ((1 << lg) < L) ++lg;
  while ((1 << e) < E) ++e;
  size_t n = 0;
  int lgp = e;
  for (int rem = lg - e; rem > 0; rem -= e, lgp += e) {
    const int nk = rem >= e ? 1 << lgp : L >> e;
    const int den = rem >= e ? E << lgp : L;
    const int nm = rem >= e ? e : rem;
    for (int m = 0; m < nm + (E == 8 ? 1 : 0); ++m)
      for (int k = 0; k < nk; ++k) {
        const double ang = m < nm ? -2.0 * M_PI * (double)(k << m) / (double)den
                                  : -2.0 * M_PI * (double)k / (double)den - 0.25 * M_PI;
        const T c = (T)std::cos(ang), s = (T)std::sin(ang);
        if (sizeof(T) == 4) { out[n++] = c; out[n++] = c; out[n++] = s; out[n++] = s; }
        else { out[n++] = c; out[n++] = s; }
      }
  }
  return n;
}

// Launch shape of a film: a CTA per unit of the wider pass (its lines run on as few CTAs' threads
// as the pass leaves idle), no more than fit the GPU at once.
inline void film_shape(Desc& d, int coresident) {
  const int ru = row_unit(d.precision);
  const int rows = d.ny / ru, cols = (d.nx / 2 + 1 + ru / 2 - 1) / (ru / 2);
  const int want = rows > cols ? rows : cols;
  d.rows_per_item = ru;
  d.zs_per_item = ru;
  d.grid = want < coresident ? want : coresident;
}
// Elements per thread E of a film's passes along an axis of n points (mf_core.cuh).  A radix-E stage
// costs one exchange through shared memory, so the large films take E = 8 (2048 points: 3 exchanges
// per transform).  Where a pass does not fill the chip, its time is one thread's chain of
// instructions, and fewer elements per thread make it shorter.
//   FP64: an FP64 instruction occupies an SM sub-partition for 64 cycles whatever the number of
//     active lanes, so while E = 2 gives at most one warp per sub-partition (256^2 cells: 512 warps
//     on 608) the pass takes a quarter of the instructions of E = 8.  One right-hand side with 4 / 5 /
//     5 iterations at 64^2 / 128^2 / 256^2: 202 / 251 / 288 us against 389 / 514 / 550 us.  E = 4 above:
//     512 x 256 / 512^2 / 1024^2 427 / 540 / 2070 us against 441 / 570 us with E = 2 (lines of up to 512
//     points) and, with E = 8, 625 us at 512^2 and 2082 us at 1024^2.
//   FP32: E = 4 up to 2^20 cells (1024^2: 256 lines of 256 threads): 64^2 / 512^2 / 1024^2 with 5
//     iterations 171 / 216 / 304 us against 230 / 240 / 339 us with E = 8; lines of 2048 points would
//     need 512 threads.
inline int elems_per_thread(const Desc& d, int n) {
  const long long cells = (long long)d.nx * d.ny;
  if (d.precision == 0) return cells <= 65536 && n <= 2 * NT ? 2 : n <= 4 * NT ? 4 : 8;
  return cells <= 1048576 && n <= 4 * NT ? 4 : 8;
}

// Elements per thread and items of a bulk body's passes (the kernel has E = 4 / 8 in FP32, 2 / 4 in FP64
// along x, 4 and in FP32 8 along y, 4 and in FP64 2 along z).  Few elements where a pass does not fill
// the chip and one thread's chain of instructions sets its time, more (fewer exchanges) where the passes
// stream.  One right-hand side with 4 iterations, in us, with the smaller against the larger E:
//   x FP32: 4 to 2^21 cells: 128 x 64 x 64 / 128^3 588 / 1098 against 718 / 1175; 256 x 128 x 128 / 256^3
//     2140 / 8752 against 2004 / 7799.
//   x FP64: 2 to 2^18 cells: 64^3 1363 against 1437 (1822 with 8: an item of 64^3 is 4 row units of 8
//     threads then, one warp in a CTA, and three sub-partitions idle); 128 x 64 x 64 / 128 x 128 x 64 2358 /
//     4738 against 2339 / 4580 (4725 with 8).
//   y FP32: 4 to 2^18 cells: 64^3 460 against 467; 128 x 64 x 64 / 256^3 602 / 8534 against 588 / 7799.
//   y FP64: 4: 64 x 64 x 32 / 128 x 128 x 64 / 128^3 823 / 4725 / 9345 against 863 / 4827 / 9712 with 8.
//   z: three components are transformed together, so 4 (48 data registers); 2 for FP64 to 2^16 cells.
// An x item is a block of row units whose residual is summed together: as many as fill a CTA, but at
// least 304 items (two CTAs on each of 152 SMs), whatever the launch width, so that it changes nothing.
inline void bulk_shape(Desc& d, int coresident) {
  const bool f32 = d.precision != 0;
  d.ex = f32 ? (d.ncell <= 2097152 ? 4 : 8) : (d.ncell <= 262144 ? 2 : 4);
  d.ey = f32 && d.ncell > 262144 ? 8 : 4;
  d.ez = !f32 && d.ncell <= 65536 ? 2 : 4;
  const int ru = row_unit(d.precision);
  const long long units = (long long)d.nz * d.ny / ru;
  long long ub = NT / (d.nx / d.ex);
  while (ub > 1 && (units / ub < 304 || units % ub)) ub /= 2;
  d.rows_per_item = (int)ub * ru;
  d.zs_per_item = 1;
  const long long lines = 3LL * d.nz / (ru / 2) * (d.nx / 2 + 1);
  d.grid = (int)std::min<long long>(coresident, std::max(units / ub, lines));
}

// mask classes of `units` row units from the row-major mask of their rows, 2 bits per row
inline void pack_mask(const unsigned char* mask, int nx, int ru, long long units, unsigned char* out) {
  for (long long u = 0; u < units; ++u, mask += (long long)ru * nx, out += nx) {
    const unsigned char *a = mask, *b = mask + nx, *c = a, *d = b;
    if (ru == 4) {
      c = mask + 2 * (long long)nx;
      d = mask + 3 * (long long)nx;
      for (int x = 0; x < nx; ++x) out[x] = (unsigned char)(a[x] | b[x] << 2 | c[x] << 4 | d[x] << 6);
    } else {
      for (int x = 0; x < nx; ++x) out[x] = (unsigned char)(a[x] | b[x] << 2);
    }
  }
}
// a row-major field by row units, in the transform precision
template <typename T>
inline void field_by_units(const double* f, int nx, int ru, long long units, T* out) {
  for (long long u = 0; u < units; ++u, f += (long long)ru * nx)
    for (int x = 0; x < nx; ++x)
      for (int r = 0; r < ru; ++r) *out++ = (T)f[(long long)r * nx + x];
}

}  // namespace mf
