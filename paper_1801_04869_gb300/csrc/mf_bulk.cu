// Bulk (3D) right-hand side in the magnetic-field formulation and its BS23 integrator, as one
// persistent cooperative kernel.
//
// Method: Section 3.1 of Prigozhin & Sokolovsky (arXiv:1801.04869).  The state h has three
// components (component-major).  A vector "round trip" F^-1[M F(v)] runs as five passes
// separated by grid barriers, all on one spectrum S[c][z][kx][y] in place:
//   X   x pass: rows of the real field, R2C along x
//   Yf  y pass: forward along y (contiguous lines)
//   Z   z pass: forward along z, the 3x3 multiplier M, inverse along z
//   Yi  y pass: inverse along y
//   X   x pass: C2R along x, epilogue, and the forward x pass of the next round trip's input
// Multipliers: the Gaussian-smoothed curl i G k x (Section 3.1, last paragraph) and the
// Biot-Savart operator Phi = (i/|k|^2) k x (Eq. 17, 1/|k|^2 -> 0 at k = 0).
// One right-hand side (Eqs. 13-14 and the iteration of Eq. 18):
//   j = curl h;  e = rho(|j|) j (Eq. 13) or rho_out j;  h_dot_in = -curl e on the conductor
//   repeat: j_dot = curl h_dot, kept on the conductor;  h_dot_out = h_e_dot + Phi[j_dot] on
//   free space;  stop when mean_out |h_dot^{i+1} - h_dot^i| < delta_it max(|h_e_dot|, 1).
//
// The passes run on the transform core (mf_core.cuh); real fields and the mask lie by row units
// (mf_units.cuh).
//
// What bounds the passes, and what they measured (one right-hand side with 4 outside iterations; the
// design before kept two spectra per component and transformed 16 values per thread through two shared
// buffers): 256^3 FP32 by memory latency at 16 warps per SM, with 8 bytes per cell and component moved
// each way per pass (13.3 -> 7.8 ms), so that every pass brings its next unit's spectra to shared memory
// with asynchronous copies while it works on this one; 128^3 FP32 by the chain of loads, exchanges and
// barriers per unit (1.66 -> 1.10 ms); FP64 from 64^3 by the FP64 unit (64^3 1.64 -> 1.36 ms, 128^3 12.1 ->
// 9.2 ms); 32^3 by the latencies of 42 phases (FP32 390 -> 318 us, FP64 940 -> 578 us).
#include <type_traits>

#include "mf_units.cuh"

namespace mf {

enum Op3 { OP3_CURL = 0, OP3_CURLNEG = 1, OP3_PHI = 2 };

// raw pointers and sizes the x-pass epilogues need, held by value (registers)
template <typename T>
struct BulkPtrs {
  const uint8_t* mask;
  const T* jcmap;
  T* hd;
  int ncell, nx, ny;
};

template <typename T>
struct Bulk {
  using V = typename Lane<T>::V;
  static constexpr int RU = Lane<T>::RU, NL = Lane<T>::NL;
  const Desc& d;
  CV<V>* sm;         // the CTA's shared memory: a pass's exchange buffers, then its staging buffer, in which
                     // the next unit's spectra arrive while a unit is worked on
  Shared& sh;
  int nx, ny, nz, lgx, lgy, lgz, half, nkx;
  int nspec, ncell;  // indexes of the three components' values stay below 2^31 (512^3 cells)
  C2<T>* S;          // spectra of the three components, [c][z][kx][y]
  T* tmp;            // two real fields by row units (joint epilogues)
  T* hd;
  const uint8_t* mask;
  const T* jcmap;
  const CV<V>* twx; const CV<V>* twy; const CV<V>* twz;   // twiddle tables in shared memory
  const T* ktab; const T* gtab;     // kx (nkx), ky (ny), kz (nz)
  T scale;           // 1/(2 cells): the x pass leaves twice the half spectra
  T ig2, ib0;        // 1/gamma^2; 1/b0 of the Kim law, 0: none
  int ex, ey, ez, lgG, lgGx, ub, lgu;   // elements per thread; log2 lines per z, x group; row units per x item; log2 units per z
  int max_items;
  double* partials;
  GridBarrier* gb;
  unsigned long long barrier_ns;

  __device__ Bulk(const Desc& dd, unsigned char* smem, Shared& shr) : d(dd), sm((CV<V>*)smem), sh(shr) {
    nx = d.nx; ny = d.ny; nz = d.nz; lgx = d.lgx; lgy = d.lgy; lgz = d.lgz;
    half = nx / 2; nkx = half + 1;
    nspec = nkx * ny * nz;
    ncell = nx * ny * nz;
    S = (C2<T>*)d.Sa; tmp = (T*)d.Sb;
    hd = (T*)d.hd;
    mask = d.mask; jcmap = (const T*)d.jcmap;
    ex = d.ex; ey = d.ey; ez = d.ez;
    twx = sm + bulk_slots(d);
    const CV<V>* const t = twx + core_table_len(lgx, ex);
    twy = one_table(d) ? twx : t;
    twz = one_table(d) ? t : t + core_table_len(lgy, ey);
    ktab = (const T*)d.ktab; gtab = (const T*)d.gtab;
    scale = (T)0.5 / (T)ncell;
    ig2 = (T)(1.0 / (d.gamma * d.gamma));
    ib0 = d.b0 > 0.0 ? (T)(1.0 / d.b0) : (T)0;
    lgG = z_group_lg(lgz, ez);
    ub = d.rows_per_item / RU;
    lgGx = x_group_lg(d);
    lgu = lgy - (RU == 4 ? 2 : 1);
    max_items = d.max_items;
    partials = d.partials;
    gb = d.gb;
    barrier_ns = d.barrier_ns;
    sh.inv_nout = d.nout > 0 ? 1.0 / (double)d.nout : 0.0;
  }

  __device__ bool sync(int where) { return grid_sync(gb, gridDim.x, where, &sh.bar_passed, barrier_ns); }

  // members of the law's epilogues
  template <class Epi> __device__ __forceinline__ void law(Epi& e) const {
    e.n = (T)d.n; e.e0 = (T)d.e0; e.jc = (T)d.jc; e.rho_out = (T)d.rho_out;
    e.ig2 = ig2; e.ib0 = ib0;
  }

  __device__ BulkPtrs<T> ptrs() const { return BulkPtrs<T>{mask, jcmap, hd, ncell, nx, ny}; }

  // ---- x pass: up to 4 row units side by side on the lanes, so that a warp's accesses to the spectra
  // are 128 contiguous bytes per kx (32 with one unit); the spectra arrive by asynchronous copies (both
  // together: 256^3 FP32 8.28 -> 7.77 ms, 128^3 1.43 -> 1.19 ms).  Items of ub row units; per unit the components one after the other: inverse (NIN),
  // epilogue, forward (NOUT).  An epilogue that needs the three components of a cell together (kJoint)
  // lets the first two wait in `tmp` (the same thread's elements) while the third is transformed. ----
  template <int E, bool NIN, bool NOUT, class Epi>
  __device__ __noinline__ void xpass_e(const Epi& epi_in, int slot) {
    Epi epi = epi_in;                   // register copy of the epilogue
    const int nx = this->nx, ub = this->ub;
    const int ny = this->ny, nspec = this->nspec, ncell = this->ncell;
    const int lgG = this->lgGx;
    Team<T, E> t(sm, twx, lgx, lgG);
    const int q = t.step();
    const int nitems = (nz << lgu) / ub;
    const int first = (((int)threadIdx.x & ~31) >> t.lgt) << lgG;        // line of the warp's first lane
    const bool mine = t.slot < ub;
    // the group's part of the staging buffer, and its values at nx/2
    uint4* const stg0 = (uint4*)sm + x_slots(lgx, E);
    uint4* const stg = stg0 + (((int)threadIdx.x >> t.lgt) << (lgx + lgG));
    uint4* const top = stg0 + E * NT + (((int)threadIdx.x >> t.lgt) << (1 + lgG));
    Q<T>* const park = (Q<T>*)(stg0 + x_stage(lgx, E)) + threadIdx.x;    // this thread's slots, NT apart
    auto spectra = [&](int it, int slot) {
      const int unit = it * ub + (mine ? slot : 0);
      const int z = unit >> lgu, y0 = (unit - (z << lgu)) * RU;
      return S + z * nkx * ny + y0;
    };
    const int slot0 = t.slot - t.u;                                      // the group's first unit
    if (NIN && first < ub && (int)blockIdx.x < nitems) row_stage(t, lgG, stg, top, spectra((int)blockIdx.x, slot0), nx, ny);
    for (int it = (int)blockIdx.x; it < nitems; it += (int)gridDim.x) {
      epi.reset();
      if (first < ub) {
        const int unit = it * ub + (mine ? t.slot : 0);
        C2<T>* const Su = spectra(it, t.slot);
        // component c's spectra from the staging buffer; the next component's (item's) are then issued
        auto gather = [&](auto& v, int c) {
          row_gather_staged(v, t, lgG, stg, top, nx);
          const int nit = c < 2 ? it : it + (int)gridDim.x;
          if (nit < nitems) row_stage(t, lgG, stg, top, spectra(nit, slot0) + (c < 2 ? c + 1 : 0) * nspec, nx, ny);
        };
        const int iu = unit * nx + t.i;                 // 16-byte vector of a component
        const int ir = unit * RU * nx + t.i;            // row-major cell of the first row
        constexpr int B = Epi::kBatch < E ? Epi::kBatch : E;
        if constexpr (Epi::kJoint) {
          T* const tmp = this->tmp;
          CV<V> v[E];
#pragma unroll 1
          for (int c = 0; c < 3; ++c) {
            gather(v, c);
            core_fft<+1>(v, t);
            if (c < 2 && mine) {
#pragma unroll
              for (int j = 0; j < E; ++j) st_q(tmp + c * ncell + (iu + j * q) * RU, to_q(v[j]));
            }
          }
          if (mine) {
#pragma unroll
            for (int j0 = 0; j0 < E; j0 += B) {
              typename Epi::Ld ld[B];
              Q<T> in[B][3], out[3];
#pragma unroll
              for (int b = 0; b < B; ++b) {
                const int i = iu + (j0 + b) * q;
                ld[b] = epi.load(i, ir + (j0 + b) * q);
                in[b][0] = ld_q(tmp + i * RU);
                in[b][1] = ld_q(tmp + ncell + i * RU);
                in[b][2] = to_q(v[j0 + b]);
              }
#pragma unroll
              for (int b = 0; b < B; ++b) {
                const int i = iu + (j0 + b) * q;
                epi.apply(ld[b], t.i + (j0 + b) * q, unit, ir + (j0 + b) * q, in[b], out);
                if constexpr (NOUT) {
                  st_q(tmp + i * RU, out[0]);
                  st_q(tmp + ncell + i * RU, out[1]);
                  v[j0 + b] = to_e(out[2]);
                }
              }
            }
          }
          if constexpr (NOUT) {
#pragma unroll 1
            for (int c = 2; c >= 0; --c) {
              if (c < 2) {
#pragma unroll
                for (int j = 0; j < E; ++j) v[j] = to_e(ld_q(tmp + c * ncell + (iu + j * q) * RU));
              }
              core_fft<-1>(v, t);
              row_scatter(v, t, Su + c * nspec, nx, ny, mine);
            }
          }
        } else {
#pragma unroll 1
          for (int c = 0; c < 3; ++c) {
            CV<V> v[E];
            typename Epi::Ld ld[2][B];
            if constexpr (NIN) gather(v, c);
#pragma unroll
            for (int b = 0; b < B; ++b) ld[0][b] = epi.load(c, iu + b * q, ir + b * q);
            if constexpr (NIN) core_fft<+1>(v, t);
#pragma unroll
            for (int j0 = 0; j0 < E; j0 += B) {
              if (j0 + B < E) {
#pragma unroll
                for (int b = 0; b < B; ++b) ld[(j0 / B + 1) & 1][b] = epi.load(c, iu + (j0 + B + b) * q, ir + (j0 + B + b) * q);
              }
              if (mine) {
#pragma unroll
                for (int b = 0; b < B; ++b) {
                  const int j = j0 + b;
                  Q<T> in, out;
                  if constexpr (NIN) in = to_q(v[j]);
                  epi.apply(ld[(j0 / B) & 1][b], c, park + j * NT, iu + j * q, ir + j * q, in, out);
                  if constexpr (NOUT) v[j] = to_e(out);
                }
              }
            }
            if constexpr (NOUT) {
              core_fft<-1>(v, t);
              row_scatter(v, t, Su + c * nspec, nx, ny, mine);
            }
          }
        }
      }
      if (slot >= 0) {
        const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        constexpr int NS = Epi::kSums;
        __syncthreads();                // the item before has been summed
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          if constexpr (Epi::kMax) {
            const auto m = warp_max((double)epi.acc[k]);
            if (l == 0) sh.redn[k][w] = m;
          } else {
            const auto s = warp_sum(epi.acc[k]);
            if (l == 0) sh.redn[k][w] = (double)s;
          }
        }
        __syncthreads();
        if (l == 0 && w < NS) {         // one sum per warp: an FP64 addition takes 64 cycles
          double s = sh.redn[w][0];
          for (int k = 1; k < NT / 32; ++k) s = Epi::kMax ? fmax(s, sh.redn[w][k]) : s + sh.redn[w][k];
          partials[(size_t)(slot + w) * max_items + it] = s;
        }
      }
    }
  }
  // fill(epi) sets the epilogue's members
  template <template <class, int> class EPI, bool NIN, bool NOUT, class Fill>
  __device__ __forceinline__ void xpass(Fill fill, int slot = -1) {
    constexpr int FEW = sizeof(T) == 4 ? 4 : 2, MANY = 2 * FEW;
    if (ex == FEW) {
      EPI<T, FEW> e;
      e.P = ptrs();
      fill(e);
      xpass_e<FEW, NIN, NOUT>(e, slot);
    } else {
      EPI<T, MANY> e;
      e.P = ptrs();
      fill(e);
      xpass_e<MANY, NIN, NOUT>(e, slot);
    }
  }
  __device__ double total(int slot, bool is_max = false) {
    return reduce_partials(partials, max_items, slot, (nz << lgu) / ub, is_max, sh.red);
  }

  // ---- y pass: contiguous lines in place, z neighbours together in FP32; kx slowest ----
  template <int E, int DIR>
  __device__ __noinline__ void ypass_e() {
    const int ny = this->ny, nspec = this->nspec, nkx = this->nkx;
    Team<T, E> t(sm, twy, lgy);
    const int q = t.step();
    const int nzp = nz / NL, units = 3 * nzp * (int)nkx;
    const int per = NT / t.threads(), want = (units + (int)gridDim.x - 1) / (int)gridDim.x;
    const int nuc = want < per ? want : per;
    const int first = ((int)threadIdx.x & ~31) >> (lgy - lg_of(E));
    const int next = nkx * ny;         // the line of z + 1
    auto line = [&](int u) {
      const int kx = u / (3 * nzp), r = u - kx * 3 * nzp, c = r / nzp, z = (r - c * nzp) * NL;
      return S + c * nspec + (z * nkx + kx) * ny;
    };
    // a unit's NL lines lie one after the other in its part of the staging buffer, 16 bytes per copy
    uint4* const stg = (uint4*)sm + slots_of(E) + ((t.slot * t.threads()) << lg_of(E));
    auto issue = [&](const C2<T>* p) {
      const int half_l = 1 << (lgy - (NL - 1));          // 16-byte pieces per line
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const int k = t.i + j * q, l = NL == 2 ? k >> (lgy - 1) : 0;
        cp16(stg + k, (const uint4*)(p + l * next) + (k & (half_l - 1)));
      }
      cp_commit();
    };
    if (first >= nuc) return;
    int u0 = (int)blockIdx.x * nuc;
    auto unit_of = [&](int u0) { return t.slot < nuc && u0 + t.slot < units ? u0 + t.slot : u0; };
    if (u0 + first < units) issue(line(unit_of(u0)));
    for (; u0 + first < units; u0 += (int)gridDim.x * nuc) {
      const bool mine = t.slot < nuc && u0 + t.slot < units;
      C2<T>* const p = line(unit_of(u0)) + t.i;
      CV<V> v[E];
      cp_wait();
      t.sync();
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const C2<T>* const a = (const C2<T>*)stg + t.i + j * q;
        if constexpr (NL == 2) {
          const C2<T> x = a[0], y = a[1 << lgy];
          v[j] = {pk(x.x, y.x), pk(x.y, y.y)};
        } else {
          v[j] = {a[0].x, a[0].y};
        }
      }
      t.sync();                              // every thread has read: the next unit's lines may land
      const int nu = u0 + (int)gridDim.x * nuc;
      if (nu + first < units) issue(line(unit_of(nu)));
      core_fft<DIR>(v, t);
      if (mine) {
#pragma unroll
        for (int j = 0; j < E; ++j) st_col(p + j * q, next, true, v[j]);
      }
    }
  }
  template <int DIR> __device__ __forceinline__ void ypass() {
    if (sizeof(T) == 8 || ey == 4) ypass_e<4, DIR>();
    else ypass_e<8, DIR>();
  }

  // ---- z pass: forward, 3x3 multiplier, inverse on groups of lines (kx, y0 ..), the three components of
  // a line in one thread's registers, so that the multiplier needs no exchange and the transforms share
  // their barriers; bound by the exchanges through shared memory and their barriers (256^3 FP32: some
  // 27 k cycles per group of 4 lines, of which the exchanges' bytes account for 11 k) ----
  static __device__ __forceinline__ CV<F2> ld_z(const float4& f) { return {pk(f.x, f.z), pk(f.y, f.w)}; }
  static __device__ __forceinline__ CV<double> ld_z(const double2& f) { return {f.x, f.y}; }
  static __device__ __forceinline__ void st_z(C2<float>* p, const CV<F2>& v) {
    float4 f;
    upk(v.x, f.x, f.z);
    upk(v.y, f.y, f.w);
    *(float4*)p = f;
  }
  static __device__ __forceinline__ void st_z(C2<double>* p, const CV<double>& v) { st_col(p, 0, false, v); }
  // 1/k2 (0 at k = 0)
  static __device__ __forceinline__ T inv(T k2) {
    if constexpr (sizeof(T) == 4) return k2 > 0.f ? __frcp_rn(k2) : 0.f;
    const T r = k2 > (T)0 ? rsqrt(k2) : (T)0;
    return r * r;
  }
  template <int E>
  __device__ __noinline__ void zpass_e(int op) {
    const int ny = this->ny, half = this->half;
    const int nspec = this->nspec, zs = nkx * ny;
    Team<T, E> t(sm, twz, lgz, lgG);
    const int q = t.step();
    const int gl = NL << lgG, ngy = ny / gl;                  // y lines per group, groups per kx
    const int units = nkx * ngy;
    const int per = NT >> t.lgt, slot = (int)threadIdx.x >> t.lgt, want = (units + (int)gridDim.x - 1) / (int)gridDim.x;
    const int nuc = want < per ? want : per;
    const int first = ((int)threadIdx.x & ~31) >> t.lgt;
    using Raw = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    uint4* const stg = (uint4*)sm + z_slots(lgz, E) + threadIdx.x;       // this thread's elements, NT apart
    // from the last kx to the first: what the y pass before left in L2 last comes first
    auto group_of = [&](int u0) { return units - 1 - (slot < nuc && u0 + slot < units ? u0 + slot : u0); };
    auto lines = [&](int g) {
      const int kx = g / ngy, y = (g - kx * ngy) * gl + t.u * NL;
      return S + kx * ny + y + t.i * zs;
    };
    auto issue = [&](const C2<T>* p) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int j = 0; j < E; ++j) cp16(stg + (c * E + j) * NT, p + c * nspec + j * q * zs);
      }
      cp_commit();
    };
    if (first >= nuc) return;
    int u0 = (int)blockIdx.x * nuc;
    if (u0 + first < units) issue(lines(group_of(u0)));
    for (; u0 + first < units; u0 += (int)gridDim.x * nuc) {
      const bool mine = slot < nuc && u0 + slot < units;
      const int g = group_of(u0);
      const int kx = g / ngy, y = (g - kx * ngy) * gl + t.u * NL;
      C2<T>* const p = lines(g);
      CV<V> v[3][E];
      cp_wait();
#pragma unroll
      for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int j = 0; j < E; ++j) v[c][j] = ld_z(*(const Raw*)(stg + (c * E + j) * NT));
      }
      t.sync();                              // the elements have been read: the next group's may land
      const int nu = u0 + (int)gridDim.x * nuc;
      if (nu + first < units) issue(lines(group_of(nu)));
      // wavenumbers of the line(s); odd multipliers are 0 at the Nyquist index of their axis
      const T kx1 = ldg_tab(&ktab[kx]), gx = ldg_tab(&gtab[kx]);
      const T kxo = kx == half ? (T)0 : kx1;
      V ky, ky2, gxy;
      if constexpr (sizeof(T) == 4) {
        const float a = ldg_tab(&ktab[nkx + y]), b = ldg_tab(&ktab[nkx + y + 1]);
        ky = pk(y == (ny >> 1) ? 0.f : a, y + 1 == (ny >> 1) ? 0.f : b);
        ky2 = pk(fmaf(kx1, kx1, a * a), fmaf(kx1, kx1, b * b));
        gxy = pk(gx * ldg_tab(&gtab[nkx + y]), gx * ldg_tab(&gtab[nkx + y + 1]));
      } else {
        const double a = ldg_tab(&ktab[nkx + y]);
        ky = y == (ny >> 1) ? 0.0 : a;
        ky2 = fma(kx1, kx1, a * a);
        gxy = gx * ldg_tab(&gtab[nkx + y]);
      }
      core_fft_n<-1, 3>(v, t);
      const V kxv = vset(kxo, (V*)nullptr), nkxv = vneg(kxv), nky = vneg(ky);
      const T sc = op == OP3_CURLNEG ? -scale : scale;
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const int kz = t.i + j * q;
        const T kz1 = ldg_tab(&ktab[nkx + ny + kz]);
        const V kzv = vset(kz == (nz >> 1) ? (T)0 : kz1, (V*)nullptr), nkz = vneg(kzv);
        V f;
        if (op == OP3_PHI) {                                 // Eq. 17
          const V k2 = vfma(vset(kz1, (V*)nullptr), vset(kz1, (V*)nullptr), ky2);
          if constexpr (sizeof(T) == 4) {
            float a, b;
            upk(k2, a, b);
            f = pk(inv(a) * sc, inv(b) * sc);
          } else {
            f = inv(k2) * sc;
          }
        } else {                                             // smoothed curl
          f = vmul(gxy, vset(ldg_tab(&gtab[nkx + ny + kz]) * sc, (V*)nullptr));
        }
        // i f (k x v)
        const CV<V> a = v[0][j], b = v[1][j], c = v[2][j];
        const CV<V> x = {vfma(ky, c.x, vmul(nkz, b.x)), vfma(ky, c.y, vmul(nkz, b.y))};
        const CV<V> yv = {vfma(kzv, a.x, vmul(nkxv, c.x)), vfma(kzv, a.y, vmul(nkxv, c.y))};
        const CV<V> z = {vfma(kxv, b.x, vmul(nky, a.x)), vfma(kxv, b.y, vmul(nky, a.y))};
        const V nf = vneg(f);
        v[0][j] = {vmul(x.y, nf), vmul(x.x, f)};
        v[1][j] = {vmul(yv.y, nf), vmul(yv.x, f)};
        v[2][j] = {vmul(z.y, nf), vmul(z.x, f)};
      }
      core_fft_n<+1, 3>(v, t);
      if (mine) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
          for (int j = 0; j < E; ++j) st_z(p + c * nspec + j * q * zs, v[c][j]);
        }
      }
    }
  }
  __device__ __forceinline__ void zpass(int op) {
    if constexpr (sizeof(T) == 8) {
      if (ez == 2) { zpass_e<2>(op); return; }
    }
    zpass_e<4>(op);
  }

  // Yf, Z(op), Yi with barriers; the x passes before and after are separate
  __device__ bool yzy(int op, int where) {
    ypass<-1>();
    if (!sync(where)) return false;
    zpass(op);
    if (!sync(where + 1)) return false;
    ypass<+1>();
    return sync(where + 2);
  }
};

// ------------------------------------------------------------------------------------------
// Epilogues of the x pass.  load(c, i, r) reads what the RU rows of one element of component c need (i:
// the component's 16-byte vector, r: the row-major cell of the first row, the others nx apart);
// apply(ld, c, s, i, r, in, out) works on one element, which has 16 bytes of shared memory s of its own
// for what passes from component to component; reset() starts an item.  Joint ones take the three
// components at once.
// ------------------------------------------------------------------------------------------
template <typename T, int NS = 1, bool MAX = false>
struct BEpi {
  BulkPtrs<T> P;
  static constexpr int RU = Lane<T>::RU, kSums = NS, kBatch = 4;
  static constexpr bool kJoint = false, kMax = MAX;
  T acc[NS];
  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0;
  }
  __device__ __forceinline__ int msk(int i) const { return ld_mask(P.mask + i); }
};

// Stage state y + sum c_j k_j.
template <typename T, int E>
struct BStage : BEpi<T> {
  static constexpr int RU = Lane<T>::RU, kBatch = 2;
  StageIn in;
  struct Ld { double v[RU]; };
  __device__ __forceinline__ double value(int o) const {
    double v = ld_s(in.y + o);
    for (int j = 0; j < in.nk; ++j) v += in.c[j] * ld_s(in.k[j] + o);
    return v;
  }
  __device__ __forceinline__ Ld load(int c, int, int r) const {
    Ld l;
    const int o = c * this->P.ncell + r;
#pragma unroll
    for (int q = 0; q < RU; ++q) l.v[q] = ld_s(in.y + o + q * this->P.nx);
    for (int j = 0; j < in.nk; ++j) {
      double k[RU];
#pragma unroll
      for (int q = 0; q < RU; ++q) k[q] = ld_s(in.k[j] + o + q * this->P.nx);
#pragma unroll
      for (int q = 0; q < RU; ++q) l.v[q] += in.c[j] * k[q];
    }
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int c, Q<T>*, int, int r, const Q<T>&, Q<T>& out) {
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      if (in.ynew) in.ynew[c * this->P.ncell + r + q * this->P.nx] = l.v[q];
      out.v[q] = (T)l.v[q];
    }
  }
};
// The same with a field-dependent critical current: the stage field's magnitude |h| is kept, in the
// transform precision, in the first component of the h_dot iterate at superconductor cells: those entries
// are rewritten by BInit before anything reads them as an iterate, and the warm start lives on free space
// only.  (The sum of squares in FP64, from all three components with the last one.)
template <typename T, int E>
struct BStageKim : BStage<T, E> {
  static constexpr int RU = Lane<T>::RU, kBatch = 1;
  using Ld = typename BStage<T, E>::Ld;
  __device__ __forceinline__ void apply(const Ld& l, int c, Q<T>* s, int i, int r, const Q<T>& in, Q<T>& out) {
    BStage<T, E>::apply(l, c, s, i, r, in, out);
    if (c < 2) return;
    const int m = this->msk(i);
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      if (cls(m, q) != 1) continue;
      const int o = r + q * this->P.nx;
      const double a = this->value(o), b = this->value(this->P.ncell + o);
      this->P.hd[i * RU + q] = (T)sqrt(a * a + b * b + l.v[q] * l.v[q]);
    }
  }
};

// j -> e (Eq. 13 / Ohm law): critical current jc, per cell or Kim-type jc / (1 + |h|/b0) when ib0 > 0
// (|h| left by BStageKim), and the elliptic weight 1/gamma^2 of j_z
template <typename T>
struct BLaw : BEpi<T> {
  static constexpr int RU = Lane<T>::RU, kBatch = 1;
  static constexpr bool kJoint = true;
  T n, e0, jc, rho_out, ig2, ib0;
  struct Ld { int m; Q<T> jc, h; };
  __device__ __forceinline__ Ld load(int i, int) const {
    Ld l;
    l.m = this->msk(i);
    if (this->P.jcmap) {
      l.jc = ldg_q(this->P.jcmap + i * RU);
    } else {
#pragma unroll
      for (int q = 0; q < RU; ++q) l.jc.v[q] = jc;
    }
    if (ib0 > (T)0) l.h = ld_q(this->P.hd + i * RU);
    return l;
  }
  __device__ __forceinline__ void law(const Ld& l, const Q<T>* in, Q<T>* e) const {
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      const int m = cls(l.m, q);
      T jcl = l.jc.v[q];
      if (ib0 > (T)0 && m == 1) jcl = jcl / ((T)1 + l.h.v[q] * ib0);
      const T a = m == 1 ? ig2 : (T)1;
      const T x = in[0].v[q], y = in[1].v[q], z = in[2].v[q];
      const T rho = resistivity<T>(x * x + y * y + z * z * a, jcl, m, n, e0, rho_out);
      e[0].v[q] = rho * x; e[1].v[q] = rho * y; e[2].v[q] = rho * z * a;
    }
  }
};
template <typename T, int E>
struct BPower : BLaw<T> {
  using Ld = typename BLaw<T>::Ld;
  __device__ __forceinline__ void apply(const Ld& l, int, int, int, const Q<T>* in, Q<T>* out) { this->law(l, in, out); }
};
template <typename T, int E>
struct BStoreE : BLaw<T> {                 // readout of e (FP64)
  using Ld = typename BLaw<T>::Ld;
  double* out;
  __device__ __forceinline__ void apply(const Ld& l, int, int, int r, const Q<T>* in, Q<T>*) {
    Q<T> e[3];
    this->law(l, in, e);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int q = 0; q < Lane<T>::RU; ++q) out[c * this->P.ncell + r + q * this->P.nx] = e[c].v[q];
    }
  }
};

template <typename T, int E>
struct BInit : BEpi<T> {                   // h_dot^0: h_dot_in on the conductor, warm or h_e_dot outside
  static constexpr int RU = Lane<T>::RU, kBatch = 2;
  bool warm;
  T hed[3];
  struct Ld { int m; Q<T> w; };
  __device__ __forceinline__ Ld load(int c, int i, int) const {
    Ld l;
    l.m = this->msk(i);
    if (warm) l.w = ld_q(this->P.hd + (c * this->P.ncell + i * RU));
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int c, Q<T>*, int i, int, const Q<T>& in, Q<T>& out) {
    const T he = c == 0 ? hed[0] : c == 1 ? hed[1] : hed[2];
#pragma unroll
    for (int q = 0; q < RU; ++q) out.v[q] = cls(l.m, q) != 0 ? in.v[q] : warm ? l.w.v[q] : he;   // -curl e (Eq. 14)
    st_q(this->P.hd + (c * this->P.ncell + i * RU), out);
  }
};

template <typename T, int E>
struct BMaskCond : BEpi<T> {               // j_dot_in: keep on the conductor only
  struct Ld { int m; };
  __device__ __forceinline__ Ld load(int, int i, int) const { return Ld{this->msk(i)}; }
  __device__ __forceinline__ void apply(const Ld& l, int, Q<T>*, int, int, const Q<T>& in, Q<T>& out) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) out.v[q] = cls(l.m, q) != 0 ? in.v[q] : (T)0;
  }
};

template <typename T, int E>
struct BUpdate : BEpi<T> {                 // Eq. 18 on free space, residual, forward
  static constexpr int RU = Lane<T>::RU, kBatch = 2;
  T hed[3];
  struct Ld { int m; Q<T> h; };
  __device__ __forceinline__ Ld load(int c, int i, int) const {
    return Ld{this->msk(i), ld_q(this->P.hd + (c * this->P.ncell + i * RU))};
  }
  // s: |h_dot^{i+1} - h_dot^i|^2 of the element's cells over the components so far
  __device__ __forceinline__ void apply(const Ld& l, int c, Q<T>* s, int i, int, const Q<T>& in, Q<T>& out) {
    const T he = c == 0 ? hed[0] : c == 1 ? hed[1] : hed[2];
    Q<T> e2;
    if (c > 0) e2 = *s;
    out = l.h;
    bool any = false;
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      T e = (T)0;
      if (cls(l.m, q) == 0) {
        const T n = he + in.v[q];
        e = n - l.h.v[q];
        out.v[q] = n;
        any = true;
      }
      e2.v[q] = c == 0 ? e * e : e2.v[q] + e * e;
      if (c == 2) this->acc[0] += sqrt(e2.v[q]);
    }
    if (any) st_q(this->P.hd + (c * this->P.ncell + i * RU), out);
    if (c < 2) *s = e2;
  }
};

template <typename T, int E, bool err>
struct BFinalT : BEpi<T, 1, true> {        // h_dot out (FP64); optional BS23 error contribution
  static constexpr int RU = Lane<T>::RU, NE = err ? RU : 1, kBatch = err ? 1 : 4;
  double* kout;
  double h, rtol, atol;
  const double* k1; const double* k2; const double* k3; const double* y; const double* ynew;
  struct Ld { Q<T> g; double a1[NE], a2[NE], a3[NE], y[NE], yn[NE]; };
  __device__ __forceinline__ Ld load(int c, int i, int r) const {
    Ld l;
    l.g = ld_q(this->P.hd + (c * this->P.ncell + i * RU));
    if constexpr (err) {
#pragma unroll
      for (int q = 0; q < RU; ++q) {
        const int o = c * this->P.ncell + r + q * this->P.nx;
        l.a1[q] = ld_s(k1 + o); l.a2[q] = ld_s(k2 + o); l.a3[q] = ld_s(k3 + o);
        l.y[q] = ld_s(y + o); l.yn[q] = ld_s(ynew + o);
      }
    }
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int c, Q<T>*, int, int r, const Q<T>&, Q<T>&) {
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      const double g = (double)l.g.v[q];
      kout[c * this->P.ncell + r + q * this->P.nx] = g;
      if constexpr (err) {
        const double E_ = h * (-5.0 / 72.0 * l.a1[q] + 1.0 / 12.0 * l.a2[q] + 1.0 / 9.0 * l.a3[q] - 0.125 * g);
        const double sc = atol + rtol * fmax(fabs(l.y[q]), fabs(l.yn[q]));
        T e;                                                 // the ratio in the transform precision
        if constexpr (sizeof(T) == 4) e = __fdiv_rn((float)fabs(E_), (float)sc);
        else e = fabs(E_) / sc;
        if (!(e == e)) e = (T)INFINITY;                      // non-finite -> rejected step
        this->acc[0] = this->acc[0] > e ? this->acc[0] : e;
      } else if (!isfinite(l.g.v[q])) {
        this->acc[0] = (T)1;
      }
    }
  }
};
template <typename T, int E> using BFinal = BFinalT<T, E, false>;
template <typename T, int E> using BFinalErr = BFinalT<T, E, true>;

template <typename T, int E>
struct BStoreJ : BEpi<T> {                 // readout of j = curl h (FP64)
  double* out;
  using Ld = NoLd;
  __device__ __forceinline__ Ld load(int, int, int) const { return Ld{}; }
  __device__ __forceinline__ void apply(const Ld&, int c, Q<T>*, int, int r, const Q<T>& in, Q<T>&) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) out[c * this->P.ncell + r + q * this->P.nx] = in.v[q];
  }
};

template <typename T, int E>
struct BMoment : BEpi<T, 3> {              // m = 1/2 sum dV r x j over the conductor
  static constexpr int RU = Lane<T>::RU, kBatch = 2;
  static constexpr bool kJoint = true;
  double acc[3];
  double Lx, Ly, Lz, dx, dy, dz;
  struct Ld { int m; };
  __device__ __forceinline__ void reset() { acc[0] = acc[1] = acc[2] = 0.0; }
  __device__ __forceinline__ Ld load(int i, int) const { return Ld{this->msk(i)}; }
  __device__ __forceinline__ void apply(const Ld& l, int x, int unit, int, const Q<T>* in, Q<T>*) {
    if (l.m == 0) return;
    const int row = unit * RU, z = row / this->P.ny, y0 = row - z * this->P.ny;
    const double rx = -Lx + (x + 0.5) * dx, rz = -Lz + (z + 0.5) * dz;
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      if (cls(l.m, q) == 0) continue;
      const double ry = -Ly + (y0 + q + 0.5) * dy;
      const double jx = in[0].v[q], jy = in[1].v[q], jz = in[2].v[q];
      acc[0] += ry * jz - rz * jy;
      acc[1] += rz * jx - rx * jz;
      acc[2] += rx * jy - ry * jx;
    }
  }
};

// ------------------------------------------------------------------------------------------
// one bulk right-hand side
// ------------------------------------------------------------------------------------------
template <typename T>
__device__ __noinline__ RhsOut bulk_rhs(Bulk<T>& B, double t, int seg, const StageIn& sin, double* kout,
                                        int force_iters, bool want_err, double h_err, const double* e_k1,
                                        const double* e_k2, const double* e_k3, const double* e_y,
                                        const double* e_ynew) {
  const Desc& d = B.d;
  Shared& sh = B.sh;
  RhsOut res{ST_OK, 0, 0.0, 0.0, 0};
  if (threadIdx.x == 0) {               // scalar FP64 work: one thread (see Control)
    const double hs = he_dot(d, t, seg);
    double n2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      sh.hed3[c] = hs * d.he_dir[c];
      sh.hed3f[c] = (float)sh.hed3[c];
      n2 += sh.hed3[c] * sh.hed3[c];
    }
    sh.thresh = d.iter_tol * fmax(sqrt(n2), 1.0);
    sh.r = 0.0;
  }
  auto hed = [&](T* e) {
    for (int c = 0; c < 3; ++c) {
      if constexpr (sizeof(T) == 4) e[c] = sh.hed3f[c];
      else e[c] = sh.hed3[c];
    }
  };
#define BSYNC(w) if (!B.sync(w)) { res.status = ST_BARRIER; return res; }
#define BYZY(op, w) if (!B.yzy(op, w)) { res.status = ST_BARRIER; return res; }
  if (d.b0 > 0.0) B.template xpass<BStageKim, false, true>([&](auto& e) { e.in = sin; });
  else B.template xpass<BStage, false, true>([&](auto& e) { e.in = sin; });
  BSYNC(101);
  BYZY(OP3_CURL, 102);                                                   // j = curl h
  B.template xpass<BPower, true, true>([&](auto& e) { B.law(e); });      // e = rho j
  BSYNC(105);
  BYZY(OP3_CURLNEG, 106);                                                // -curl e
  B.template xpass<BInit, true, true>([&](auto& e) { e.warm = sh.warm_valid != 0; hed(e.hed); });   // h_dot^0
  BSYNC(109);
  const bool have_out = d.nout > 0;
  const bool by_count = force_iters > 0 || d.iter_tol <= 0.0;
  const int itmax = force_iters > 0 ? force_iters : d.iter_max;
  int i = 0;
  if (have_out) {
    for (; i < itmax; ++i) {
      BYZY(OP3_CURL, 110);                                               // j_dot = curl h_dot
      B.template xpass<BMaskCond, true, true>([&](auto&) {});            // j_dot_in
      BSYNC(113);
      BYZY(OP3_PHI, 114);                                                // Phi[j_dot_in]
      B.template xpass<BUpdate, true, true>([&](auto& e) { hed(e.hed); }, 0);   // Eq. 18
      BSYNC(117);
      const double s = B.total(0);
      if (threadIdx.x == 0) {
        sh.r = s * sh.inv_nout;
        sh.stop = !by_count && sh.r < sh.thresh;
      }
      __syncthreads();
      if (sh.stop) { ++i; break; }
    }
    if (i > itmax) i = itmax;
  }
  res.iters = i;
  if (threadIdx.x == 0) {
    const double r = sh.r;
    sh.ok = !have_out || d.iter_tol <= 0.0 || r < sh.thresh;
    // a call that failed with a residual above 1e3 times the threshold (or not finite) diverged:
    // the next call starts cold
    sh.warm_valid = !sh.ok && !(r < 1e3 * sh.thresh) ? 0 : 1;
  }
  {
    auto fill = [&](auto& e) {
      e.kout = kout; e.h = h_err; e.rtol = d.rtol; e.atol = d.atol;
      e.k1 = e_k1; e.k2 = e_k2; e.k3 = e_k3; e.y = e_y; e.ynew = e_ynew;
    };
    if (want_err) B.template xpass<BFinalErr, false, false>(fill, 3);
    else B.template xpass<BFinal, false, false>(fill, 3);
  }
  BSYNC(120);
  res.status = sh.ok ? ST_OK : ST_NOCONV;
  res.r = sh.r;
  const double q = B.total(3, true);
  if (want_err) res.err = isinf(q) ? 1e300 : q;
  else res.nonfinite = __double_as_longlong(q) > 0;
#undef BSYNC
#undef BYZY
  return res;
}

template <typename T>
struct BulkRhs {
  Bulk<T>& B;
  __device__ RhsOut operator()(double t, int seg, const StageIn& in, double* kout, int force,
                               bool want_err, double h, const double* k1, const double* k2,
                               const double* k3, const double* y, const double* yn) {
    return bulk_rhs<T>(B, t, seg, in, kout, force, want_err, h, k1, k2, k3, y, yn);
  }
  __device__ void on_accept() {}     // 3D: every call starts from the most recent iterate
  __device__ void on_attempt() {}
};

template <typename T>
__global__ void __launch_bounds__(NT, 2) bulk_kernel(const Desc* __restrict__ dg, KernelArgs a) {
  __shared__ Shared sh;
  // one copy of the pass object per CTA, in shared memory: its members are read as broadcasts
  // instead of per-thread local-memory copies
  __shared__ __align__(16) unsigned char objraw[sizeof(Bulk<T>)];
  const Desc& d = *dg;
  SolverState* st = d.st;
  if (threadIdx.x == 0) {
    sh.warm_valid = st->warm_valid;
    sh.bar_passed = 0;
    sh.A_prev = 0.0;
    new (objraw) Bulk<T>(d, mf_dsmem, sh);
  }
  {
    // the twiddle tables, behind the exchange buffer (see film_tables)
    uint4* to = (uint4*)mf_dsmem + bulk_slots(d);
    auto copy = [&](const void* tab, int n) {
      for (int k = threadIdx.x; k < n; k += NT) to[k] = ((const uint4*)tab)[k];
      to += n;
    };
    copy(d.tw_x, core_table_len(d.lgx, d.ex));
    if (!one_table(d)) copy(d.tw_y, core_table_len(d.lgy, d.ey));
    copy(d.tw_z, core_table_len(d.lgz, d.ez));
  }
  __syncthreads();
  Bulk<T>& B = *reinterpret_cast<Bulk<T>*>(objraw);
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  int status = ST_OK;

  if (a.mode == MODE_RHS) {
    StageIn in{a.y_in, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
    RhsOut r = bulk_rhs<T>(B, a.t, a.seg, in, a.out, a.force_iters, false, 0.0, nullptr, nullptr,
                           nullptr, nullptr, nullptr);
    status = r.status == ST_OK && r.nonfinite ? ST_NONFINITE : r.status;
    if (leader) { st->last_iters = r.iters; st->last_r = r.r; st->n_rhs += 1; st->n_iters += r.iters; }
  } else if (a.mode == MODE_J || a.mode == MODE_E || a.mode == MODE_MOMENT) {
    StageIn in{a.y_in, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
    if (a.mode == MODE_E && d.b0 > 0.0) B.template xpass<BStageKim, false, true>([&](auto& e) { e.in = in; });
    else B.template xpass<BStage, false, true>([&](auto& e) { e.in = in; });
    bool ok = B.sync(201) && B.yzy(OP3_CURL, 202);
    if (ok) {
      if (a.mode == MODE_J) {
        B.template xpass<BStoreJ, true, false>([&](auto& e) { e.out = a.out; });
      } else if (a.mode == MODE_E) {
        B.template xpass<BStoreE, true, false>([&](auto& e) { B.law(e); e.out = a.out; });
      } else {
        B.template xpass<BMoment, true, false>([&](auto& e) {
          e.Lx = d.Lx; e.Ly = d.Ly; e.Lz = d.Lz; e.dx = d.dx; e.dy = d.dy; e.dz = d.dz;
        }, 4);
        ok = B.sync(205);
        if (ok) {
          for (int c = 0; c < 3; ++c) {
            const double s = B.total(4 + c);
            if (leader) a.out[c] = 0.5 * s * d.dx * d.dy * d.dz;
          }
        }
      }
    }
    if (!ok) status = ST_BARRIER;
  } else if (a.mode == MODE_ADVANCE) {
    BulkRhs<T> R{B};
    status = bs23_advance(R, d, st, a, leader, sh.ctl);
  }
  if (leader) {
    st->warm_valid = sh.warm_valid;
    st->status = status;
    publish_state(d, st);
  }
}

int bulk_max_blocks(int precision, size_t smem) {
  int nb = 0;
  if (precision) {
    cudaFuncSetAttribute(bulk_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BULK_SMEM_MAX);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, bulk_kernel<float>, NT, smem);
  } else {
    cudaFuncSetAttribute(bulk_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BULK_SMEM_MAX);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, bulk_kernel<double>, NT, smem);
  }
  return nb;
}

cudaError_t bulk_launch(int precision, const Desc& d, const KernelArgs& a, cudaStream_t s) {
  const Desc* dg = d.dev;
  KernelArgs aa = a;
  void* args[] = {&dg, &aa};
  const size_t smem = kernel_smem_bytes(d);
  const void* fn = precision ? (const void*)bulk_kernel<float> : (const void*)bulk_kernel<double>;
  return cudaLaunchCooperativeKernel(fn, dim3(d.grid), dim3(NT), args, smem, s);
}

}  // namespace mf
