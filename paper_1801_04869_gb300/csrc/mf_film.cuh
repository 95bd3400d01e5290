// Thin-film (2D) right-hand side and BS23 integrator: the device code of the persistent kernels.
//
// Method: Section 2 of Prigozhin & Sokolovsky (arXiv:1801.04869).  One right-hand side
// f(t, g) runs, as phases separated by grid barriers:
//   P1  x pass of the stage input g_s = y + h sum a_j k_j           -> Sa
//   P2  y pass: smoothed gradient  i k_{x,y} G                         (Section 2.2)
//   P3  x pass: j = (g_y, -g_x) (Eq. 2), e = rho(|j|) j (Eq. 3), forward x pass of e -> Sb
//   P4  y pass: -curl e = -i G (k_x e_y - k_y e_x)                     (Eq. 4 / Eq. 9)
//   P5  x pass: h_dot_in on the conductor, warm h_dot on free space, sum for A (Eq. 10)
//   loop (Eqs. 11-12):
//   P6  y pass: 2/|k|
//   P7  x pass: g_dot = raw - A q1 - C, residual sum over free space of |g_dot| (the stop
//       test of Section 2.3), forward of mask_out g_dot
//   P9  y pass: lambda (|k|/2) G (only when the stop test did not end the loop)
//   P10 x pass: h_dot_out <- h_dot_out - A - w, sums for the next A and C, forward
//   end: g_dot on the conductor, 0 on free space (FP64)
// The shift A (Eq. 10) is applied lazily through q1 = F^-1[K1 F(out)] (exact by linearity).
// The centring constant C (Eq. 11), the mean over free space of raw - A q1, is known before
// the x pass that forms g_dot: K1 is real and even, so sum_out F^-1[K1 F h] = <q1, h>, and
// C = (<q1, h> - A sum_out q1) / n_out with <q1, h> summed where h is written (P5, P10).
//
// Both passes run on the transform core (mf_core.cuh).  The real fields of the workspace (h_dot,
// g_dot, q1, q2, the jc map) and the mask are kept by row units: the RU rows that one element of a
// row pass holds (4 in FP32, 2 in FP64) lie together for each x, 16 bytes, and their mask classes
// in one byte, so that an epilogue moves one 16-byte vector per element.
//
// What bounds a pass, and what it measured (one right-hand side, 5 outside iterations = 24 passes with
// their grid barriers; the design before transformed through two shared buffers at 16 values per
// thread): small grids are bound by one thread's chain of instructions, the barrier and the load
// latencies (128^2: FP32 250 -> 166 us, FP64 514 -> 227 us); FP64 grids from 512^2 by the FP64 unit,
// 2 lanes per cycle and SM, and the last round of units, 513 columns on 152 SMs (1024^2 2.85 -> 2.04 ms,
// 2048^2 11.2 -> 8.5 ms); 2048^2 FP32 by the latency of exchanges and loads at 16 warps per SM (979 -> 760
// us), 512^2 and 1024^2 by both (350 -> 195 us, 513 -> 290 us).  What did not pay at 2048^2: spectra
// staged asynchronously as in the bulk passes (823 us: most CTAs have one unit or two), a second exchange
// buffer in place of every other barrier (755 us, but 64^2 FP64 176 -> 182 us), k_y and its Gaussian in
// shared memory (767 us).
#pragma once
#include "mf_units.cuh"

namespace mf {

enum Op2 { OP_GRAD = 0, OP_CURLNEG = 1, OP_K1 = 2, OP_K2 = 3, OP_KH = 4, OP_ID = 5 };

// raw pointers and sizes the x-pass epilogues need, held by value (registers)
template <typename T>
struct FilmPtrs {
  const uint8_t* mask;
  const T* jcmap;
  T* hd;
  T* u;
  const T* q1;
  const T* q2;
  int nx;
};

template <typename T>
struct Film {
  using V = typename Lane<T>::V;
  static constexpr int RU = Lane<T>::RU, NL = Lane<T>::NL;
  const Desc& d;
  CV<V>* sm;         // the CTA's exchange buffer
  Shared& sh;
  int nx, ny, lgx, lgy, half, nkx;
  int nspec, ncell;
  C2<T>* Sa;
  C2<T>* Sb;
  T* hd;
  T* u;
  const T* q1;
  const T* q2;
  const uint8_t* mask;
  const T* jcmap;
  const CV<V>* twx;  // twiddle tables, behind the exchange buffer in shared memory
  const CV<V>* twy;
  const T* ktab;     // kx values (half entries), then ky values (ny entries)
  const T* gtab;     // Gaussian factors, same layout
  T lam, scale, ig2;  // lambda; 1/(2 cells); 1/gamma^2
  int ex, ey;        // elements per thread of the x and y passes
  int max_items;     // members of the descriptor that every phase reads, at hand in shared memory (a
  double* partials;  // grid barrier's acquire empties L1)
  GridBarrier* gb;
  unsigned long long barrier_ns;
  double iter_tol;
  int vb;            // this CTA's index among the CTAs that run this film
  unsigned nblocks;  // how many CTAs run this film

  __device__ Film(const Desc& dd, unsigned char* smem, Shared& shr, int vblock, unsigned nblk)
      : d(dd), sm((CV<V>*)smem), sh(shr) {
    nx = d.nx; ny = d.ny; lgx = d.lgx; lgy = d.lgy; half = nx / 2; nkx = half + 1;
    nspec = nkx * ny;
    ncell = nx * ny;
    Sa = (C2<T>*)d.Sa; Sb = (C2<T>*)d.Sb;
    hd = (T*)d.hd; u = (T*)d.u; q1 = (const T*)d.q1; q2 = (const T*)d.q2;
    mask = d.mask; jcmap = (const T*)d.jcmap;
    ex = d.ex; ey = d.ey;
    const int slots = film_slots(d);
    twx = sm + slots;
    twy = one_table(d) ? twx : twx + core_table_len(lgx, ex);
    max_items = d.max_items;
    partials = d.partials;
    gb = d.gb;
    barrier_ns = d.barrier_ns;
    iter_tol = d.iter_tol;
    ktab = (const T*)d.ktab;
    gtab = (const T*)d.gtab;
    lam = (T)d.lam;
    scale = (T)0.5 / (T)ncell;         // a power of two
    ig2 = (T)(1.0 / (d.gamma * d.gamma));
    vb = vblock;
    nblocks = nblk;
    sh.N = (double)ncell;
    sh.inv_nout = d.nout > 0 ? 1.0 / (double)d.nout : 0.0;
  }

  __device__ bool sync(int where) { return grid_sync(gb, nblocks, where, &sh.bar_passed, barrier_ns); }

  __device__ FilmPtrs<T> ptrs() const { return FilmPtrs<T>{mask, jcmap, hd, u, q1, q2, nx}; }

  // ---- y pass: forward, multiplier, inverse on the lines of NL consecutive x-wavenumbers ----
  struct Coef { V kxo, kx2, gx; };     // per line: k_x (0 at its Nyquist index), k_x^2, G_x
  __device__ __forceinline__ Coef coef_x(int kx) const {
    if constexpr (sizeof(T) == 4) {
      const int k1 = kx + 1 < nkx ? kx + 1 : kx;
      const float a = ldg_tab(&ktab[kx]), b = ldg_tab(&ktab[k1]);
      return {pk(kx == half ? 0.f : a, k1 == half ? 0.f : b), pk(a * a, b * b),
              pk(ldg_tab(&gtab[kx]), ldg_tab(&gtab[k1]))};
    } else {
      const double a = ldg_tab(&ktab[kx]);
      return {kx == half ? 0.0 : a, a * a, ldg_tab(&gtab[kx])};
    }
  }
  // k_y (m in FFT order) and its Gaussian factor
  __device__ __forceinline__ void coef_y(int ky, T& k, T& g) const {
    k = ldg_tab(&ktab[nkx + ky]);
    g = ldg_tab(&gtab[nkx + ky]);
  }
  // multiplier of a one-field operator at |k|^2 = k2.  |k| and 1/|k| come from one reciprocal
  // square root (1 ulp in double; a few ulp in single, far below the transform's error)
  __device__ __forceinline__ static T inv_abs(T k2) {
    if constexpr (sizeof(T) == 4) return k2 > 0.f ? rsqrtf(k2) : 0.f;
    else return k2 > 0.0 ? rsqrt(k2) : 0.0;
  }
  // c1 / |k| (OP_K1: c1 = 2) or c2 |k| g (OP_K2: c2 = lambda/2, g the Gaussian; OP_KH: 1/2 and 1)
  __device__ __forceinline__ static V mult_k1(const V& kx2, T ky, T c1) {
    if constexpr (sizeof(T) == 4) {
      float a, b;
      upk(vfma(pk(ky, ky), pk(ky, ky), kx2), a, b);
      return vmul(pk(inv_abs(a), inv_abs(b)), pk(c1, c1));
    } else {
      return inv_abs(fma(ky, ky, kx2)) * c1;
    }
  }
  __device__ __forceinline__ static V mult_k(const V& kx2, T ky, const V& g) {
    if constexpr (sizeof(T) == 4) {
      float a, b;
      const F2 k2 = vfma(pk(ky, ky), pk(ky, ky), kx2);
      upk(k2, a, b);
      return vmul(vmul(k2, pk(inv_abs(a), inv_abs(b))), g);
    } else {
      const double k2 = fma(ky, ky, kx2);
      return k2 * inv_abs(k2) * g;
    }
  }

  template <int E, int NIN, int NOUT>
  __device__ __noinline__ void cols_e(const C2<T>* Sin, C2<T>* Sout, int op) {
    const int ny = this->ny;
    const int nspec = this->nspec;
    Team<T, E> t(sm, twy, lgy);
    const int units = (nkx + NL - 1) / NL;
    const int per = NT / t.threads();
    // lines that a CTA runs at a time: as few as spread the pass over all CTAs
    const int want = (units + (int)nblocks - 1) / (int)nblocks;
    const int nuc = want < per ? want : per;
    const int q = t.step();
    for (int u0 = vb * nuc; u0 < units; u0 += (int)nblocks * nuc) {
      const int first = ((int)threadIdx.x & ~31) >> (lgy - Team<T, E>::LGE);   // slot of the warp's first lane
      if (first >= nuc || u0 + first >= units) continue;
      const bool mine = t.slot < nuc && u0 + t.slot < units;
      const int kx = mine ? (u0 + t.slot) * NL : 0;
      const bool two = NL == 2 && kx + 1 < nkx;
      const C2<T>* const src = Sin + kx * ny + t.i;
      C2<T>* const dst = Sout + kx * ny + t.i;
      const Coef c = coef_x(kx);
      CV<V> v[E];
#pragma unroll
      for (int j = 0; j < E; ++j) v[j] = ld_col(src + j * q, ny, two);
      core_fft<-1>(v, t);
      if constexpr (NIN == 1 && NOUT == 1) {
        if (op == OP_K1) {
          const T c1 = (T)2 * scale;
#pragma unroll
          for (int j = 0; j < E; ++j)
            v[j] = escale(v[j], mult_k1(c.kx2, ldg_tab(&ktab[nkx + t.i + j * q]), c1));
        } else if (op == OP_ID) {
#pragma unroll
          for (int j = 0; j < E; ++j) v[j] = escale(v[j], vset(scale, (V*)nullptr));
        } else {
          const bool smooth = op == OP_K2;
          const T c2 = (smooth ? lam : (T)1) * (T)0.5 * scale;
          const V gx = smooth ? vmul(c.gx, vset(c2, (V*)nullptr)) : vset(c2, (V*)nullptr);
#pragma unroll
          for (int j = 0; j < E; ++j) {
            T ky, gy;
            coef_y(t.i + j * q, ky, gy);
            v[j] = escale(v[j], mult_k(c.kx2, ky, smooth ? vmul(gx, vset(gy, (V*)nullptr)) : gx));
          }
        }
      } else if constexpr (NOUT == 2) {
        // smoothed gradient i k G (odd factors are 0 at the Nyquist index of their axis); the
        // transformed line waits in the second output's place (the same thread's positions)
#pragma unroll
        for (int j = 0; j < E; ++j) {
          T ky, gy;
          coef_y(t.i + j * q, ky, gy);
          const V g = vmul(vmul(c.gx, vset(gy * scale, (V*)nullptr)), c.kxo);
          if (mine) st_col(dst + nspec + j * q, ny, two, v[j]);
          v[j] = CV<V>{vneg(vmul(v[j].y, g)), vmul(v[j].x, g)};
        }
        core_fft<+1>(v, t);
#pragma unroll
        for (int j = 0; j < E; ++j) {
          if (mine) st_col(dst + j * q, ny, two, v[j]);
          v[j] = ld_col(dst + nspec + j * q, ny, two);
        }
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int ky = t.i + j * q;
          T k, gy;
          coef_y(ky, k, gy);
          if (ky == (ny >> 1)) k = (T)0;
          const V g = vmul(c.gx, vset(gy * scale * k, (V*)nullptr));
          v[j] = CV<V>{vneg(vmul(v[j].y, g)), vmul(v[j].x, g)};
        }
      } else {
        // -(i kx G e_y - i ky G e_x) = i G (ky e_x - kx e_y); the first field's part waits in the
        // output's place
#pragma unroll
        for (int j = 0; j < E; ++j) {
          if (mine) st_col(dst + j * q, ny, two, v[j]);
          v[j] = ld_col(src + nspec + j * q, ny, two);
        }
        core_fft<-1>(v, t);
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int ky = t.i + j * q;
          T k, gy;
          coef_y(ky, k, gy);
          if (ky == (ny >> 1)) k = (T)0;
          const CV<V> a = ld_col(dst + j * q, ny, two);
          const V kv = vset(k, (V*)nullptr), kn = vneg(c.kxo);
          const V g = vmul(c.gx, vset(gy * scale, (V*)nullptr));
          const CV<V> b = {vfma(kv, a.x, vmul(kn, v[j].x)), vfma(kv, a.y, vmul(kn, v[j].y))};
          v[j] = CV<V>{vneg(vmul(b.y, g)), vmul(b.x, g)};
        }
      }
      core_fft<+1>(v, t);
      C2<T>* const out = NOUT == 2 ? dst + nspec : dst;
      if (mine) {
#pragma unroll
        for (int j = 0; j < E; ++j) st_col(out + j * q, ny, two, v[j]);
      }
    }
  }
  template <int NIN, int NOUT>
  __device__ __forceinline__ void cols_n(const C2<T>* Sin, C2<T>* Sout, int op) {
    if (ey == 2) cols_e<2, NIN, NOUT>(Sin, Sout, op);
    else if (ey == 4) cols_e<4, NIN, NOUT>(Sin, Sout, op);
    else cols_e<8, NIN, NOUT>(Sin, Sout, op);
  }
  __device__ __forceinline__ void cols(const C2<T>* Sin, int nin, C2<T>* Sout, int nout, int op) {
    if (nin == 2) cols_n<2, 1>(Sin, Sout, op);
    else if (nout == 2) cols_n<1, 2>(Sin, Sout, op);
    else cols_n<1, 1>(Sin, Sout, op);
  }

  // ---- x pass over units of RU rows: inverse of NIN fields, epilogue, forward of NOUT ----
  // Row pass over the units of RU rows with optional per-unit sums into partials slots `slot` (acc,
  // or the maximum of accmax) and `slot2` (acc2).  epi(i, r, in, out) is called for every element: i
  // is the index of the unit's 16-byte vector (and mask byte), r the row-major index of its first
  // row's cell.  With two inputs or two outputs one of the fields waits in `tmp` (a real field by row
  // units) while the other one is transformed, so that a thread never holds two fields' elements.
  // The sums are per unit whatever the number of CTAs, so a film gives the same bits on any launch.
  template <int E, int NIN, int NOUT, class Epi>
  __device__ __noinline__ void rows_e(const C2<T>* Sin, C2<T>* Sout, const Epi& epi_in, int slot, int slot2, T* tmp) {
    Epi epi = epi_in;                   // register copy of the epilogue
    const int nx = this->nx, ny = this->ny;
    const int nspec = this->nspec;
    Team<T, E> t(sm, twx, lgx);
    const int q = t.step(), tt = t.threads();
    const int units = ny / RU;
    const int want = (units + (int)nblocks - 1) / (int)nblocks, per = NT / tt;
    const int nuc = want < per ? want : per;       // units that a CTA runs at a time
    const int first = ((int)threadIdx.x & ~31) >> (lgx - Team<T, E>::LGE);   // slot of the warp's first lane
    for (int u0 = vb * nuc; u0 < units; u0 += (int)nblocks * nuc) {
      if (first >= nuc || u0 + first >= units) continue;
      const bool mine = t.slot < nuc && u0 + t.slot < units;
      const int unit = mine ? u0 + t.slot : u0;
      const int y0 = unit * RU;
      const int iu = unit * nx + t.i;
      const int ir = y0 * nx + t.i;
      epi.acc = 0;
      epi.accmax = 0;
      epi.acc2 = 0;
      CV<V> v[E];
      // the epilogue's fields, B elements at a time: the first batch is on its way during the
      // inverse transform, each further one while the batch before is worked on
      constexpr int B = Epi::kBatch < E ? Epi::kBatch : E;
      typename Epi::Ld ld[2][B];
      if constexpr (NIN > 0) row_gather(v, t, Sin + y0, nx, ny);
      if constexpr (NIN == 2) {
        core_fft<+1>(v, t);
        if (mine) {
#pragma unroll
          for (int j = 0; j < E; ++j) st_q(tmp + (iu + j * q) * RU, to_q(v[j]));
        }
        row_gather(v, t, Sin + nspec + y0, nx, ny);
      }
#pragma unroll
      for (int b = 0; b < B; ++b) ld[0][b] = epi.load(iu + b * q, ir + b * q);
      if constexpr (NIN > 0) core_fft<+1>(v, t);
#pragma unroll
      for (int j0 = 0; j0 < E; j0 += B) {
        if (j0 + B < E) {
#pragma unroll
          for (int b = 0; b < B; ++b) ld[(j0 / B + 1) & 1][b] = epi.load(iu + (j0 + B + b) * q, ir + (j0 + B + b) * q);
        }
        Q<T> in0[B];
        if constexpr (NIN == 2) {
#pragma unroll
          for (int b = 0; b < B; ++b) in0[b] = ld_q(tmp + (iu + (j0 + b) * q) * RU);
        }
        if (mine) {
#pragma unroll
          for (int b = 0; b < B; ++b) {
            const int j = j0 + b;
            Q<T> in[NIN > 0 ? NIN : 1], out[NOUT > 0 ? NOUT : 1];
            const int i = iu + j * q;
            if constexpr (NIN == 2) { in[0] = in0[b]; in[1] = to_q(v[j]); }
            if constexpr (NIN == 1) in[0] = to_q(v[j]);
            epi.apply(ld[(j0 / B) & 1][b], i, ir + j * q, in, out);
            if constexpr (NOUT > 0) v[j] = to_e(out[0]);
            if constexpr (NOUT == 2) st_q(tmp + i * RU, out[1]);
          }
        }
      }
      if constexpr (NOUT > 0) {
        core_fft<-1>(v, t);
        row_scatter(v, t, Sout + y0, nx, ny, mine);
      }
      if constexpr (NOUT == 2) {
#pragma unroll
        for (int j = 0; j < E; ++j) v[j] = to_e(ld_q(tmp + (iu + j * q) * RU));
        core_fft<-1>(v, t);
        row_scatter(v, t, Sout + nspec + y0, nx, ny, mine);
      }
      if (slot >= 0) unit_sums(epi, t, unit, mine, slot, slot2);
    }
  }
  // a unit's sums: over the lanes of its team, then (teams of several warps) over the team's warps in
  // FP64 by one thread per sum (threads of two sub-partitions: an FP64 addition takes 64 cycles)
  template <int E, class Epi>
  __device__ __forceinline__ void unit_sums(const Epi& epi, const Team<T, E>& t, int unit, bool mine, int slot, int slot2) {
    const int tt = t.threads(), w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int width = tt < 32 ? tt : 32;
    auto a = epi.is_max ? epi.accmax : epi.acc;
    auto b = epi.acc2;
    for (int o = width >> 1; o > 0; o >>= 1) {
      const auto x = __shfl_xor_sync(0xffffffffu, a, o);
      a = epi.is_max ? (x > a ? x : a) : a + x;
      if (slot2 >= 0) b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    double* const pa = partials + (size_t)slot * max_items + unit;
    double* const pb = partials + (size_t)slot2 * max_items + unit;
    if (tt <= 32) {
      if (t.i == 0 && mine) {
        *pa = (double)a;
        if (slot2 >= 0) *pb = (double)b;
      }
      return;
    }
    t.sync();                           // the unit before has been summed
    if (l == 0) {
      sh.red[w] = (double)a;
      if (slot2 >= 0) sh.red2[w] = (double)b;
    }
    t.sync();
    // by lanes 0 .. warps - 1 of the team's first warp (acc) and second warp (acc2)
    const int nw = tt / 32;
    if ((t.i >> 5) == 0) {
      double s = sh.red[w + (l & (nw - 1))];
      for (int o = nw >> 1; o > 0; o >>= 1) {
        const double x = __shfl_xor_sync(0xffffffffu, s, o);
        s = epi.is_max ? (x > s ? x : s) : s + x;
      }
      if (l == 0) *pa = s;
    } else if ((t.i >> 5) == 1 && slot2 >= 0) {
      double s = sh.red2[w - 1 + (l & (nw - 1))];
      for (int o = nw >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (l == 0) *pb = s;
    }
  }
  template <int NIN, int NOUT, class Epi>
  __device__ __forceinline__ void rows(const C2<T>* Sin, C2<T>* Sout, const Epi& epi, int slot, int slot2 = -1, T* tmp = nullptr) {
    if (ex == 2) rows_e<2, NIN, NOUT>(Sin, Sout, epi, slot, slot2, tmp);
    else if (ex == 4) rows_e<4, NIN, NOUT>(Sin, Sout, epi, slot, slot2, tmp);
    else rows_e<8, NIN, NOUT>(Sin, Sout, epi, slot, slot2, tmp);
  }
  // Sums over the units of slots a and (b >= 0) b, in a fixed order: the last warps first, which have
  // no line to run while the pass before is narrow, so that the sums of a small film are formed
  // beside its column pass.  The result is valid in thread SUMS, which the caller lets go on.
  static constexpr int SUMS = NT - 32;
  __device__ double2 partial_sums(int a, int b) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int n = ny / RU;
    const bool few = n <= 128;             // two warps per slot, else four
    const int per = few ? 2 : 4;
    const int sl = few ? (w < 4 ? -1 : w < 6 ? a : b) : (w < 4 ? b : a);
    if (sl >= 0) {
      const double* p = partials + (size_t)sl * max_items;
      double v = 0.0;
      for (int i = (w & (per - 1)) * 32 + l; i < n; i += per * 32) v += __ldcg(p + i);
      v = warp_sum(v);
      if (l == 0) sh.red[w] = v;
    }
    __syncthreads();
    double2 r = make_double2(0.0, 0.0);
    if (threadIdx.x == SUMS) {
      const double* q = sh.red;
      if (few) {
        r.x = q[4] + q[5];
        if (b >= 0) r.y = q[6] + q[7];
      } else {
        r.x = (q[4] + q[5]) + (q[6] + q[7]);
        if (b >= 0) r.y = (q[0] + q[1]) + (q[2] + q[3]);
      }
    }
    return r;
  }
  // sum (max) over the units of a slot, the same in every thread of every CTA
  __device__ double total(int slot, bool is_max = false) {
    return reduce_partials(partials, max_items, slot, ny / RU, is_max, sh.red);
  }
  // Eq. 10 and Eq. 11 constants from the sums of h (slot 0) and q1 h (slot 5) of the pass that
  // wrote h: A = (sum h - N h_e_dot) / n_out, C = (<q1, h> - A sum_out q1) / n_out
  __device__ void shifts() {
    const double2 t = partial_sums(0, 5);
    if (threadIdx.x == SUMS) {
      const double A = (t.x - sh.N * sh.hed) * sh.inv_nout;
      const double C = (t.y - A * sh.q11) * sh.inv_nout;
      sh.A = A;
      sh.C = C;
      sh.Af = (float)A;
      sh.Cf = (float)C;
    }
    __syncthreads();
  }
  // the sum of a slot / n_out (sh.A), in the transform precision
  __device__ T mean_of(int slot) {
    const double2 t = partial_sums(slot, -1);
    if (threadIdx.x == SUMS) {
      sh.A = t.x * sh.inv_nout;
      sh.Af = (float)sh.A;
    }
    __syncthreads();
    return At();
  }
  // the outside iteration's scalars in the transform precision
  __device__ __forceinline__ T At() const { if constexpr (sizeof(T) == 4) return sh.Af; else return sh.A; }
  __device__ __forceinline__ T Ct() const { if constexpr (sizeof(T) == 4) return sh.Cf; else return sh.C; }
  // Section 2.3: r = mean over free space of |g_dot| (slot 2) and the decision to stop
  __device__ void stop_test(bool by_count, bool last) {
    const double2 t = partial_sums(2, -1);
    if (threadIdx.x == SUMS) {
      const double r = t.x * sh.inv_nout;
      sh.r = r;
      sh.stop = by_count ? last : (r < iter_tol || last);
    }
    __syncthreads();
  }
};

// ------------------------------------------------------------------------------------------
// epilogues
// ------------------------------------------------------------------------------------------
// Epilogues of the x pass: load(i, r) reads the fields of the RU rows of one element, with the index
// i of their 16-byte vector and the row-major index r of the first row's cell (the others nx
// apart); apply(ld, i, r, in, out) works on them with the inverse-transformed inputs
// in[f].v[0 .. RU) and sets the outputs out[f].v[0 .. RU).  kBatch elements are loaded together
// (a store could alias a later load as far as the compiler knows, so a load placed behind a store
// waits for the whole latency of the loads before it).

// P1 / readouts: field from the FP64 stage input
template <typename T>
struct EpiStage : EpiBase<T> {
  static constexpr int RU = Lane<T>::RU;
  FilmPtrs<T> P;
  StageIn in;
  static constexpr int kBatch = 2;
  struct Ld { double v[RU]; };
  __device__ __forceinline__ Ld load(int, int r) const {
    Ld l;
#pragma unroll
    for (int q = 0; q < RU; ++q) l.v[q] = ld_s(in.y + r + q * P.nx);
    for (int j = 0; j < in.nk; ++j) {
      double k[RU];
#pragma unroll
      for (int q = 0; q < RU; ++q) k[q] = ld_s(in.k[j] + r + q * P.nx);
#pragma unroll
      for (int q = 0; q < RU; ++q) l.v[q] += in.c[j] * k[q];
    }
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int, int r, const Q<T>*, Q<T>* out) {
    if (in.ynew) {
#pragma unroll
      for (int q = 0; q < RU; ++q) in.ynew[r + q * P.nx] = l.v[q];
    }
#pragma unroll
    for (int q = 0; q < RU; ++q) out[0].v[q] = (T)l.v[q];
  }
};

// mask indicator of free space (set-up of q1, q2)
template <typename T>
struct EpiOut : EpiBase<T> {
  FilmPtrs<T> P;
  static constexpr int kBatch = 4;
  struct Ld { int m; };
  __device__ __forceinline__ Ld load(int i, int) const { return Ld{ld_mask(P.mask + i)}; }
  __device__ __forceinline__ void apply(const Ld& l, int, long long, const Q<T>*, Q<T>* out) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) out[0].v[q] = cls(l.m, q) == 0 ? (T)1 : (T)0;
  }
};

// store a real field (set-up); sum of it over free space
template <typename T>
struct EpiStoreT : EpiBase<T> {
  FilmPtrs<T> P;
  T* dst;
  static constexpr int kBatch = 4;
  struct Ld { int m; };
  __device__ __forceinline__ Ld load(int i, int) const { return Ld{ld_mask(P.mask + i)}; }
  __device__ __forceinline__ void apply(const Ld& l, int i, int, const Q<T>* in, Q<T>*) {
    st_q(dst + i * Lane<T>::RU, in[0]);
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q)
      if (cls(l.m, q) == 0) this->acc += (double)in[0].v[q];
  }
};
// h_z readout (FP64)
template <typename T>
struct EpiStoreHz : EpiBase<T> {
  FilmPtrs<T> P;
  double* dst;
  double he;
  static constexpr int kBatch = 4;
  using Ld = NoLd;
  __device__ __forceinline__ Ld load(int, int) const { return Ld{}; }
  __device__ __forceinline__ void apply(const Ld&, int, int r, const Q<T>* in, Q<T>*) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) dst[r + q * P.nx] = he + (double)in[0].v[q];
  }
};

// P3: power law.  ig2 = 1/gamma^2 of the elliptic law e = rho(j_eff) (j_x, j_y/gamma^2),
// j_eff^2 = j_x^2 + j_y^2/gamma^2 in the superconductor (Eq. 3 at gamma = 1, where the extra
// products by 1 are exact)
template <typename T>
struct EpiPower : EpiBase<T> {
  FilmPtrs<T> P;
  T n, e0, jc, rho_out, ig2;
  static constexpr int kBatch = 4;
  struct Ld { int m; Q<T> jc; };
  __device__ __forceinline__ Ld load(int i, int) const {
    Ld l;
    l.m = ld_mask(P.mask + i);
    if (P.jcmap) {
      l.jc = ldg_q(P.jcmap + i * Lane<T>::RU);
    } else {
#pragma unroll
      for (int q = 0; q < Lane<T>::RU; ++q) l.jc.v[q] = jc;
    }
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int, long long, const Q<T>* in, Q<T>* out) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) {
      const T gx = in[0].v[q], gy = in[1].v[q];
      const T jx = gy, jy = -gx;                              // Eq. 2
      const int mq = cls(l.m, q);
      const T a = mq == 1 ? ig2 : (T)1;
      const T rho = resistivity<T>(jx * jx + jy * jy * a, l.jc.v[q], mq, n, e0, rho_out);
      out[0].v[q] = rho * jx;                                 // Eq. 3
      out[1].v[q] = rho * jy * a;
    }
  }
};

// P5: initial h_dot (warm start), sum over D
template <typename T>
struct EpiInit : EpiBase<T, T> {
  FilmPtrs<T> P;
  bool warm;
  const T* wsrc;          // warm start (the previous time step's or the most recent iterate)
  T A_prev, hed;
  static constexpr int kBatch = 4;
  struct Ld { int m; Q<T> w, q1; };
  __device__ __forceinline__ Ld load(int i, int) const {
    Ld l;
    l.m = ld_mask(P.mask + i);
    if (warm) l.w = ld_q(wsrc + i * Lane<T>::RU);
    l.q1 = ldg_q(P.q1 + i * Lane<T>::RU);
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int i, int, const Q<T>* in, Q<T>* out) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) {
      T h;
      if (cls(l.m, q) != 0) h = in[0].v[q];                   // h_dot_in on the conductor
      else h = warm ? l.w.v[q] - A_prev : hed;                // warm start (Section 2.2)
      this->acc += h;
      this->acc2 += l.q1.v[q] * h;                              // <q1, h> for C
      out[0].v[q] = h;
    }
    st_q(P.hd + i * Lane<T>::RU, out[0]);
  }
};

// P7: g_dot = raw - A q1 - C (Eq. 11), stored where the unit touches the conductor (all that the
// final pass reads); residual sum over free space of |g_dot| (Section 2.3); forward of
// mask_out g_dot (the input of Eq. 12)
template <typename T>
struct EpiU : EpiBase<T, T> {
  FilmPtrs<T> P;
  T A, C;
  static constexpr int kBatch = 4;
  struct Ld { int m; Q<T> q1; };
  __device__ __forceinline__ Ld load(int i, int) const {
    return Ld{ld_mask(P.mask + i), ldg_q(P.q1 + i * Lane<T>::RU)};
  }
  __device__ __forceinline__ void apply(const Ld& l, int i, int, const Q<T>* in, Q<T>* out) {
    Q<T> v;
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) {
      v.v[q] = (in[0].v[q] - A * l.q1.v[q]) - C;
      const bool o = cls(l.m, q) == 0;
      if (o) this->acc += fabs(v.v[q]);
      out[0].v[q] = o ? v.v[q] : (T)0;
    }
    if (l.m != 0) st_q(P.u + i * Lane<T>::RU, v);
  }
};

// P10: h_dot update on free space (Eq. 12: w is the transform of mask_out g_dot), sums over D
// of h (for A) and of q1 h (for C), forward
template <typename T>
struct EpiUpdate : EpiBase<T, T> {
  FilmPtrs<T> P;
  T A;
  static constexpr int kBatch = 4;
  struct Ld { int m; Q<T> h, q1; };
  __device__ __forceinline__ Ld load(int i, int) const {
    return Ld{ld_mask(P.mask + i), ld_q(P.hd + i * Lane<T>::RU), ldg_q(P.q1 + i * Lane<T>::RU)};
  }
  __device__ __forceinline__ void apply(const Ld& l, int i, int, const Q<T>* in, Q<T>* out) {
    Q<T> h = l.h;
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) {
      if (cls(l.m, q) == 0) h.v[q] = (h.v[q] - A) - in[0].v[q];
      this->acc += h.v[q];
      this->acc2 += l.q1.v[q] * h.v[q];
    }
    st_q(P.hd + i * Lane<T>::RU, h);
    out[0] = h;
  }
};

// finalize: g_dot (stored by P7) on the conductor; optional BS23 error contribution
template <typename T, bool err>
struct EpiFinal : EpiBase<T, T> {
  FilmPtrs<T> P;
  double* kout;
  // err: error estimate (stage 4 of a step): E = h (e1 k1 + e2 k2 + e3 k3 + e4 k4)
  double h, rtol, atol;
  const double* k1; const double* k2; const double* k3; const double* y; const double* ynew;
  static constexpr int RU = Lane<T>::RU, NE = err ? RU : 1, kBatch = err ? 1 : 4;
  struct Ld { int m; Q<T> u; double a1[NE], a2[NE], a3[NE], y[NE], yn[NE]; };
  __device__ __forceinline__ Ld load(int i, int r) const {
    Ld l;
    l.m = ld_mask(P.mask + i);
    l.u = ld_q(P.u + i * RU);                              // defined on the conductor's units only
    if constexpr (err) {
#pragma unroll
      for (int q = 0; q < RU; ++q) {
        const int c = r + q * P.nx;
        l.a1[q] = ld_s(k1 + c); l.a2[q] = ld_s(k2 + c); l.a3[q] = ld_s(k3 + c);
        l.y[q] = ld_s(y + c); l.yn[q] = ld_s(ynew + c);
      }
    }
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int, int r, const Q<T>*, Q<T>*) {
#pragma unroll
    for (int q = 0; q < RU; ++q) {
      const bool in = cls(l.m, q) != 0;
      const double g = in ? (double)l.u.v[q] : 0.0;
      kout[r + q * P.nx] = g;
      if constexpr (err) {
        const double E = h * (-5.0 / 72.0 * l.a1[q] + 1.0 / 12.0 * l.a2[q] + 1.0 / 9.0 * l.a3[q] - 0.125 * g);
        const double sc = atol + rtol * fmax(fabs(l.y[q]), fabs(l.yn[q]));
        // E and its scale in FP64; their ratio, which only feeds the accept test and the step
        // size factor, in the transform precision (FP64 division runs at a small fraction of the
        // FP32 rate on this part)
        T e;
        if constexpr (sizeof(T) == 4) e = __fdiv_rn((float)fabs(E), (float)sc);
        else e = fabs(E) / sc;
        if (!(e == e)) e = (T)INFINITY;                      // non-finite -> rejected step
        this->accmax = this->accmax > e ? this->accmax : e;
      } else if (in && !isfinite(l.u.v[q])) {
        this->accmax = (T)1;
      }
    }
  }
};

// e readout (FP64, 2 fields): e = rho(|j|) j with j = (g_y, -g_x) (Eq. 2, Eq. 3), Ohm law
// rho_out j on free space and filled holes
template <typename T>
struct EpiStoreE : EpiBase<T> {
  FilmPtrs<T> P;
  T n, e0, jc, rho_out, ig2;
  double* dst;
  int ncell;
  static constexpr int kBatch = 4;
  using Ld = typename EpiPower<T>::Ld;
  __device__ __forceinline__ EpiPower<T> law() const {       // the law of P3
    EpiPower<T> p;
    p.P = P; p.n = n; p.e0 = e0; p.jc = jc; p.rho_out = rho_out; p.ig2 = ig2;
    return p;
  }
  __device__ __forceinline__ Ld load(int i, int r) const { return law().load(i, r); }
  __device__ __forceinline__ void apply(const Ld& l, int i, int r, const Q<T>* in, Q<T>*) {
    Q<T> e[2];
    law().apply(l, i, r, in, e);
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) {
      dst[r + q * P.nx] = (double)e[0].v[q];
      dst[ncell + r + q * P.nx] = (double)e[1].v[q];
    }
  }
};

// magnetization: sum over D of g (times dx dy on the host side)
template <typename T>
struct EpiMoment : EpiBase<T> {
  FilmPtrs<T> P;
  const double* g;
  static constexpr int kBatch = 4;
  struct Ld { double v[Lane<T>::RU]; };
  __device__ __forceinline__ Ld load(int, int r) const {
    Ld l;
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) l.v[q] = ld_s(g + r + q * P.nx);
    return l;
  }
  __device__ __forceinline__ void apply(const Ld& l, int, long long, const Q<T>*, Q<T>*) {
#pragma unroll
    for (int q = 0; q < Lane<T>::RU; ++q) this->acc += l.v[q];
  }
};

// ------------------------------------------------------------------------------------------
// one right-hand side.  Returns ST_OK / ST_NOCONV / ST_BARRIER (same in every CTA).
// ------------------------------------------------------------------------------------------
template <typename T>
__device__ __noinline__ RhsOut film_rhs(Film<T>& F, double t, int seg, const StageIn& sin, double* kout,
                           int force_iters, bool want_err, double h_err, const double* e_k1,
                           const double* e_k2, const double* e_k3, const double* e_y,
                           const double* e_ynew) {
  const Desc& d = F.d;
  RhsOut res{ST_OK, 0, 0.0, 0.0, 0};
  const bool first = F.sh.attempt_first != 0;   // read by every thread before it is cleared
  // h_dot buffers: this call writes hdw; hdc holds the committed (accepted-step) h_dot
  T* const hdw = (T*)(F.sh.hd_sel ? d.hd2 : d.hd);
  const T* const hdc = (const T*)(F.sh.hd_sel ? d.hd : d.hd2);
  if (threadIdx.x == 0) {               // scalar FP64 work: one thread (see Control)
    const double hed = he_dot(d, t, seg);
    const double Ap = first && F.sh.com_valid != 0 ? F.sh.A_com : F.sh.A_prev;
    F.sh.hed = hed;
    F.sh.rq = (float)hed;
    F.sh.A = Ap;
    F.sh.Af = (float)Ap;
  }

  // P1
  {
    EpiStage<T> e; e.P = F.ptrs(); e.in = sin;
    F.rows<0, 1>(nullptr, F.Sa, e, -1);
  }
  if (!F.sync(1)) { res.status = ST_BARRIER; return res; }
  F.cols(F.Sa, 1, F.Sa, 2, OP_GRAD);                                    // P2
  if (!F.sync(2)) { res.status = ST_BARRIER; return res; }
  {
    EpiPower<T> e; e.P = F.ptrs();
    e.n = (T)d.n; e.e0 = (T)d.e0; e.jc = (T)d.jc; e.rho_out = (T)d.rho_out;
    e.ig2 = F.ig2;
    F.rows<2, 2>(F.Sa, F.Sb, e, -1, -1, F.u);                           // P3
  }
  if (!F.sync(3)) { res.status = ST_BARRIER; return res; }
  F.cols(F.Sb, 2, F.Sb, 1, OP_CURLNEG);                                 // P4
  if (!F.sync(4)) { res.status = ST_BARRIER; return res; }

  const bool have_out = d.nout > 0;
  {
    // initial approximation "from the previous time step" (Section 2.2): the first evaluation
    // of a step attempt starts from the accepted step's h_dot, later stages (and calls outside
    // the integrator) from the most recent call's iterate; the very first call from h_e_dot
    EpiInit<T> e; e.P = F.ptrs(); e.P.hd = hdw;
    const bool com = first && F.sh.com_valid != 0;
    e.warm = com || F.sh.warm_valid != 0;
    e.wsrc = com ? hdc : hdw;
    e.A_prev = F.At();                   // the warm start's shift (set above)
    if constexpr (sizeof(T) == 4) e.hed = F.sh.rq;
    else e.hed = F.sh.hed;
    F.rows<1, 1>(F.Sb, F.Sa, e, 0, 5);                                  // P5
  }
  if (!F.sync(5)) { res.status = ST_BARRIER; return res; }
  if (!have_out) {
    if (threadIdx.x == 0) { F.sh.A = 0.0; F.sh.C = 0.0; F.sh.Af = 0.f; F.sh.Cf = 0.f; F.sh.r = 0.0; }
    __syncthreads();
  }
  const bool forced = force_iters > 0;
  const bool by_count = forced || d.iter_tol <= 0.0;
  int itmax = forced ? force_iters : d.iter_max;
  if (!have_out) itmax = 1;
  int i = 0;
  for (; i < itmax; ++i) {
    F.cols(F.Sa, 1, F.Sa, 1, OP_K1);                                    // P6
    // Eq. 10: A; Eq. 11: C = (<q1, h> - A sum_out q1) / n_out (K1 is real and even).  P6 does not
    // need them, so the sums of P5 / P10 are combined beside it.
    if (have_out) F.shifts();
    if (!F.sync(6)) { res.status = ST_BARRIER; return res; }
    {
      EpiU<T> e; e.P = F.ptrs(); e.A = F.At(); e.C = F.Ct();
      F.rows<1, 1>(F.Sa, F.Sb, e, 2);                                   // P7
    }
    if (!F.sync(7)) { res.status = ST_BARRIER; return res; }
    if (!have_out) break;
    if (!by_count || i == itmax - 1) {
      F.stop_test(by_count, i == itmax - 1);                            // Section 2.3
      if (F.sh.stop) break;
    }
    F.cols(F.Sb, 1, F.Sb, 1, OP_K2);                                    // P9 (Eq. 12)
    if (!F.sync(8)) { res.status = ST_BARRIER; return res; }
    {
      EpiUpdate<T> e; e.P = F.ptrs(); e.P.hd = hdw; e.A = F.At();
      F.rows<1, 1>(F.Sb, F.Sa, e, 0, 5);                                // P10
    }
    if (!F.sync(10)) { res.status = ST_BARRIER; return res; }
  }
  res.iters = i + 1;
  if (threadIdx.x == 0) {
    const double r = F.sh.r;
    F.sh.ok = !have_out || d.iter_tol <= 0.0 || r < d.iter_tol;
    // warm start for the next call: h_dot stored, A still to subtract on free space.  A call that
    // failed with a residual above 1e3 tol (or not finite) diverged: the next call starts cold.
    F.sh.warm_valid = !F.sh.ok && !(r < 1e3 * d.iter_tol) ? 0 : 1;
    F.sh.A_prev = F.sh.A;
    F.sh.attempt_first = 0;
  }

  // finalize
  {
    auto fill = [&](auto& e) {
      e.P = F.ptrs(); e.kout = kout; e.is_max = true;
      e.h = h_err; e.rtol = d.rtol; e.atol = d.atol;
      e.k1 = e_k1; e.k2 = e_k2; e.k3 = e_k3; e.y = e_y; e.ynew = e_ynew;
    };
    if (want_err) { EpiFinal<T, true> e; fill(e); F.rows<0, 0>(nullptr, nullptr, e, 3); }
    else { EpiFinal<T, false> e; fill(e); F.rows<0, 0>(nullptr, nullptr, e, 3); }
  }
  if (!F.sync(11)) { res.status = ST_BARRIER; return res; }
  res.status = F.sh.ok ? ST_OK : ST_NOCONV;
  res.r = F.sh.r;
  const double q = F.total(3, true);
  if (want_err) res.err = isinf(q) ? 1e300 : q;
  else res.nonfinite = __double_as_longlong(q) > 0;
  return res;
}

// adapter used by the shared BS23 integrator loop
template <typename T>
struct FilmRhs {
  Film<T>& F;
  __device__ RhsOut operator()(double t, int seg, const StageIn& in, double* kout, int force,
                               bool want_err, double h, const double* k1, const double* k2,
                               const double* k3, const double* y, const double* yn) {
    return film_rhs<T>(F, t, seg, in, kout, force, want_err, h, k1, k2, k3, y, yn);
  }
  // the integrator accepted a step: the last call's h_dot (written to hd_sel) becomes the
  // committed initial approximation, and later calls write the other buffer
  __device__ void on_attempt() {
    if (threadIdx.x == 0) F.sh.attempt_first = 1;
    __syncthreads();
  }
  __device__ void on_accept() {
    __syncthreads();
    const int sel = F.sh.hd_sel;
    const double A = F.sh.A_prev;
    __syncthreads();
    if (threadIdx.x == 0) { F.sh.com_valid = 1; F.sh.A_com = A; F.sh.hd_sel = sel ^ 1; }
    __syncthreads();
  }
};

// ------------------------------------------------------------------------------------------
// the persistent kernel
// ------------------------------------------------------------------------------------------
// The twiddle tables into shared memory, behind the exchange buffer (a grid barrier's acquire empties
// L1, so tables in global memory would come from L2 again in every phase).
template <typename T>
__device__ __forceinline__ void film_tables(const Desc& d) {
  uint4* const to = (uint4*)mf_dsmem + film_slots(d);
  const uint4* const x = (const uint4*)d.tw_x;
  const uint4* const y = (const uint4*)d.tw_y;
  const int nx = core_table_len(d.lgx, d.ex), ny = one_table(d) ? 0 : core_table_len(d.lgy, d.ey);
  for (int k = threadIdx.x; k < nx; k += NT) to[k] = x[k];
  for (int k = threadIdx.x; k < ny; k += NT) to[nx + k] = y[k];
}
// The body of a launch for one film, run by CTAs vb = 0 .. vn - 1 of that film.
template <typename T>
__device__ __forceinline__ void film_main(const Desc& d, const KernelArgs& a, int vb, unsigned vn) {
  __shared__ Shared sh;
  // one copy of the pass object per CTA, in shared memory: its members are read as broadcasts
  // instead of per-thread local-memory copies
  __shared__ __align__(16) unsigned char objraw[sizeof(Film<T>)];
  SolverState* st = d.st;
  if (threadIdx.x == 0) {
    sh.warm_valid = st->warm_valid;
    sh.bar_passed = 0;
    sh.A_prev = st->A_prev;
    sh.com_valid = st->com_valid;
    sh.hd_sel = st->hd_sel;
    sh.A_com = st->A_com;
    sh.attempt_first = 0;
    sh.q11 = st->q11;
  }
  if (threadIdx.x == 0) new (objraw) Film<T>(d, mf_dsmem, sh, vb, vn);
  film_tables<T>(d);
  __syncthreads();
  Film<T>& F = *reinterpret_cast<Film<T>*>(objraw);
  const bool leader = vb == 0 && threadIdx.x == 0;
  int status = ST_OK;

  if (a.mode == MODE_SETUP) {
    // q1 = F^-1[K1 F(out)], q2 = F^-1[K2 F(out)]
    for (int pass = 0; pass < 2; ++pass) {
      EpiOut<T> eo; eo.P = F.ptrs();
      F.rows<0, 1>(nullptr, F.Sa, eo, -1);
      if (!F.sync(20)) { status = ST_BARRIER; break; }
      F.cols(F.Sa, 1, F.Sa, 1, pass == 0 ? OP_K1 : OP_K2);
      if (!F.sync(21)) { status = ST_BARRIER; break; }
      EpiStoreT<T> es; es.P = F.ptrs(); es.dst = (T*)(pass == 0 ? d.q1 : d.q2);
      F.rows<1, 0>(F.Sa, nullptr, es, 4);
      if (!F.sync(22)) { status = ST_BARRIER; break; }
      if (pass == 0) {
        const double q11 = F.total(4);          // sum over free space of q1
        if (leader) st->q11 = q11;
      }
    }
  } else if (a.mode == MODE_HZ) {
    EpiStage<T> e; e.P = F.ptrs(); e.in = StageIn{a.y_in, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
    if (threadIdx.x == 0) sh.hed = he_value(d, a.t);
    F.rows<0, 1>(nullptr, F.Sa, e, -1);
    if (F.sync(30)) {
      F.cols(F.Sa, 1, F.Sa, 1, OP_KH);
      if (F.sync(31)) {
        EpiStoreHz<T> es; es.P = F.ptrs(); es.dst = a.out; es.he = sh.hed;
        F.rows<1, 0>(F.Sa, nullptr, es, -1);
      } else status = ST_BARRIER;
    } else status = ST_BARRIER;
  } else if (a.mode == MODE_E) {
    EpiStage<T> e; e.P = F.ptrs(); e.in = StageIn{a.y_in, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
    F.rows<0, 1>(nullptr, F.Sa, e, -1);
    if (F.sync(50)) {
      F.cols(F.Sa, 1, F.Sa, 2, OP_GRAD);
      if (F.sync(51)) {
        EpiStoreE<T> es; es.P = F.ptrs(); es.dst = a.out; es.ncell = F.ncell;
        es.n = (T)d.n; es.e0 = (T)d.e0; es.jc = (T)d.jc; es.rho_out = (T)d.rho_out;
        es.ig2 = F.ig2;
        F.rows<2, 0>(F.Sa, nullptr, es, -1, -1, F.u);
      } else status = ST_BARRIER;
    } else status = ST_BARRIER;
  } else if (a.mode == MODE_MOMENT) {
    EpiMoment<T> e; e.P = F.ptrs(); e.g = a.y_in;
    F.rows<0, 0>(nullptr, nullptr, e, 4);
    if (F.sync(40)) {
      const double s = F.total(4);
      if (leader) a.out[0] = s * d.dx * d.dy;
    } else status = ST_BARRIER;
  } else if (a.mode == MODE_RHS) {
    StageIn in{a.y_in, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
    RhsOut r = film_rhs<T>(F, a.t, a.seg, in, a.out, a.force_iters, false, 0.0, nullptr, nullptr,
                           nullptr, nullptr, nullptr);
    status = r.status == ST_OK && r.nonfinite ? ST_NONFINITE : r.status;
    if (leader) { st->last_iters = r.iters; st->last_r = r.r; st->n_rhs += 1; st->n_iters += r.iters; }
  } else if (a.mode == MODE_ADVANCE) {
    FilmRhs<T> R{F};
    status = bs23_advance(R, d, st, a, leader, sh.ctl);
  }
  if (leader) {
    st->warm_valid = sh.warm_valid;
    st->A_prev = sh.A_prev;
    st->com_valid = sh.com_valid;
    st->hd_sel = sh.hd_sel;
    st->A_com = sh.A_com;
    st->status = status;
    publish_state(d, st);
  }
}

// CTAs per SM of the film kernels: 2 leave 128 registers per thread.  4 (64 registers) spill in every
// pass, 3 spill too and leave the 513 line pairs of a 2048^2 pass 456 places.  One right-hand side with 5
// iterations, 2 / 3 / 4 per SM: 2048^2 FP32 759 / 1120 / 935 us, 1024^2 FP32 289 / 312 / 333 us, 1024^2 FP64
// 2080 / 2997 us.  A shared launch of 24 / 8 films of up to 128^2 cells with 3 per SM: FP32 5.1 / 2.7 ms
// against 5.5 / 2.3 ms, FP64 24.4 / 10.6 ms against 23.9 / 8.7 ms.
constexpr int FILM_CTAS = 2;

}  // namespace mf
