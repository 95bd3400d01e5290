// The transform core: one line's FFT held in the registers of the threads that share the line.
//
// A transform of length L = 2^lg runs on L / E threads, thread i holding the E elements at
// positions i + j L/E (j < E), before and after, in natural order both times.  So a pass loads
// straight into registers (lanes read neighbouring positions), transforms, works pointwise,
// transforms back and stores, with no shared-memory staging at either end; between the radix-E
// stages the elements move through one padded shared buffer.
//
// An element is 16 bytes in both precisions: in FP64 one complex value; in FP32 two complex
// values of two lines that are transformed together, as (re, re), (im, im), so that every
// complex add and multiply is done for both lines by the packed two-way FP32 instructions
// (add/mul/fma.f32x2), which halve the issue slots of a transform, and every shared-memory
// access moves 16 bytes per lane.
//
// E (elements per thread, the radix) trades exchanges for parallelism (elems_per_thread in
// mf_tables.h has the rule and its measurements).
#pragma once
#include "mf_common.cuh"

namespace mf {

// ------------------------------------------------------------------------------------------
// arithmetic on an element's real (or imaginary) part: two FP32 lanes or one double
// ------------------------------------------------------------------------------------------
struct F2 { unsigned long long u; };
__device__ __forceinline__ F2 pk(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk(F2 a, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.u));
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b) { F2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u)); return r; }
__device__ __forceinline__ F2 vsub(F2 a, F2 b) { F2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u)); return r; }
__device__ __forceinline__ F2 vmul(F2 a, F2 b) { F2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u)); return r; }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
  return r;
}
__device__ __forceinline__ F2 vneg(F2 a) { return vmul(a, pk(-1.f, -1.f)); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vneg(double a) { return -a; }

// per precision: the element part type V, the real rows that one element holds in a row pass
// (two per complex line) and the lines that are transformed together
template <typename T> struct Lane;
template <> struct Lane<float> { using V = F2; static constexpr int RU = 4, NL = 2; };
template <> struct Lane<double> { using V = double; static constexpr int RU = 2, NL = 1; };
__device__ __forceinline__ F2 vconst(double s, F2*) { return pk((float)s, (float)s); }
__device__ __forceinline__ double vconst(double s, double*) { return s; }
__device__ __forceinline__ F2 vset(float s, F2*) { return pk(s, s); }
__device__ __forceinline__ double vset(double s, double*) { return s; }

template <class V> struct alignas(16) CV { V x, y; };
template <class V> __device__ __forceinline__ CV<V> eadd(const CV<V>& a, const CV<V>& b) { return {vadd(a.x, b.x), vadd(a.y, b.y)}; }
template <class V> __device__ __forceinline__ CV<V> esub(const CV<V>& a, const CV<V>& b) { return {vsub(a.x, b.x), vsub(a.y, b.y)}; }
// a + t, a - t for t = DIR i b
template <int DIR, class V> __device__ __forceinline__ CV<V> eadd_i(const CV<V>& a, const CV<V>& b) {
  return DIR > 0 ? CV<V>{vsub(a.x, b.y), vadd(a.y, b.x)} : CV<V>{vadd(a.x, b.y), vsub(a.y, b.x)};
}
template <class V> __device__ __forceinline__ CV<V> escale(const CV<V>& a, const V& s) { return {vmul(a.x, s), vmul(a.y, s)}; }
template <class V> __device__ __forceinline__ CV<V> ezero();
template <> __device__ __forceinline__ CV<F2> ezero<F2>() { return {F2{0ull}, F2{0ull}}; }
template <> __device__ __forceinline__ CV<double> ezero<double>() { return {0.0, 0.0}; }

// Shared-memory position of element e of a line: one spare slot per 8 keeps the
// 16-byte accesses of 8 consecutive lanes (one wavefront) on distinct banks for every stage's
// writes and reads.
__host__ __device__ __forceinline__ constexpr int spe(int e) { return e + (e >> 3); }
// ------------------------------------------------------------------------------------------
// butterflies
// ------------------------------------------------------------------------------------------
// A twiddle for direction DIR (the table holds exp(-i phi); DIR = +1 uses the conjugate), with the
// negated imaginary part beside it (the packed instructions take no negated operands).
template <class V> struct Tw { V x, y, ny; };
template <int DIR, class V> __device__ __forceinline__ Tw<V> mk_tw(const CV<V>& w) {
  const V n = vneg(w.y);
  return DIR > 0 ? Tw<V>{w.x, n, w.y} : Tw<V>{w.x, w.y, n};
}
__device__ __forceinline__ double sqrt_half(double*) { return 0.70710678118654752440; }
__device__ __forceinline__ F2 sqrt_half(F2*) { return pk(0.70710678118654752440f, 0.70710678118654752440f); }
// (a, b) <- (a + w b, a - w b)
__device__ __forceinline__ void bf_tw(CV<F2>& a, CV<F2>& b, const Tw<F2>& w) {
  const CV<F2> t = {vfma(w.x, b.x, vmul(w.ny, b.y)), vfma(w.x, b.y, vmul(w.y, b.x))};
  b = esub(a, t);
  a = eadd(a, t);
}
// FP64: 6 instructions (a - w b = 2 a - (a + w b)), the FP64 unit is what bounds those passes
__device__ __forceinline__ void bf_tw(CV<double>& a, CV<double>& b, const Tw<double>& w) {
  const CV<double> s = {fma(w.ny, b.y, fma(w.x, b.x, a.x)), fma(w.y, b.x, fma(w.x, b.y, a.y))};
  b = {fma(2.0, a.x, -s.x), fma(2.0, a.y, -s.y)};
  a = s;
}
// (a, b) <- (a + DIR i w b, a - DIR i w b)
template <int DIR>
__device__ __forceinline__ void bf_tw_i(CV<F2>& a, CV<F2>& b, const Tw<F2>& w) {
  const CV<F2> t = {vfma(w.x, b.x, vmul(w.ny, b.y)), vfma(w.x, b.y, vmul(w.y, b.x))};
  b = eadd_i<-DIR>(a, t);
  a = eadd_i<DIR>(a, t);
}
template <int DIR>
__device__ __forceinline__ void bf_tw_i(CV<double>& a, CV<double>& b, const Tw<double>& w) {
  bf_tw(a, b, DIR > 0 ? Tw<double>{w.ny, w.x, -w.x} : Tw<double>{w.y, -w.x, w.x});
}
template <class V> __device__ __forceinline__ void bf(CV<V>& a, CV<V>& b) {
  const CV<V> s = eadd(a, b);
  b = esub(a, b);
  a = s;
}
template <int DIR, class V> __device__ __forceinline__ void bf_i(CV<V>& a, CV<V>& b) {
  const CV<V> s = eadd_i<DIR>(a, b);
  b = eadd_i<-DIR>(a, b);
  a = s;
}
// (a, b) <- (a + u b, a - u b), u = exp(DIR i pi/4) or exp(DIR 3 i pi/4): u b = h ((+-bx - DIR by),
// (DIR bx +- by))
template <int DIR, class V> __device__ __forceinline__ void bf_oct(CV<V>& a, CV<V>& b) {
  const V h = sqrt_half((V*)nullptr), n = vneg(h);
  const V p = vadd(b.x, b.y), m = DIR > 0 ? vsub(b.x, b.y) : vsub(b.y, b.x);
  const CV<V> t = DIR > 0 ? CV<V>{m, p} : CV<V>{p, m};
  b = {vfma(n, t.x, a.x), vfma(n, t.y, a.y)};
  a = {vfma(h, t.x, a.x), vfma(h, t.y, a.y)};
}
template <int DIR, class V> __device__ __forceinline__ void bf_oct3(CV<V>& a, CV<V>& b) {
  const V h = sqrt_half((V*)nullptr), n = vneg(h);
  // DIR > 0: u b = h (-(bx + by), bx - by); DIR < 0: h (by - bx, -(bx + by))
  const V p = vadd(b.x, b.y), m = DIR > 0 ? vsub(b.x, b.y) : vsub(b.y, b.x);
  if (DIR > 0) {
    const CV<V> s = {vfma(n, p, a.x), vfma(h, m, a.y)};
    b = {vfma(h, p, a.x), vfma(n, m, a.y)};
    a = s;
  } else {
    const CV<V> s = {vfma(h, m, a.x), vfma(n, p, a.y)};
    b = {vfma(n, m, a.x), vfma(h, p, a.y)};
    a = s;
  }
}

__host__ __device__ constexpr int bitrev(int j, int r) {
  int o = 0;
  for (int k = 0; k < r; ++k) { o = (o << 1) | (j & 1); j >>= 1; }
  return o;
}

// The radix-2^r butterflies on a thread's E elements, in natural order in and out: E >> r
// independent sets, set s = elements s + (E >> r) m, by decimation in time in r radix-2 levels.
// w[m] is the stage's twiddle w to the power 2^m of set 0; set s has w zeta^s with zeta =
// exp(DIR 2 pi i / E), so every butterfly's factor is a power of w times a power of zeta.
// FIRST: w = 1 and r = log2 E.
template <int DIR, int E, int r, bool FIRST, class V>
__device__ __forceinline__ void dft_stage(CV<V>* x, const CV<V>* w) {
  constexpr int R = 1 << r, NS = E >> r;
  CV<V> y[E];                          // set s at y[s R ..], bit-reversed
#pragma unroll
  for (int s = 0; s < NS; ++s) {
#pragma unroll
    for (int m = 0; m < R; ++m) y[s * R + bitrev(m, r)] = x[s + NS * m];
  }
#pragma unroll
  for (int l = 1; l <= r; ++l) {
    // T zeta^c for the c' = c mod E/4 that occur (c >= E/4: a further factor DIR i)
    Tw<V> t[E >= 8 ? E / 4 : 1];
    if constexpr (!FIRST) {
      t[0] = mk_tw<DIR>(w[r - l]);
      if constexpr (E == 8) t[1] = mk_tw<DIR>(w[r]);
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
#pragma unroll
      for (int k = 0; k < R / 2; ++k) {
        const int h = 1 << (l - 1), b = k & (h - 1), g = k >> (l - 1);
        CV<V>& p = y[s * R + (g << l) + b];
        CV<V>& q = y[s * R + (g << l) + b + h];
        const int c = s * (1 << (r - l)) + b * (E >> l);
        constexpr int Q = E >= 4 ? E / 4 : 1;
        if (E == 2 || c < Q) {
          if (!FIRST) bf_tw(p, q, t[c % Q]);
          else if (c == 0) bf(p, q);
          else bf_oct<DIR>(p, q);
        } else {
          if (!FIRST) bf_tw_i<DIR>(p, q, t[c % Q]);
          else if (c == Q) bf_i<DIR>(p, q);
          else bf_oct3<DIR>(p, q);
        }
      }
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
#pragma unroll
    for (int m = 0; m < R; ++m) x[s + NS * m] = y[s * R + m];
  }
}

// ------------------------------------------------------------------------------------------
// the threads that share one line
// ------------------------------------------------------------------------------------------
__host__ __device__ constexpr int lg_of(int E) { return E == 2 ? 1 : E == 4 ? 2 : 3; }

// A group of G = 2^lgG lines (neighbours in memory) is interleaved on the lanes: thread i of line u is
// thread (i << lgG) + u of the group, so that a warp moves G neighbouring values per position.  A group
// of up to 32 threads lies inside a warp; longer ones (2, 4 or 8 warps) have a named barrier each, so
// that the groups of a CTA do not wait for one another.
template <typename T, int E> struct Team {
  using V = typename Lane<T>::V;
  static constexpr int LGE = lg_of(E);
  CV<V>* s;              // the line's part of the shared buffer
  const CV<V>* tw;       // twiddle table of this length and radix (shared memory)
  int i, u, slot;        // thread of the line; line of the group; line of the CTA
  int lg, lgt, fs;       // log2 of the length and of the group's threads; buffer elements per field
  __device__ __forceinline__ Team(CV<V>* buf, const CV<V>* table, int lgL, int lgG = 0) : tw(table), lg(lgL) {
    lgt = lg - LGE + lgG;
    u = (int)threadIdx.x & ((1 << lgG) - 1);
    i = ((int)threadIdx.x >> lgG) & ((1 << (lg - LGE)) - 1);
    slot = (((int)threadIdx.x >> lgt) << lgG) + u;
    const int stride = line_stride(lg, lgG);
    s = buf + slot * stride;
    fs = ((NT >> lgt) << lgG) * stride;
  }
  __device__ __forceinline__ int threads() const { return 1 << (lg - LGE); }
  __device__ __forceinline__ int step() const { return 1 << (lg - LGE); }    // position stride of a thread's elements
  __device__ __forceinline__ CV<V>& at(int e) const { return s[spe(e)]; }
  __device__ __forceinline__ void sync() const {
    if (lgt <= 5) __syncwarp();
    else asm volatile("bar.sync %0, %1;" :: "r"(1 + ((int)threadIdx.x >> lgt)), "r"(1 << lgt) : "memory");
  }
};

// Transforms of length 2^lg >= E of NF fields together (they share the exchanges' barriers; field f's
// buffer starts f t.fs elements behind the first one's), unnormalised.
template <int DIR, int NF, class V, int E, class TM>
__device__ __forceinline__ void core_fft_n(CV<V> (&v)[NF][E], const TM& t) {
  constexpr int e = lg_of(E), X = E == 8 ? e + 1 : e;
#pragma unroll
  for (int f = 0; f < NF; ++f) dft_stage<DIR, E, e, true>(v[f], (const CV<V>*)nullptr);
  const int q = 1 << (t.lg - e), i = t.i;
  const CV<V>* tw = t.tw;
  int rem = t.lg - e;
  for (int lgp = e; rem > 0; lgp += e, rem -= e) {
    // outputs of the stage before (radix E, p / E): element r at (i - k) E + k + r p / E
    const int p = 1 << lgp;
    t.sync();
    if (lgp == e && E >= 8) {
      CV<V>* const w = t.s + (i << e) + ((i << e) >> 3);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int r = 0; r < E; ++r) w[f * t.fs + r] = v[f][r];
      }
    } else if (lgp >= e + 3) {
      const int pp = p >> e, kp = i & (pp - 1);
      CV<V>* const w = &t.at(((i - kp) << e) + kp);
      const int ws = pp + (pp >> 3);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int r = 0; r < E; ++r) w[f * t.fs + r * ws] = v[f][r];
      }
    } else {
      const int pp = p >> e, kp = i & (pp - 1), w = ((i - kp) << e) + kp;
#pragma unroll
      for (int r = 0; r < E; ++r) {
        CV<V>* const o = &t.at(w + r * pp);
#pragma unroll
        for (int f = 0; f < NF; ++f) o[f * t.fs] = v[f][r];
      }
    }
    t.sync();
    if (q >= 8) {
      const CV<V>* const rd = &t.at(i);
      const int rds = q + (q >> 3);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int j = 0; j < E; ++j) v[f][j] = rd[f * t.fs + j * rds];
      }
    } else {
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const CV<V>* const o = &t.at(i + j * q);
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f][j] = o[f * t.fs];
      }
    }
    if (rem >= e) {
      CV<V> w[X];
      const int k = i & (p - 1);
#pragma unroll
      for (int m = 0; m < X; ++m) w[m] = tw[(m << lgp) + k];
      tw += X << lgp;
#pragma unroll
      for (int f = 0; f < NF; ++f) dft_stage<DIR, E, e, false>(v[f], w);
    } else if (e > 2 && rem == 2) {
      const CV<V> w[3] = {tw[i], tw[q + i], E == 8 ? tw[2 * q + i] : tw[i]};
#pragma unroll
      for (int f = 0; f < NF; ++f) dft_stage<DIR, E, (e > 2 ? 2 : 1), false>(v[f], w);
    } else if (e > 1) {
      const CV<V> w[2] = {tw[i], E == 8 ? tw[q + i] : tw[i]};
#pragma unroll
      for (int f = 0; f < NF; ++f) dft_stage<DIR, E, 1, false>(v[f], w);
    }
  }
}
template <int DIR, class V, int E, class TM>
__device__ __forceinline__ void core_fft(CV<V> (&v)[E], const TM& t) {
  core_fft_n<DIR, 1>(reinterpret_cast<CV<V>(&)[1][E]>(v), t);
}

}  // namespace mf
