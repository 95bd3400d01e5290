// Pieces shared by the film (2D) and bulk (3D) right-hand sides: the applied field h_e(t),
// the stage input of the integrator, per-CTA scalars and epilogue/result records.
#pragma once
#include <new>

#include "mf_common.cuh"

namespace mf {

constexpr double PI_D = 3.14159265358979323846;

__device__ __forceinline__ float powt(float a, float b) { return powf(a, b); }
__device__ __forceinline__ double powt(double a, double b) { return pow(a, b); }

// x^(m/2) for x > 0 and a whole m >= 1, by squaring from the highest bit of m / 2 down, with the rounding
// error of every product carried along (fma(a, b, -a b) is exact), times sqrt(x) for an odd m: within 0.5
// ulp for an even m, 1.5 for an odd one (0.500 and 1.42 found over x = 1e-3 .. 10, m to 128); CUDA
// documents 2 for pow.
__device__ __forceinline__ double pow_half(double x, int m) {
  double hi = 1.0, lo = 0.0;
  const int k = m >> 1;
  if (k > 0) {
    hi = x;
    for (int b = 30 - __clz(k); b >= 0; --b) {
      double p = hi * hi;
      lo = fma(hi + hi, lo, fma(hi, hi, -p));
      hi = p;
      if (k >> b & 1) {
        p = hi * x;
        lo = fma(lo, x, fma(hi, x, -p));
        hi = p;
      }
    }
  }
  if (m & 1) {
    const double s = sqrt(x);
    const double p = hi * s;
    lo = fma(lo, s, fma(hi, s, -p));
    hi = p;
  }
  const double r = hi + lo;
  return r == r ? r : hi;              // an overflow leaves hi infinite and lo a NaN
}

// power law of Eq. 3 / Eq. 13:  rho = (e0/jc) (|j|/jc)^(n-1) in the superconductor (mask 1),
// rho_out elsewhere.  Takes |j|^2.
// Double: an FP64 instruction takes an SM sub-partition 64 cycles, and pow is a long run of them.  For a
// whole n up to 129 pow_half's few products take its place, and at jc = 1 (the normalised units of most
// problems) the two divisions by 1 are left out: a film's right-hand side at 64^2 / 1024^2 with 4 / 5
// iterations 173 / 2042 us against 181 / 2073 us with pow.  Single precision keeps powf, which is short.
template <typename T>
__device__ __forceinline__ T resistivity(T j2, T jc, int m, T n, T e0, T rho_out) {
  if (m != 1) return rho_out;
  T x2 = j2, f = e0, pw;
  if (sizeof(T) == 4 || jc != (T)1) {
    x2 = j2 / (jc * jc);
    f = e0 / jc;
  }
  // (|j|/jc)^(n-1) = (|j|^2/jc^2)^((n-1)/2); exactly 1 for n = 1 (including j = 0)
  if (n == (T)1) pw = (T)1;
  else if (x2 <= (T)0) pw = (T)0;
  else if (sizeof(T) == 8 && n <= (T)129 && (T)(int)n == n) pw = pow_half(x2, (int)n - 1);
  else pw = powt(x2, (n - (T)1) * (T)0.5);
  return f * pw;
}

// stage input y + sum c_j k_j (FP64), optionally written to ynew
struct StageIn {
  const double* y;
  int nk;
  double c[3];
  const double* k[3];
  double* ynew;
};

// Scalars of the integrator's current step attempt.  Thread 0 computes them and the others read
// them: an FP64 instruction occupies an SM sub-partition for 64 cycles, so the same scalar
// arithmetic done by every warp of an SM would take tens of thousands of cycles per step.
struct Control {
  double t, h, h_prop, t_lim, t_new;
  double ts[4];                  // stage times
  double c[4][3];                // stage coefficients of the derivatives
  int go, clipped, seg, outcome, status;
};

// per-CTA copy of the scalars every CTA agrees on
struct Shared {
  double red[NT / 32], red2[NT / 32];
  double redn[3][NT / 32];       // (3D) per-item sums
  double hed3[3], thresh;        // (3D) h_e_dot; residual threshold of the stop test
  float hed3f[3];
  double A, C, r, hed, N;
  float Af, Cf, rq;              // (2D) A, C and h_e_dot in the transform precision's FP32 form
  int stop, ok, diverged;        // decisions of the outside iteration
  int warm_valid;
  double A_prev;
  int com_valid, hd_sel;         // (2D) accepted-step initial approximation, see SolverState
  double A_com;
  double q11;                    // (2D) sum over free space of q1 (from the solver state)
  double inv_nout;               // 1 / free-space cells
  int attempt_first;             // (2D) the next right-hand side is the first of a step attempt
  unsigned long long bar_passed;  // grid barriers passed in this launch (thread 0)
  Control ctl;
};

// ------------------------------------------------------------------------------------------
// applied field
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int he_segment(const Desc& d, double t) {
  if (d.he_knots <= 0) return 0;
  int k = -1;
  for (int i = 0; i < d.he_knots; ++i)
    if (d.he_t[i] <= t) k = i;
  return k;
}
__device__ __forceinline__ double he_value(const Desc& d, double t) {
  if (d.he_knots <= 0) return d.he_sin_amp * sin(2.0 * PI_D * t / d.he_sin_period);
  const int k = he_segment(d, t);
  if (k < 0) return d.he_v[0];
  if (k >= d.he_knots - 1) return d.he_v[d.he_knots - 1];
  const double s = (t - d.he_t[k]) / (d.he_t[k + 1] - d.he_t[k]);
  return d.he_v[k] + s * (d.he_v[k + 1] - d.he_v[k]);
}
__device__ __forceinline__ double he_dot(const Desc& d, double t, int seg) {
  if (d.he_knots <= 0) {
    const double w = 2.0 * PI_D / d.he_sin_period;
    return d.he_sin_amp * w * cos(w * t);
  }
  const int k = (seg == -2) ? he_segment(d, t) : seg;
  if (k < 0 || k >= d.he_knots - 1) return 0.0;
  return (d.he_v[k + 1] - d.he_v[k]) / (d.he_t[k + 1] - d.he_t[k]);
}
__device__ __forceinline__ double he_next_knot(const Desc& d, double t) {
  for (int i = 0; i < d.he_knots; ++i)
    if (d.he_t[i] > t) return d.he_t[i];
  return INFINITY;
}

// Acc is the type of the per-thread partial sums: the transform precision T in the epilogues of
// the outside iteration (FP64 arithmetic runs at a small fraction of the FP32 rate on this part),
// double where a sum feeds the integrator's error norm or a readout.  The partials of a CTA
// are combined in double.
template <typename T, typename Acc = double>
struct EpiBase {
  Acc acc = 0, accmax = 0;
  Acc acc2 = 0;                 // a second sum (rows() with a second slot)
  bool is_max = false;
};

struct RhsOut {
  int status, iters;
  double r;
  double err;          // BS23 error norm when requested
  int nonfinite;
};


// ------------------------------------------------------------------------------------------
// BS23 integrator loop shared by the film and bulk kernels: adaptive steps until t_target or
// max_attempts, first same as last, every decision taken identically by every CTA (by its
// thread 0, from the same sums).
// R(t, seg, stage_in, k_out, force_iters, want_err, h, k1, k2, k3, y, ynew) evaluates one
// right-hand side.  Returns the launch status.
// ------------------------------------------------------------------------------------------
template <class Rhs>
__device__ int bs23_advance(Rhs& R, const Desc& d, SolverState* st, const KernelArgs& a, bool leader,
                            Control& ctl) {
  const bool t0 = threadIdx.x == 0;
  if (t0) { ctl.t = st->t; ctl.h = st->h; ctl.status = ST_OK; }
  int failed = st->failed, k1_valid = st->k1_valid;
  int iy = st->ybuf, iyn = st->ynewbuf, ik1 = st->k1buf, ik4 = st->k4buf;
  // k2, k3 live in the two remaining buffers
  int others[2], no = 0;
  for (int b = 0; b < 6 && no < 2; ++b)
    if (b != iy && b != iyn && b != ik1 && b != ik4) others[no++] = b;
  const int ik2 = others[0], ik3 = others[1];
  long long att = 0, n_rhs = 0, n_it = 0, n_acc = 0, n_rej = 0, n_nc = 0;
  double last_r = 0.0, last_err = 0.0;             // thread 0
  int status = ST_OK;
  for (;;) {
    __syncthreads();
    if (t0) {
      ctl.go = ctl.t < a.t_target && att < a.max_attempts;
      if (ctl.go) {
        ctl.t_lim = fmin(a.t_target, he_next_knot(d, ctl.t));
        ctl.h_prop = ctl.h;            // the controller's proposal before clipping
        ctl.clipped = ctl.t + 1.1 * ctl.h >= ctl.t_lim;
        if (ctl.clipped) ctl.h = ctl.t_lim - ctl.t;
        ctl.seg = he_segment(d, ctl.t);
        const double t = ctl.t, h = ctl.h;
        ctl.t_new = ctl.clipped ? ctl.t_lim : t + h;
        ctl.ts[0] = t; ctl.ts[1] = t + 0.5 * h; ctl.ts[2] = t + 0.75 * h; ctl.ts[3] = ctl.t_new;
        ctl.c[1][0] = 0.5 * h; ctl.c[2][0] = 0.75 * h;
        ctl.c[3][0] = h * (2.0 / 9.0); ctl.c[3][1] = h * (1.0 / 3.0); ctl.c[3][2] = h * (4.0 / 9.0);
      }
    }
    __syncthreads();
    if (!ctl.go) break;
    R.on_attempt();                    // the attempt's first evaluation starts from the accepted step
    const int seg = ctl.seg;
    const double h = ctl.h;
    int it[4] = {-1, -1, -1, -1};
    double* y = d.fbuf[iy];
    double* yn = d.fbuf[iyn];
    double* k1 = d.fbuf[ik1];
    double* k2 = d.fbuf[ik2];
    double* k3 = d.fbuf[ik3];
    double* k4 = d.fbuf[ik4];
    RhsOut r;
    r.status = ST_OK;
    r.r = 0.0;
    if (!k1_valid) {
      // a k1 whose outside iteration did not converge rejects the attempt like any other
      // stage; the warm start keeps the progress, so the next attempt continues from it
      StageIn in{y, 0, {0, 0, 0}, {nullptr, nullptr, nullptr}, nullptr};
      r = R(ctl.ts[0], seg, in, k1, 0, false, 0, nullptr, nullptr, nullptr, nullptr, nullptr);
      ++n_rhs; n_it += r.iters; it[0] = r.iters;
      if (r.status == ST_BARRIER) { status = ST_BARRIER; break; }
      if (r.status == ST_OK && r.nonfinite) { status = ST_NONFINITE; break; }
      if (r.status == ST_OK) k1_valid = 1;
    }
    if (r.status == ST_OK) {
      StageIn s2{y, 1, {ctl.c[1][0], 0, 0}, {k1, nullptr, nullptr}, nullptr};
      r = R(ctl.ts[1], seg, s2, k2, 0, false, 0, nullptr, nullptr, nullptr, nullptr, nullptr);
      ++n_rhs; n_it += r.iters; it[1] = r.iters;
      if (r.status == ST_BARRIER) { status = ST_BARRIER; break; }
    }
    if (r.status == ST_OK) {
      StageIn s3{y, 1, {ctl.c[2][0], 0, 0}, {k2, nullptr, nullptr}, nullptr};
      r = R(ctl.ts[2], seg, s3, k3, 0, false, 0, nullptr, nullptr, nullptr, nullptr, nullptr);
      ++n_rhs; n_it += r.iters; it[2] = r.iters;
      if (r.status == ST_BARRIER) { status = ST_BARRIER; break; }
    }
    if (r.status == ST_OK) {
      StageIn s4{y, 3, {ctl.c[3][0], ctl.c[3][1], ctl.c[3][2]}, {k1, k2, k3}, yn};
      r = R(ctl.ts[3], seg, s4, k4, 0, true, h, k1, k2, k3, y, yn);
      ++n_rhs; n_it += r.iters; it[3] = r.iters;
      if (r.status == ST_BARRIER) { status = ST_BARRIER; break; }
    }
    const bool reached = r.status == ST_OK;
    if (t0) {
      const double err = reached ? r.err : (double)INFINITY;
      ctl.outcome = !reached ? 2 : (err <= 1.0 ? 1 : 0);
      last_r = r.r;
      const bool clipped = ctl.clipped != 0;
      if (leader) {
        if (st->log_count < d.log_cap) {
          StepLog L; L.t = ctl.t; L.h = h; L.t_new = ctl.outcome == 1 ? ctl.t_new : ctl.t; L.err = err;
          L.outcome = ctl.outcome; for (int q = 0; q < 4; ++q) L.iters[q] = it[q]; L.pad = 0;
          d.log[st->log_count] = L;
        }
        st->log_count += 1;
      }
      if (ctl.outcome == 1) {
        const bool knot_hit = clipped && ctl.t_lim == he_next_knot(d, ctl.t);
        ctl.t = ctl.t_new;
        ctl.go = knot_hit ? 0 : 1;     // k4 serves as the next k1
        double fac = err == 0.0 ? 5.0 : fmin(5.0, fmax(0.2, 0.9 * pow(err, -1.0 / 3.0)));
        if (failed) fac = fmin(fac, 1.0);
        // a step shortened to end on a knot or output time says nothing about longer steps:
        // the next one starts from the proposal it replaced (never above it)
        ctl.h = (clipped && h < ctl.h_prop) ? ctl.h_prop * fmin(fac, 1.0) : h * fac;
        last_err = err;
      } else if (ctl.outcome == 0) {
        ctl.h = h * fmax(0.2, 0.9 * pow(err, -1.0 / 3.0));
      } else {
        ctl.h = 0.5 * h;
      }
      if (ctl.h < d.h_min) ctl.status = ST_UNDERFLOW;
    }
    __syncthreads();
    ++att;
    const int outcome = ctl.outcome;
    if (outcome == 1) {
      R.on_accept();                   // the last evaluation's iterate starts later calls
      int tmp = iy; iy = iyn; iyn = tmp;
      tmp = ik1; ik1 = ik4; ik4 = tmp;
      k1_valid = ctl.go;
      failed = 0;
      ++n_acc;
    } else {
      if (outcome == 2) ++n_nc;
      failed = 1;
      ++n_rej;
    }
    status = ctl.status;
    if (status != ST_OK) break;
  }
  if (leader) {
    st->t = ctl.t; st->h = ctl.h; st->failed = failed; st->k1_valid = k1_valid;
    st->ybuf = iy; st->ynewbuf = iyn; st->k1buf = ik1; st->k4buf = ik4;
    st->n_attempts += att; st->n_rhs += n_rhs; st->n_iters += n_it; st->n_accepted += n_acc;
    st->n_rejected += n_rej; st->n_noconv += n_nc; st->last_r = last_r; st->last_err = last_err;
  }
  return status;
}

}  // namespace mf
