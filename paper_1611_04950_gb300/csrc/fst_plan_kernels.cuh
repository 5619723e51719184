// fst_plan_kernels.cuh -- FP64 plan-time kernel bodies: the Slepian basis vectors
// of the eigen-window around K (precomputation paragraph of Section 1.3).
//
// The DPSS are the eigenvectors of Slepian's tridiagonal matrix T_{N,W}
// (diag ((N-1)/2 - n)^2 cos(2 pi W), off-diagonal n (N - n) / 2), which commutes
// with the prolate matrix B_{N,W}; its l-th largest eigenvector is s^(l).  T is
// centro-symmetric, so its eigenvectors are symmetric (even l) or antisymmetric
// (odd l) and each parity is the eigenproblem of a tridiagonal matrix of half the
// size ("reduced" matrices, built on the host):
//   N = 2m:    both parities: leading m x m block, last diagonal d[m-1] +- e[m].
//   N = 2m+1:  symmetric: leading (m+1) x (m+1) block with the coupling between
//              m-1 and m multiplied by sqrt(2) (the centre sample is sqrt(2) u_m);
//              antisymmetric: leading m x m block (the centre sample is 0).
// Bodies here: multisection bisection on Sturm counts, the eigenvector by the forward
// three-term recurrence with a first-order correction of the eigenvalue, and the expansion
// of a reduced vector to the unit-norm, sign-fixed full vector.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>
#include "fst_fft.cuh"

namespace fst {

constexpr int BISECT_MS_MAX_TARGETS = 512;   // batches up to this many targets use multisection
constexpr int BISECT_WARPS_MAX = 16;         // warps (32 points each) per target and round
constexpr int PLAN_B = 8;                    // steps of a serial recurrence whose inputs are loaded ahead

// biased exponent field of a double (0 for zeros and subnormals)
FST_HD int dexp_field(double v) {
#ifdef __CUDA_ARCH__
  return (int)((__double_as_longlong(v) >> 52) & 0x7ff);
#else
  uint64_t u;
  memcpy(&u, &v, 8);
  return (int)((u >> 52) & 0x7ff);
#endif
}

// 2^k as a double, -1022 <= k <= 1023
FST_HD double dpow2(int k) {
  const uint64_t u = (uint64_t)(k + 1023) << 52;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double v;
  memcpy(&v, &u, 8);
  return v;
#endif
}

// The FP64 unit of this part, measured: an FP64 instruction holds its warp for 64 clocks whatever
// its active lanes and dependences, up to four warps per SM (one per sub-core) run side by side at
// 76, and more only queue.  So the serial recurrences below count FP64 instructions: signs, zeros
// and exponents are tested on the integer pipe, and rare FP64 work sits behind a branch that a
// warp takes as one (any lane needs it), which the compiler cannot turn into selects.
FST_HD int dneg(double v) {
#ifdef __CUDA_ARCH__
  return (int)((unsigned)__double2hiint(v) >> 31);
#else
  return v < 0.0;
#endif
}
FST_HD bool warp_any(bool v) {
#ifdef __CUDA_ARCH__
  return __any_sync(__activemask(), v);
#else
  return v;
#endif
}
FST_HD bool dzero(double v) {
#ifdef __CUDA_ARCH__
  return ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
#else
  return v == 0.0;
#endif
}

// PLAN_B consecutive entries (the concatenated matrices begin on multiples of PLAN_B entries and
// are followed by 2 PLAN_B spare ones, so blocks are aligned and may be loaded past the end)
FST_HD void load_block(const double *a, double *v) {
#pragma unroll
  for (int k = 0; k < PLAN_B; k += 2) {
#ifdef __CUDA_ARCH__
    const double2 q = __ldg(reinterpret_cast<const double2 *>(a + k));
    v[k] = q.x;
    v[k + 1] = q.y;
#else
    v[k] = a[k];
    v[k + 1] = a[k + 1];
#endif
  }
}

// Number of eigenvalues of the reduced matrix smaller than x: the sign changes of the Sturm
// sequence of leading principal minors p_i = det(T_i - x I), p_i = (d_i - x) p_{i-1} -
// e_i^2 p_{i-2} (p_{-1} = 1, e_0 = 0), which equal the negative pivots q_i = p_i / p_{i-1} of
// T - x I = L D L^T.  The recurrence needs no division (the serial chain is one FMA per step);
// every PLAN_B steps the pair (p_i, p_{i-1}) is brought back to exponent 0 by an exact power of
// two when it has left 2^(+-128) (a step grows it by at most about 2^87 for N <= 2^23, so a block
// stays below 2^824), and an exact zero p_i is replaced by -pivmin p_{i-1} (the pivot -pivmin of the LDL^T form).
// Bound: the FP64 unit.  A step is 3 FP64 instructions (product, difference, FMA); zeros are
// looked for once per block, whose steps are then taken again one by one; the inputs of the next
// block are loaded while the current one is processed.  Measured at N = 65536 (32768 steps, four
// warps per SM): a test and branch in every step 6.1 ms a round, one per block 4.6 ms.
FST_HD int sturm_count(const double *d, const double *e2, int n, double x, double pivmin) {
  constexpr int B = PLAN_B;
  double pm = 0.0, p = 1.0;
  int neg = 0, c = 0;
  double E[B], D[B], En[B], Dn[B];
  // steps [k0, k1) of the block held in D, E, with the zero test in each
  auto slow = [&](int k1) {
    for (int k = 0; k < k1; ++k) {
      double pn = fma(D[k] - x, p, -(E[k] * pm));
      if (dzero(pn)) pn = -pivmin * p;
      const int ng = dneg(pn);
      c += ng ^ neg;
      neg = ng;
      pm = p;
      p = pn;
    }
  };
  load_block(e2, E);
  load_block(d, D);
  int i0 = 0;
  for (; i0 + B <= n; i0 += B) {
    load_block(e2 + i0 + B, En);
    load_block(d + i0 + B, Dn);
    const double p0 = p, pm0 = pm;
    const int neg0 = neg, c0 = c;
    bool zero = false;
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const double pn = fma(D[k] - x, p, -(E[k] * pm));
      zero = zero || dzero(pn);
      const int ng = dneg(pn);
      c += ng ^ neg;
      neg = ng;
      pm = p;
      p = pn;
    }
    const int ex = dexp_field(p), exm = dexp_field(pm), mx = ex > exm ? ex : exm;
    if (warp_any(zero || mx > 1023 + 128 || mx < 1023 - 128)) {
      if (zero) {
        p = p0;
        pm = pm0;
        neg = neg0;
        c = c0;
        slow(B);
      }
      const int a = dexp_field(p), b = dexp_field(pm), m = a > b ? a : b;
      const double f = (m > 1023 + 128 || m < 1023 - 128) ? dpow2(1023 - (m > 1 ? m : 1)) : 1.0;
      p *= f;
      pm *= f;
    }
#pragma unroll
    for (int k = 0; k < B; ++k) {
      E[k] = En[k];
      D[k] = Dn[k];
    }
  }
  slow(n - i0);
  return c;
}

// One round of multisection: the Sturm counts of np interior points of a target's interval
// [lo, hi] (any number of warps, on any SMs) leave the sub-interval that holds the eigenvalue.
//   point k < np of [lo, hi]: lo + (hi - lo) (k + 1) / (np + 1)
//   k = number of points whose count is <= target: the eigenvalue lies in [x_{k-1}, x_k]
// The interval ends within 4 ulp of its ends plus abstol (about eps ||T||: an eigenvalue near 0,
// e.g. every transition eigenvalue at W = 1/4 where the diagonal vanishes, needs no more).
FST_HD double bisect_point(double lo, double hi, int k, int np) {
  return lo + (hi - lo) * (double)(k + 1) / (double)(np + 1);
}
FST_HD void bisect_narrow(double *lo, double *hi, int k, int np) {
  const double a = *lo, b = *hi;
  if (k > 0) *lo = bisect_point(a, b, k - 1, np);
  if (k < np) *hi = bisect_point(a, b, k, np);
}
FST_HD bool bisect_converged(double lo, double hi, double abstol) {
  return hi - lo <= 4.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi)) + abstol;
}

// Plain bisection for one target (one thread), used when many plans are built at
// once: the throughput of thousands of independent targets matters more than the
// latency of one.  flag != 0 if it did not converge.
FST_HD void bisect1_body(const double *d, const double *e2, int n, int target, double glo, double ghi, double pivmin,
                         double abstol, double *out, int *flag) {
  double lo = glo, hi = ghi;
  int it = 0;
  for (; it < 256; ++it) {
    const double tol = 4.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi)) + abstol;
    if (hi - lo <= tol) break;
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (sturm_count(d, e2, n, mid, pivmin) > target) hi = mid;
    else lo = mid;
  }
  *out = 0.5 * (lo + hi);
  if (it == 256) *flag = 1;
}

// Descriptor of one eigen-target of a batch of plans (fst_plan_many).
struct TargetDesc {
  int64_t mat_off;   // reduced matrix: d, e, e2 at [mat_off, mat_off + n) of the concatenations
  int64_t x_off;     // this target's vector and derivative at [x_off, x_off + n), exponents at x_off / 8
  double *S;         // output: the full unit-norm Slepian vector (length N)
  int64_t N;
  int n, target, parity, pad_;
  double glo, ghi, pivmin, tol;
};

// Eigenvector of the reduced matrix (diag d, coupling e[i] between i-1 and i, r[i] = 1 / e[i+1])
// for the eigenvalue sigma, by its own rows from the edge to the centre:
//   z_0 = 1,  z_{i+1} = -((d_i - sigma) z_i + e_i z_{i-1}) / e_{i+1}.
// Row x from the centre (s = x^2, A = N^2/4) reads sigma = C s + (A - s) cos(phi), C = cos 2 pi W,
// so cos(phi) = (sigma - C s) / (A - s) is monotonic in s: every Slepian vector oscillates around
// the centre and has at most one region without oscillation, at the edge, where the recurrence
// follows the growing solution.  It is therefore stable for every index, each row is met to its
// own rounding, and only the last row is left with a residual, which is due to the rounding of
// sigma.  That is removed to first order with the derivative w = dz / d sigma,
//   (T - sigma) w = z on the same rows,  delta = -(last row of z) / (its derivative),
// and the vector is z + delta w (delta is a fraction of an ulp of ||T||).
// z and w are scaled by 2^256 at block ends (PLAN_B entries) when they leave 2^(+-128); ex holds
// each block's exponent.  A step grows them by at most about N/2 (at the edge), a block by less
// than 2^176, so one factor is enough and squares stay finite.
// Bound: a serial chain of n steps of 7 FP64 instructions of 64 clocks each; inputs are loaded
// PLAN_B steps ahead.  Measured at N = 65536 (44 targets of n = 32768): 7.8 ms; the inverse
// iteration with a partially pivoted LU that this replaced took 73.9 ms and left vectors
// orthogonal to 1e-11 where these reach 1e-13 (N = 86679, W = 0.0185).
FST_HD void fwdvec_body(const double *d, const double *e, const double *r, int n, double sigma, double *z, double *w,
                        int *ex, double *delta) {
  constexpr int B = PLAN_B;
  double zc = 1.0, zm = 0.0, wc = 0.0, wm = 0.0, rz = 0.0, rw = 0.0;
  int sh = 0;
  double D[B], E[B], R[B], Dn[B], En[B], Rn[B];
  load_block(d, D);
  load_block(e, E);
  load_block(r, R);
  for (int i0 = 0; i0 < n; i0 += B) {
    load_block(d + i0 + B, Dn);
    load_block(e + i0 + B, En);
    load_block(r + i0 + B, Rn);
    ex[i0 / B] = sh;
    auto step = [&](int k) {
      z[i0 + k] = zc;
      w[i0 + k] = wc;
      const double a = D[k] - sigma;
      rz = fma(a, zc, E[k] * zm);
      rw = fma(a, wc, fma(E[k], wm, -zc));
      zm = zc;
      wm = wc;
      zc = -rz * R[k];
      wc = -rw * R[k];
    };
    if (i0 + B <= n) {
#pragma unroll
      for (int k = 0; k < B; ++k) step(k);
    } else {
#pragma unroll
      for (int k = 0; k < B; ++k)
        if (i0 + k < n) step(k);
    }
    const int ea = dexp_field(zc), eb = dexp_field(zm), mx = ea > eb ? ea : eb;
    if (warp_any(mx > 1023 + 128 || mx < 1023 - 128)) {
      const double f = mx > 1023 + 128 ? 0x1p-256 : (mx < 1023 - 128 ? 0x1p256 : 1.0);
      zc *= f;
      zm *= f;
      wc *= f;
      wm *= f;
      sh += mx > 1023 + 128 ? 256 : (mx < 1023 - 128 ? -256 : 0);
    }
#pragma unroll
    for (int k = 0; k < B; ++k) {
      D[k] = Dn[k];
      E[k] = En[k];
      R[k] = Rn[k];
    }
  }
  const double dl = -rz / rw;   // the last row's residual over its derivative
  *delta = (dl - dl == 0.0) ? dl : 0.0;
}

// Expansion of a reduced vector (z + delta w with block exponents ex, size n, parity p) to the
// full unit-norm Slepian vector s (length N, contiguous) with the sign convention:
// symmetric vectors have positive sum, antisymmetric ones positive
// sum((N-1-2i) s[i]).  Block reductions in a fixed order.  sh: 2 * nthr doubles.
template <typename Ex>
FST_HD void finalize_body(Ex &ex, const double *z, const double *w, const int *bex, double delta, int n, int parity,
                          int64_t N, double *s, double *sh) {
  using St = typename Ex::State;
  const int nthr = ex.nthr;
  const bool odd = (N & 1) != 0;
  const int64_t m = N / 2;  // full index m is the centre when N is odd
  // entry i over 2^(largest block exponent)
  auto entry = [&](int64_t i, int top) {
    const int k = bex[i / PLAN_B] - top;
    return (k < -1792) ? 0.0 : fma(delta, w[i], z[i]) * ldexp(1.0, k < -1000 ? -1000 : k) * (k < -1000 ? ldexp(1.0, k + 1000) : 1.0);
  };
  ex.phase([&](int tid, St &) {
    int top = -2147483647;
    for (int i = tid; i < (n + PLAN_B - 1) / PLAN_B; i += nthr) top = bex[i] > top ? bex[i] : top;
    sh[tid] = (double)top;
  });
  ex.phase([&](int tid, St &) {
    if (tid == 0) {
      double top = sh[0];
      for (int k = 1; k < nthr; ++k) top = fmax(top, sh[k]);
      sh[nthr] = top;
    }
  });
  // (the sums below reuse sh: the exponent travels in the last slot until it is read)
  ex.phase([&](int tid, St &st) {
    st.top = (int)sh[nthr];
  });
  ex.phase([&](int tid, St &st) {
    double nrm = 0.0, ref = 0.0;
    for (int i = tid; i < n; i += nthr) {
      const double u = entry(i, st.top);
      nrm += u * u;
      if (parity == 0) ref += (odd && i == m) ? 0.7071067811865476 * u : u;  // centre counts once, times sqrt(2)/2
      else ref += (double)(N - 1 - 2 * (int64_t)i) * u;
    }
    sh[tid] = nrm;
    sh[nthr + tid] = ref;
  });
  ex.phase([&](int tid, St &) {
    if (tid == 0) {
      double nrm = 0.0, ref = 0.0;
      for (int k = 0; k < nthr; ++k) { nrm += sh[k]; ref += sh[nthr + k]; }
      // full norm^2 = 2 * reduced norm^2 (centre sample sqrt(2) u_m when present)
      const double scale = (ref < 0.0 ? -1.0 : 1.0) / sqrt(2.0 * nrm);
      sh[0] = scale;
    }
  });
  ex.phase([&](int tid, St &st) {
    const double scale = sh[0];
    const double sgn = (parity == 0) ? 1.0 : -1.0;
    for (int64_t i = tid; i < n; i += nthr) {
      const double v = entry(i, st.top) * scale;
      if (odd && i == m) {
        s[i] = 1.4142135623730951 * v;
      } else {
        s[i] = v;
        s[N - 1 - i] = sgn * v;
      }
    }
    if (odd && parity == 1 && tid == 0) s[m] = 0.0;
  });
}

// sum_i a[i] * b[i] for vector t (contiguous, length N), fixed-order block reduction
template <typename Ex>
FST_HD void dot_body(Ex &ex, const double *a, const double *b, int64_t N, double *out, double *sh) {
  using St = typename Ex::State;
  const int nthr = ex.nthr;
  ex.phase([&](int tid, St &) {
    double acc = 0.0;
    for (int64_t i = tid; i < N; i += nthr) acc += a[i] * b[i];
    sh[tid] = acc;
  });
  ex.phase([&](int tid, St &) {
    if (tid == 0) {
      double acc = 0.0;
      for (int k = 0; k < nthr; ++k) acc += sh[k];
      *out = acc;
    }
  });
}

FST_HD double sinpi_hd(double x) {
#ifdef __CUDA_ARCH__
  return sinpi(x);
#else
  return sin(M_PI * x);
#endif
}

// b[k] = sin(2 pi W k) / (pi k), b[0] = 2W (first row of B_{N,W}, Eq. "Prolate
// matrix").  The product 2Wk is formed exactly as hi + lo (fma) and reduced mod 2
// before the sine, so large k lose no accuracy to the argument.
FST_HD double sinc_row_value(int64_t k, double W) {
  if (k == 0) return 2.0 * W;
  const double a = 2.0 * W, kd = (double)k;
  const double hi = a * kd;
  const double lo = fma(a, kd, -hi);
  double r = fmod(hi, 2.0) + lo;
  if (r > 1.0) r -= 2.0;
  return sinpi_hd(r) / (M_PI * kd);
}

// circulant embedding c of length M: c[k] = c[M-k] = b[k] for 0 <= k < N, else 0
FST_HD double sinc_embed_at(int64_t k, int64_t N, int64_t M, double W) {
  if (k < N) return sinc_row_value(k, W);
  if (k > M - N) return sinc_row_value(M - k, W);
  return 0.0;
}

}  // namespace fst
