// Krylov exponential y = exp(-i s H) x of the sweep: the Lanczos scalars, the small
// exponential, the re-orthogonalisation and the cluster-resident form (included by sweep.cu).
//
// What bounds it: latency.  A warp's FP64 instruction holds the SM's FP64 unit for about 20
// cycles whatever its lanes do, so scalars that all eight warps repeat cost as much as the
// vector work (measured per CTA: square root 2500 cycles, division 1250, pow 12800, against
// 450 for a cluster barrier).  The scalars of a step are therefore computed by one thread and
// read from shared memory, the square root and reciprocal overlap the vector update, and the
// convergence checks start with an FP32 estimate.

// ------------------------------------------------------------------ Lanczos exponential
struct KrylovShared {
  double alpha[TTNS_KMAX + 1];
  double beta[TTNS_KMAX + 2];   // beta[j] couples j-1 and j
  double scale[TTNS_KMAX + 1];  // q_j = scale[j] * K_j
  double ure[TTNS_KMAX];        // y = sum_k (ure + i uim)[k] K_k
  double uim[TTNS_KMAX];
  double rv[2][2 * (TTNS_KMAX + 1)];  // orthogonalisation: per-CTA dot partials (alternating),
  double cq[2 * (TTNS_KMAX + 1)];     // <q_i, w>
  double ck[2 * (TTNS_KMAX + 1)];     // and <q_i, w> scale_i: w -= sum_i ck_i K_i
  double beta0;                 // |x|
  double ca, cm;                // alpha_j scale_j and beta_j scale_{j-1} of the current step
  double b2;                    // |w - alpha_j q_j|^2
  double lead;
  double ratio;
  double s_done;
  int fused, check, conv, again;
  int full;                     // the last check left the expansion of its m and s in ure, uim
};
__shared__ KrylovShared s_ks;

// Scalars of the recurrence, each on one thread.
__device__ __forceinline__ void krylov_begin(KrylovShared& ks, double n2) {
  const double b = sqrt(n2);
  ks.beta0 = b;
  ks.scale[0] = b > 0.0 ? 1.0 / b : 0.0;
  ks.beta[0] = 0.0;
  ks.cm = 0.0;
  ks.lead = 1.0;
}
// alpha_j from Re <K_j, w>; in the mixed modes also
//   |w - alpha_j q_j|^2 = |w|^2 - 2 alpha_j^2 + alpha_j^2 |q_j|^2
// with |q_j|^2 from the same reduction (the error of an assumed |q_j| = 1 would grow by
// alpha^2 / beta^2 per step); used unless it cancels (the same decision on every CTA)
__device__ __forceinline__ void krylov_alpha(KrylovShared& ks, int j, double kw) {
  const double sj = ks.scale[j], aj = kw * sj;
  ks.alpha[j] = aj;
  ks.ca = aj * sj;
}
__device__ __forceinline__ void krylov_alpha(KrylovShared& ks, int j, double kw, double ww, double kk) {
  const double sj = ks.scale[j], aj = kw * sj;
  const double nq = sj * sj * kk;
  const double b2 = ww - aj * aj * (2.0 - nq);
  ks.alpha[j] = aj;
  ks.ca = aj * sj;
  ks.b2 = b2;
  ks.fused = b2 > 1e-4 * ww;
}
// beta_{j+1} = sqrt(b2) and its reciprocal, and whether step m = j + 1 is worth a convergence
// check: `lead` is the leading-order size of |e_m^T exp(-i s T_m) e_0|,
// |s|^(m-1) prod beta_i / (m-1)!
__device__ __forceinline__ void krylov_norm(KrylovShared& ks, int j, double b2, double s, double tol, int mmax) {
  double b = b2, r = 0.0;
  if (b2 > 0.0) {
    r = rsqrt(b2);
    b = b2 * r;
    b = fma(fma(-b, b, b2), 0.5 * r, b);
  }
  ks.beta[j + 1] = b;
  ks.scale[j + 1] = r;
  ks.cm = b * ks.scale[j];
  const int m = j + 1;
  const double est = b * ks.lead;
  ks.lead *= fabs(s) * b * c_inv[m];
  ks.check = est <= 1e2 * tol || m == mmax || !(b > 0.0);
}

// ------------------------------------------------------------------ tridiagonal exponential
// u = exp(-i s T) e_0 for the real symmetric tridiagonal T (diag a[0..m), off-diagonal
// b[1..m) with b[k] coupling k-1 and k), by a Chebyshev expansion on the Gershgorin interval:
//   exp(-i z X) = J_0(z) + 2 sum_n (-i)^n J_n(z) T_n(X),  X = (T - c) / R,  z = s R.
// One warp (lane k holds component k, m <= 32).  The Chebyshev vectors of a real start vector
// are real: the even orders give the real part and the odd ones the imaginary part.

// The Gershgorin interval in FP32, widened by its rounding, and the Chebyshev order K whose
// coefficients (|z|/2)^n / n! fall below 1e-18; p0, p1: those bounds for n = lane, lane + 32.
struct ChebSetup {
  float c, R, z;   // centre, radius, |s| R
  float p0, p1;
  int K;
};
__device__ __forceinline__ ChebSetup cheb_setup(const double* a, const double* b, int m, float s_abs) {
  const int lane = threadIdx.x & 31;
  const bool on = lane < m;
  const float ak = on ? (float)a[lane] : 0.f;
  const float bk = (on && lane > 0) ? fabsf((float)b[lane]) : 0.f;
  const float bk1 = (lane + 1 < m) ? fabsf((float)b[lane + 1]) : 0.f;
  float lo = on ? ak - bk - bk1 : 3e38f, hi = on ? ak + bk + bk1 : -3e38f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  ChebSetup cs;
  cs.c = 0.5f * (hi + lo);
  cs.R = 0.5f * (hi - lo) + 1e-6f * (fabsf(hi) + fabsf(lo));
  cs.z = s_abs * cs.R;
  return cs;
}
// K, p0 and p1 for the argument z (at most 32)
__device__ __forceinline__ void cheb_order(ChebSetup& cs, float z) {
  const int lane = threadIdx.x & 31;
  float p = lane > 0 ? 0.5f * z / (float)lane : 1.f;  // prefix product over the lanes: (z/2)^n / n!
  float q = 0.5f * z / (float)(lane + 32);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float a = __shfl_up_sync(0xffffffffu, p, o), b = __shfl_up_sync(0xffffffffu, q, o);
    if (lane >= o) {
      p *= a;
      q *= b;
    }
  }
  q *= __shfl_sync(0xffffffffu, p, 31);
  cs.p0 = p;
  cs.p1 = q;
  const unsigned b0 = __ballot_sync(0xffffffffu, p > 1e-18f || (float)lane < z + 2.f);
  const unsigned b1 = __ballot_sync(0xffffffffu, q > 1e-18f);
  cs.K = b1 ? 64 - __clz(b1) : 32 - __clz(b0);
}

__device__ __noinline__ void texp_warp(const double* a, const double* b, int m, double s, double* ure, double* uim) {
  const int lane = threadIdx.x & 31;
  const bool on = lane < m;
  ChebSetup cs = cheb_setup(a, b, m, fabsf((float)s));
  const double c = m > 1 ? (double)cs.c : a[0];  // one component: the phase alone
  double vre = lane == 0 ? 1.0 : 0.0, vim = 0.0;
  if (m > 1 && cs.R > 0.f && cs.z >= 1e4f) {
    // hundreds of sub-steps on one warp, for a time that no Krylov space of this size covers:
    // NaN, which the caller reports (a vector left at e_0 would pass its convergence check)
    vre = vim = __longlong_as_double(0x7ff8000000000000LL);
  } else if (m > 1 && cs.R > 0.f && cs.z > 0.f) {  // (a NaN in the input reaches the result through c)
    // sub-steps of |z| <= 28: the order stays below 64
    const int nsub = (int)ceilf(cs.z * (1.0f / 28.0f));
    const double R = (double)cs.R;
    const double z = fabs(s) * R / (double)nsub;
    cheb_order(cs, (float)z);
    const int K = cs.K;
    // Bessel functions J_n(z), n < 64 (lane n and n - 32), by backward recurrence from an order
    // beyond K, normalised by J_0 + 2 sum J_2k = 1 (Miller's algorithm).  The factor 2 n / z is
    // formed anew at every order: stepped down by 2 / z its error reaches N roundings of the first
    // factor at the small orders, which carry the norm (error of the exponential at z = 3: 6.6e-15
    // against 7e-16).  J_0 is what the others leave of 1, to half a rounding for small z.
    double J0 = 0.0, J1 = 0.0;
    if (z > 1e-9) {
      const int N = ((K + 9) / 2) * 2;
      const double h = 2.0 / z;
      double f = 1e-30, f1 = 0.0, even = 0.0, dn = (double)N;
      for (int n = N; n > 0; --n) {
        if (n == lane) J0 = f;
        if (n == lane + 32) J1 = f;
        if ((n & 1) == 0) even += f;
        const double fm = fma(dn * h, f, -f1);
        dn -= 1.0;
        f1 = f;
        f = fm;
      }
      const double inv = 1.0 / fma(2.0, even, f);  // f: order 0
      J0 = lane == 0 ? fma(-2.0 * inv, even, 1.0) : J0 * inv;
      J1 *= inv;
    } else {  // the first two terms of each power series
      J0 = lane == 0 ? 1.0 : (lane == 1 ? 0.5 * z : (lane == 2 ? 0.125 * z * z : 0.0));
    }
    const double rinv = 1.0 / R;
    const double dk = on ? 2.0 * (a[lane] - c) * rinv : 0.0;
    const double ek = (on && lane > 0) ? 2.0 * b[lane] * rinv : 0.0;
    const double fk = lane + 1 < m ? 2.0 * b[lane + 1] * rinv : 0.0;
    // E v = sum over even n, O v = sum over odd n of (-1)^(n/2) (2 -) J_n T_n(X) v, v real
    auto cheb = [&](double v, double& E, double& O) {
      E = 0.0;
      O = 0.0;
      double t = v, tm = 0.0;
      for (int n = 0; n < K; ++n) {
        const double jn = __shfl_sync(0xffffffffu, n < 32 ? J0 : J1, n & 31);
        const double w = (n & 2) ? -jn : jn;
        if (n & 1)
          O = fma(w, t, O);
        else
          E = fma(n ? w : 0.5 * w, t, E);
        const double tl = __shfl_up_sync(0xffffffffu, t, 1), tr = __shfl_down_sync(0xffffffffu, t, 1);
        // 2 X t (ek of lane 0 and fk of lane m - 1 are zero); the first step takes X t
        double x = fma(dk, t, n ? -tm : 0.0);
        x = fma(ek, tl, x);
        x = fma(fk, tr, x);
        tm = t;
        t = n ? x : 0.5 * x;
      }
      E += E;
      O += O;
    };
    const double sg = s < 0.0 ? 1.0 : -1.0;  // exp(-i z X) v = E v - i O v for s > 0
    for (int sub = 0; sub < nsub; ++sub) {
      double E, O, E2 = 0.0, O2 = 0.0;
      cheb(vre, E, O);
      if (sub > 0) cheb(vim, E2, O2);
      vre = fma(-sg, O2, E);
      vim = fma(sg, O, E2);
    }
  }
  // global phase exp(-i s c)
  double sn, cn;
  sincos(-s * c, &sn, &cn);
  if (on) {
    ure[lane] = vre * cn - vim * sn;
    uim[lane] = vre * sn + vim * cn;
  }
  __syncwarp();
}

// Convergence of step m: beta_m |e_m^T exp(-i s T_m) e_0| <= tol, decided as the FP64 expansion
// decides it.  That takes 4 us and more on one warp, so an FP32 estimate comes first and answers
// where it is certain.  Component m has no contribution from orders below m - 1, and the series of
// an order n loses about z^2 / (2 n) / ln 10 digits to cancellation.  For components of 1e-15 and
// more the estimate was off by at most 6e-4 up to z^2 = 12 m and 6e-3 up to 20 m (15000 random and
// Krylov matrices of m = 2 to 32 against FP64; beyond 30 m it can be off by any factor).  Within 1 %
// or 5 % of the tolerance, with wider spectra and for smaller tolerances the FP64 expansion decides:
// one step more or less changes what is left below the tolerance, and the QR's null decisions can
// amplify that.  (With 12 m as the limit, 256 chains of up to 40 sites took 4.8 % longer.)  `full`:
// ure and uim hold the FP64 expansion.
__device__ __noinline__ bool krylov_small(const KrylovShared& ks, int m, double s, double tol, double* ure,
                                          double* uim, bool* nonfinite, bool* full) {
  const int lane = threadIdx.x & 31;
  const double bn = ks.beta[m];
  ChebSetup cs = cheb_setup(ks.alpha, ks.beta, m, fabsf((float)s));
  *nonfinite = false;
  *full = false;
  const float width = cs.z * cs.z / (float)m;
  if (width <= 20.f && tol >= 1e-15 * bn) {
    cheb_order(cs, cs.z);
    const int K = min(64, cs.K + 4);
    const float y = -0.25f * cs.z * cs.z;
    float h0 = 1.f, h1 = 1.f;
    for (int j = 8 + (int)(2.f * cs.z); j >= 1; --j) {  // J_n = (z/2)^n / n! sum_j y^j n! / (j! (n+j)!)
      h0 = fmaf(h0 * y, __fdividef(1.f, (float)(j * (j + lane))), 1.f);
      h1 = fmaf(h1 * y, __fdividef(1.f, (float)(j * (j + lane + 32))), 1.f);
    }
    const float J0 = cs.p0 * h0, J1 = cs.p1 * h1;
    const float ri = cs.R > 1e-30f ? 2.f / cs.R : 0.f;  // (a smaller radius is zero: its reciprocal overflows)
    const float dk = lane < m ? ri * (float)(ks.alpha[lane] - (double)cs.c) : 0.f;
    const float ek = (lane < m && lane > 0) ? ri * (float)ks.beta[lane] : 0.f;
    const float fk = lane + 1 < m ? ri * (float)ks.beta[lane + 1] : 0.f;
    float t = lane == 0 ? 1.f : 0.f, tm = 0.f, E = 0.f, O = 0.f;
    for (int n = 0; n < K; ++n) {
      const float jn = __shfl_sync(0xffffffffu, n < 32 ? J0 : J1, n & 31);
      const float w = ((n & 2) ? -jn : jn) * 1.099511627776e12f;  // 2^40: the squares stay in range
      if (n & 1)
        O = fmaf(w, t, O);
      else
        E = fmaf(n ? w : 0.5f * w, t, E);
      const float tl = __shfl_up_sync(0xffffffffu, t, 1), tr = __shfl_down_sync(0xffffffffu, t, 1);
      const float x = fmaf(fk, tr, fmaf(ek, tl, fmaf(dk, t, n ? -tm : 0.f)));
      tm = t;
      t = n ? x : 0.5f * x;
    }
    float um = 2.f * sqrtf(E * E + O * O) * 9.094947017729282e-13f;
    um = __shfl_sync(0xffffffffu, um, m - 1);
    const double err = bn * (double)um;
    const double margin = width <= 12.f ? 0.01 : 0.05;
    if (err <= (1.0 - margin) * tol) return true;
    if (err >= (1.0 + margin) * tol) return false;
  }
  texp_warp(ks.alpha, ks.beta, m, s, ure, uim);
  *full = true;
  const double r = ure[m - 1], i = uim[m - 1];
  const double err = bn * sqrt(r * r + i * i);
  if (!(err == err)) *nonfinite = true;
  return err <= tol || !(bn > 0.0);
}
__device__ __forceinline__ void krylov_check(KrylovShared& ks, int m, double s, double tol) {
  bool bad, full;
  const bool ok = krylov_small(ks, m, s, tol, ks.ure, ks.uim, &bad, &full);
  if ((threadIdx.x & 31) == 0) {
    ks.conv = bad ? 2 : (ok ? 1 : 0);
    ks.full = full;
  }
}
// After the last step (warp 0): the time that the space covers (s, or with `halve` the largest
// s / 2^k, k <= 30, that reaches the tolerance) and the coefficients of the result, which a check in
// FP64 has left behind.  (A step ends with a check: at the last m of a space at the latest.)
__device__ __noinline__ void krylov_exp(KrylovShared& ks, int m, double s, double tol, bool halve) {
  const int lane = threadIdx.x & 31;
  bool full = ks.full != 0;
  if (halve) {
    for (int k = 0; k < 30; ++k) {
      s *= 0.5;
      bool bad;
      if (krylov_small(ks, m, s, tol, ks.ure, ks.uim, &bad, &full)) break;
    }
  }
  if (!full) texp_warp(ks.alpha, ks.beta, m, s, ks.ure, ks.uim);
  if (lane < m) {
    const double sc = ks.beta0 * ks.scale[lane];
    ks.ure[lane] *= sc;
    ks.uim[lane] *= sc;
  }
  if (lane == 0) ks.s_done = s;
}

// Full reorthogonalisation of the FP64 path: after the three-term recurrence, a classical
// Gram-Schmidt pass of w against all q_i = scale_i K_i, i = 0..j,
//   w <- w - sum_i <q_i, w> q_i,  <q_i, w> = scale_i <K_i, w>,
// and a second one where the first removed more than 1e-6 of w (below that the first leaves w
// orthogonal to rounding: "twice is enough").  A pass costs one team reduction (fixed order); it
// also sums |w|^2, so that |w|^2 afterwards is |w|^2 - sum |<q_i, w>|^2 without another
// reduction, unless that cancels (ks.fused = 0: the caller sums the returned shares of |w|^2).
__device__ __forceinline__ void orth_store(KrylovShared& ks, int j, int k, double sum) {
  const int i = k >> 1;
  if (i <= j) {
    const double c = sum * ks.scale[i];
    ks.cq[k] = c;
    ks.ck[k] = c * ks.scale[i];
  } else {
    ks.cq[k] = sum;  // |w|^2 in the real slot of the vector after the last
  }
}
__device__ __forceinline__ void orth_scalars(KrylovShared& ks, int j, int pass) {  // one warp
  const int lane = threadIdx.x & 31;
  double c = 0.0;
  if (lane <= j) c = fma(ks.cq[2 * lane], ks.cq[2 * lane], ks.cq[2 * lane + 1] * ks.cq[2 * lane + 1]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) {
    const double ww = ks.cq[2 * (j + 1)];
    ks.b2 = ww - c;
    ks.fused = ks.b2 > 0.25 * ww;
    ks.again = pass == 0 && !(c <= 1e-12 * ww);
  }
}

// Vectors in global memory, elements idx = gtid + k * nthr (op_expm):
__device__ __noinline__ double orth_strided(Team& tm, long long N, const double2* x, const double2* Kb, long long kv,
                                            double2* W, int j, KrylovShared& ks) {
  __shared__ double s_wp[NWARP][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto Kp = [&](int i) -> const double2* { return i == 0 ? x : Kb + (long long)(i - 1) * kv; };  // Kp(j + 1) is W
  double nrm = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    double* mine = ks.rv[pass];
    const int nv = j + 2;
    for (int i0 = 0; i0 < nv; i0 += 8) {
      const int ni = min(8, nv - i0);
      double acc[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) acc[q] = 0.0;
      for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
        const double2 w = W[idx];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (q < ni) {
            const double2 k = Kp(i0 + q)[idx];
            acc[2 * q] = fma(k.x, w.x, fma(k.y, w.y, acc[2 * q]));
            acc[2 * q + 1] = fma(k.x, w.y, fma(-k.y, w.x, acc[2 * q + 1]));
          }
        }
      }
      const double t = warp_reduce_t<16>(acc);
      if ((lane & 1) == 0) s_wp[warp][warp_reduce_vid<16>(lane)] = t;
      __syncthreads();
      if (threadIdx.x < 2 * ni) {
        double sum = 0.0;
        for (int w = 0; w < NWARP; ++w) sum += s_wp[w][threadIdx.x];
        mine[2 * i0 + threadIdx.x] = sum;
      }
      __syncthreads();
    }
    team_reduce_vec(tm, mine, 2 * nv, [&](int k, double v) { orth_store(ks, j, k, v); });
    if (warp == NWARP - 1) orth_scalars(ks, j, pass);
    nrm = 0.0;
    for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
      double2 w = W[idx], w1 = make_double2(0.0, 0.0);
      int i = 0;
      for (; i + 1 <= j; i += 2) {  // two chains
        const double2 k0 = Kp(i)[idx], k1 = Kp(i + 1)[idx];
        const double r0 = ks.ck[2 * i], i0 = ks.ck[2 * i + 1], r1 = ks.ck[2 * i + 2], i1 = ks.ck[2 * i + 3];
        w.x = fma(-r0, k0.x, fma(i0, k0.y, w.x));
        w.y = fma(-r0, k0.y, fma(-i0, k0.x, w.y));
        w1.x = fma(-r1, k1.x, fma(i1, k1.y, w1.x));
        w1.y = fma(-r1, k1.y, fma(-i1, k1.x, w1.y));
      }
      if (i <= j) {
        const double2 k0 = Kp(i)[idx];
        const double r0 = ks.ck[2 * i], i0 = ks.ck[2 * i + 1];
        w.x = fma(-r0, k0.x, fma(i0, k0.y, w.x));
        w.y = fma(-r0, k0.y, fma(-i0, k0.x, w.y));
      }
      w.x += w1.x;
      w.y += w1.y;
      W[idx] = w;
      nrm = fma(w.x, w.x, fma(w.y, w.y, nrm));
    }
    __syncthreads();  // ks.again, fused and b2; the coefficients are rewritten by the next pass
    if (!ks.again) break;
  }
  return nrm;
}

struct PhaseClock {
  long long t;
  bool on;
  bool grid;  // phases of grid-team ops go to their own counters
  __device__ void start(bool enable, bool grid_team = false) {
    on = enable;
    grid = grid_team;
    t = clock64();
  }
  __device__ void lap(Ctl* ctl, int phase) {
    if (!on) return;
    const long long now = clock64();
    atomicAdd(grid ? &ctl->phase_cycles_grid[phase] : &ctl->phase_cycles[phase], (unsigned long long)(now - t));
    t = now;
  }
};

// ------------------------------------------------------------------ cluster-resident form
// Each CTA of the cluster owns a contiguous slice of every Krylov vector in its shared memory
// (vectors beyond the shared memory's room go to the worker's global workspace).  Every CTA
// holds the whole input vector of an application: the owner of an element writes it to all
// CTAs through distributed shared memory when it updates it, before the cluster barrier that
// the step needs anyway, so that an application starts from local shared memory.  Operators
// are staged once per exponential: of a factor on the outermost leg only the rows that the own
// slice reads.  The arithmetic is the same as op_expm's (same recurrence, same convergence and
// substep rules).
//
// An application's work items are (element, term group) pairs: the slices are a few to a few
// hundred elements, so one thread per element would leave most of the CTA idle while it walks
// through all terms; the groups' partial values are added in a fixed order by the element's
// owner.
struct ClTerm {
  int dD, dst, dl, doff;            // dense factor: dimension (0: none), stride, leg, staged position of row 0
  int dr;                           // staged row length, odd: lanes on different rows read different banks
  int r0, nr;                       // staged rows
  int snnz, sD, sst, sl, soff;      // row-sparse factor: entries per row (0: none), ...
  int xo;                           // input: offset from xs (0, or a first factor's result)
  int lo, hi;                       // first factors of two-stage terms: element range
  long long dmat, sp;               // pool offsets
};

// leg indices of element e, eight bits each
__device__ __forceinline__ unsigned long long leg_pack(const NodeDesc& nd, int e) {
  unsigned long long p = 0;
  for (int l = 0; l < nd.nl; ++l) {
    const int i = fdivu(e, nd.strides[l], nd.inv_strides[l]);
    e -= i * nd.strides[l];
    p |= (unsigned long long)i << (8 * l);
  }
  return p;
}

template <typename T>
__device__ __forceinline__ typename C2<T>::t dot_at(const typename C2<T>::t* row, int D, const typename C2<T>::t* x,
                                                    int st) {
  using V = typename C2<T>::t;
  V a0, a1, a2, a3;
  a0.x = a0.y = a1.x = a1.y = a2.x = a2.y = a3.x = a3.y = (T)0;
  int k = 0;
  for (; k + 3 < D; k += 4) {
    const V m0 = row[k], m1 = row[k + 1], m2 = row[k + 2], m3 = row[k + 3];
    const V x0 = x[0], x1 = x[st], x2 = x[2 * st], x3 = x[3 * st];
    x += 4 * st;
    cmac<T>(a0, m0, x0);
    cmac<T>(a1, m1, x1);
    cmac<T>(a2, m2, x2);
    cmac<T>(a3, m3, x3);
  }
  for (; k < D; ++k, x += st) cmac<T>(a0, row[k], x[0]);
  a0.x += a1.x + (a2.x + a3.x);
  a0.y += a1.y + (a2.y + a3.y);
  return a0;
}

// value of one term at element e (sm: the staged operators)
template <typename T>
__device__ __forceinline__ typename C2<T>::t cl_term(const ClTerm& c, const typename C2<T>::t* sm,
                                                     const typename C2<T>::t* xs, int e, unsigned long long pk) {
  using V = typename C2<T>::t;
  const V* x = xs + c.xo;
  const int i = (int)(pk >> (8 * c.dl)) & 255;
  const V* row = sm + c.doff + i * c.dr;
  if (c.snnz == 0) return dot_at<T>(row, c.dD, x + (e - i * c.dst), c.dst);
  const int is = (int)(pk >> (8 * c.sl)) & 255;
  const V* vals = sm + c.soff + is * c.snnz;
  const V* cols = vals + c.sD * c.snnz;
  V acc;
  acc.x = acc.y = (T)0;
  for (int q = 0; q < c.snnz; ++q) {
    const V v = vals[q];
    if (v.x == (T)0 && v.y == (T)0) continue;
    const int e2 = e + ((int)cols[q].x - is) * c.sst;
    const V d = c.dD ? dot_at<T>(row, c.dD, x + (e2 - i * c.dst), c.dst) : x[e2];
    cmac<T>(acc, v, d);
  }
  return acc;
}

// shared-memory plan of one exponential (byte offsets; the same on every CTA of the cluster)
struct ClPlan {
  int ok, G, cap;                     // term groups; Krylov vectors held in shared memory
  int pk, mats, xs, py, basis;
};
__shared__ ClPlan s_cl;

template <typename T>
__device__ void cl_plan(const KernelParams& P, const NodeDesc& nd, const TermList& L, int S, int e0, int e1, int mmax,
                        ClTerm* ct) {
  using V = typename C2<T>::t;
  const int N = nd.size, nt = L.count, n2 = L.n2;
  // term t < nt: its last factor (second factors of two-stage terms act on a first factor's
  // result); nt <= t < nt + n2: the first factors
  for (int t = threadIdx.x; t < nt + n2; t += NT) {
    const Term& T_ = P.terms[L.first + (t < nt ? t : t - n2)];
    ClTerm c{};
    const bool second = t < nt && t >= nt - n2;
    c.lo = max(0, e0);
    c.hi = max(c.lo, e1);
    if (second || t >= nt) {
      // first factors on the slice widened to whole blocks of the second factor's leg
      const int l2 = T_.f[1].leg;
      const int blk = nd.dims[l2] * nd.strides[l2];
      if (e1 > e0 && t >= nt) {
        c.lo = (e0 / blk) * blk;
        c.hi = min(N, ((e1 - 1) / blk + 1) * blk);
      }
      c.xo = second ? -((e0 / blk) * blk) : 0;  // completed below
      c.nr = S + 2 * blk;                       // room of the result (uniform over the CTAs)
    }
    int ext = second || t < nt ? S : c.nr;  // extent of the range whose rows are staged
    const int nf = (second || t >= nt) ? 1 : T_.nf;
    for (int q = 0; q < nf; ++q) {
      const Factor& f = second ? T_.f[1] : T_.f[q];
      if (f.nnz > 0) {
        c.snnz = f.nnz;
        c.sD = nd.dims[f.leg];
        c.sst = nd.strides[f.leg];
        c.sl = f.leg;
        c.sp = f.sp;
      } else {
        c.dD = nd.dims[f.leg];
        c.dr = c.dD | 1;
        c.dst = nd.strides[f.leg];
        c.dl = f.leg;
        c.dmat = f.mat;
      }
    }
    if (nf == 2 && T_.f[0].nnz > 0 && T_.f[1].nnz > 0) c.sD = -1;  // (not produced by the compiler)
    c.soff = ext;
    ct[t] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ClPlan& pl = s_cl;
    long long off = (long long)(nt + n2) * sizeof(ClTerm);
    off = (off + 15) & ~15LL;
    pl.pk = (int)off;
    off += (long long)S * 8;
    off = (off + 15) & ~15LL;
    pl.mats = (int)off;
    long long m = 0;
    long long tmp = N;
    bool bad = false;
    for (int t = 0; t < nt + n2; ++t) {
      ClTerm& c = ct[t];
      const int ext = c.soff;
      bad |= c.sD < 0;
      if (t >= nt - n2 && t < nt) {  // second factor: reads its first factor's result
        c.xo += (int)tmp;
        tmp += c.nr;
      }
      c.soff = 0;
      c.r0 = 0;
      c.nr = c.dD;
      if (c.dD) {
        int rows = c.dD;
        if (c.dD * c.dst == N) {  // outermost leg: the rows of the own range
          rows = min(c.dD, ext / c.dst + 2);
          c.r0 = c.hi > c.lo ? c.lo / c.dst : 0;
          c.nr = c.hi > c.lo ? (c.hi - 1) / c.dst - c.r0 + 1 : 0;
        }
        c.doff = (int)m - c.r0 * c.dr;
        m += (long long)rows * c.dr;
      }
      if (c.snnz) {
        c.soff = (int)m;
        m += 2LL * max(0, c.sD) * c.snnz;
      }
    }
    off += m * (long long)sizeof(V);
    off = (off + 15) & ~15LL;
    pl.xs = (int)off;
    off += tmp * (long long)sizeof(V);
    pl.G = max(1, min(nt, NT / max(S, 1)));
    pl.py = (int)off;
    if (pl.G > 1) off += (long long)pl.G * S * sizeof(V);
    off = (off + 15) & ~15LL;
    pl.basis = (int)off;
    const long long room = off < P.smem_bytes ? (P.smem_bytes - off) / ((long long)S * (long long)sizeof(double2)) : 0;
    pl.cap = (int)min((long long)mmax + 1, room);
    pl.ok = !bad && pl.cap >= min(mmax + 1, 6);
  }
  __syncthreads();
}

template <typename T>
__device__ void cl_stage(const KernelParams& P, const ClTerm* ct, int n, typename C2<T>::t* sm) {
  using V = typename C2<T>::t;
  const V* src = ops<T>(P);
  auto cp = [&](V* d, const V* s) {
    if constexpr (sizeof(V) == 16)
      cp_async16(d, s);
    else
      cp_async8(d, s);
  };
  for (int t = 0; t < n; ++t) {
    const ClTerm& c = ct[t];
    if (c.dD) {
      V* d = sm + c.doff + c.r0 * c.dr;
      const V* s = src + c.dmat + (long long)c.r0 * c.dD;
      const int pad = c.dr - c.dD;
      const float inv = 1.0f / (float)c.dD;
      for (int k = threadIdx.x; k < c.nr * c.dD; k += NT) cp(d + k + pad * fdivu(k, c.dD, inv), s + k);
    }
    if (c.snnz)
      for (int k = threadIdx.x; k < 2 * c.sD * c.snnz; k += NT) cp(sm + c.soff + k, src + c.sp + k);
  }
  cp_async_wait_all();
}

// orthogonalisation with the own slices, elements [0, n_own): Ks(i) is vector i's slice
template <typename KF>
__device__ __forceinline__ double orth_slices(Team& tm, KF&& Ks, int n_own, int j, KrylovShared& ks) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double2* W = Ks(j + 1);
  double nrm = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    double* mine = ks.rv[pass];
    const int nv = j + 2;
    __syncthreads();  // w was written with the thread-strided mapping; the dots read it per lane
    for (int i0 = 4 * warp; i0 < nv; i0 += 4 * NWARP) {  // four vectors per warp, lanes over the slice
      const double2* K[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) K[q] = Ks(min(i0 + q, nv - 1));
      double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int e = lane; e < n_own; e += 32) {
        const double2 w = W[e];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double2 k = K[q][e];
          acc[2 * q] = fma(k.x, w.x, fma(k.y, w.y, acc[2 * q]));
          acc[2 * q + 1] = fma(k.x, w.y, fma(-k.y, w.x, acc[2 * q + 1]));
        }
      }
      const double t = warp_reduce_t<8>(acc);
      if ((lane & 3) == 0) {
        const int vid = warp_reduce_vid<8>(lane);
        if (i0 + (vid >> 1) < nv) mine[2 * i0 + vid] = t;
      }
    }
    team_reduce_vec(tm, mine, 2 * nv, [&](int k, double v) { orth_store(ks, j, k, v); });
    if (warp == NWARP - 1) orth_scalars(ks, j, pass);
    nrm = 0.0;
    for (int e = threadIdx.x; e < n_own; e += NT) {
      double2 w = W[e], w1 = make_double2(0.0, 0.0);
      int i = 0;
      for (; i + 1 <= j; i += 2) {  // two chains
        const double2 k0 = Ks(i)[e], k1 = Ks(i + 1)[e];
        const double r0 = ks.ck[2 * i], i0 = ks.ck[2 * i + 1], r1 = ks.ck[2 * i + 2], i1 = ks.ck[2 * i + 3];
        w.x = fma(-r0, k0.x, fma(i0, k0.y, w.x));
        w.y = fma(-r0, k0.y, fma(-i0, k0.x, w.y));
        w1.x = fma(-r1, k1.x, fma(i1, k1.y, w1.x));
        w1.y = fma(-r1, k1.y, fma(-i1, k1.x, w1.y));
      }
      if (i <= j) {
        const double2 k0 = Ks(i)[e];
        const double r0 = ks.ck[2 * i], i0 = ks.ck[2 * i + 1];
        w.x = fma(-r0, k0.x, fma(i0, k0.y, w.x));
        w.y = fma(-r0, k0.y, fma(-i0, k0.x, w.y));
      }
      w.x += w1.x;
      w.y += w1.y;
      W[e] = w;
      nrm = fma(w.x, w.x, fma(w.y, w.y, nrm));
    }
    __syncthreads();  // ks.again, fused and b2
    if (!ks.again) break;
  }
  return nrm;
}

// y = beta0 sum_k u_k q_k into the own part of K_0; returns this thread's share of |y|^2
template <typename KF>
__device__ __forceinline__ double krylov_combine(const KrylovShared& ks, KF&& Ks, int n_own, int m) {
  double ny = 0.0;
  for (int e = threadIdx.x; e < n_own; e += NT) {
    double yr = 0.0, yi = 0.0, zr = 0.0, zi = 0.0;  // two chains
    int k = 0;
    for (; k + 1 < m; k += 2) {
      const double2 q = Ks(k)[e], p = Ks(k + 1)[e];
      yr = fma(ks.ure[k], q.x, fma(-ks.uim[k], q.y, yr));
      yi = fma(ks.ure[k], q.y, fma(ks.uim[k], q.x, yi));
      zr = fma(ks.ure[k + 1], p.x, fma(-ks.uim[k + 1], p.y, zr));
      zi = fma(ks.ure[k + 1], p.y, fma(ks.uim[k + 1], p.x, zi));
    }
    if (k < m) {
      const double2 q = Ks(k)[e];
      yr = fma(ks.ure[k], q.x, fma(-ks.uim[k], q.y, yr));
      yi = fma(ks.ure[k], q.y, fma(ks.uim[k], q.x, yi));
    }
    yr += zr;
    yi += zi;
    Ks(0)[e] = make_double2(yr, yi);
    ny = fma(yr, yr, fma(yi, yi, ny));
  }
  return ny;
}

template <typename T>
__device__ __noinline__ bool op_expm_cluster(const KernelParams& P, Team& tm, const Instr& I, double2* work,
                                             double tau) {
  using V = typename C2<T>::t;
  KrylovShared& ks = s_ks;
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0);
  const NodeDesc nd = P.nodes[I.node];
  const TermList L = P.lists[I.terms];
  const int N = nd.size;
  const int cs = tm.size;
  const int S = (N + cs - 1) / cs;  // slice length
  const int e0 = min(N, tm.rank * S);
  const int e1 = min(N, e0 + S);
  const int n_own = e1 - e0;
  const int mmax = min(P.mmax, min(N, TTNS_KMAX));
  const int nt = L.count, n2 = L.n2;
  // room for the term records and the input vector at least (the same decision on every CTA)
  if ((long long)(nt + n2) * (long long)sizeof(ClTerm) + (long long)N * (long long)sizeof(V) > P.smem_bytes) return false;
  __syncthreads();
  ClTerm* ct = reinterpret_cast<ClTerm*>(dyn_smem);
  cl_plan<T>(P, nd, L, S, e0, e1, mmax, ct);
  const ClPlan pl = s_cl;
  if (!pl.ok) return false;
  unsigned long long* pk = reinterpret_cast<unsigned long long*>(dyn_smem + pl.pk);
  V* sm = reinterpret_cast<V*>(dyn_smem + pl.mats);
  V* xs = reinterpret_cast<V*>(dyn_smem + pl.xs);
  V* py = reinterpret_cast<V*>(dyn_smem + pl.py);
  double2* basis = reinterpret_cast<double2*>(dyn_smem + pl.basis);
  cl_stage<T>(P, ct, nt + n2, sm);
  constexpr bool kShadow = !std::is_same<T, double>::value;  // mixed modes: FP64 basis, FP32 operand
  cg::cluster_group cl = cg::this_cluster();
  auto Ks = [&](int j) -> double2* {
    return j < pl.cap ? basis + j * S : work + (long long)(j - pl.cap) * P.kvec + e0;
  };
  // element e of the input vector, written to every CTA
  auto publish = [&](int e, V v) {
    if (cs == 1) {
      xs[e] = v;
    } else {
      for (int r = 0; r < cs; ++r) cl.map_shared_rank(xs, r)[e] = v;
    }
  };
  double2* x = P.pool + nd.off;
  double s_rem = I.sign * tau / HBAR_EVFS;
  int total_m = 0, m = 0;
  for (int e = threadIdx.x; e < n_own; e += NT) {
    Ks(0)[e] = x[e0 + e];
    pk[e] = leg_pack(nd, e0 + e);
  }
  const int G = pl.G;
  const float inv_own = n_own > 0 ? 1.0f / (float)n_own : 0.0f;
  // range of all first factors, for one loop over (term, element)
  int lo1 = 0, w1 = 0;
  if (n2 > 0) {
    lo1 = N;
    int hi1 = 0;
    for (int t = nt; t < nt + n2; ++t) {
      lo1 = min(lo1, ct[t].lo);
      hi1 = max(hi1, ct[t].hi);
    }
    w1 = max(0, hi1 - lo1);
  }
  const float inv_w1 = w1 > 0 ? 1.0f / (float)w1 : 0.0f;
  __syncthreads();
  pc.lap(P.ctl, 0);
  for (int chunk = 0; chunk < 64; ++chunk) {
    double v[1] = {0.0};
    for (int e = threadIdx.x; e < n_own; e += NT) {
      const double2 a = Ks(0)[e];
      v[0] = fma(a.x, a.x, fma(a.y, a.y, v[0]));
      publish(e0 + e, cvt<T>(a));
    }
    team_reduce<1>(tm, v, [&](const double* t) { krylov_begin(ks, t[0]); }, n_own);
    pc.lap(P.ctl, 6);
    const double beta0 = ks.beta0;
    if (!(beta0 > 0.0)) {
      if (!(beta0 == 0.0)) set_status(P.ctl, ST_NONFINITE, I.op, I.node);
      break;
    }
    m = 0;
    bool conv = false;
    double nsq = v[0];  // this thread's share of |K_j|^2
    for (int j = 0; j < mmax; ++j) {
      if (n2 > 0) {
        for (int it = threadIdx.x; it < n2 * w1; it += NT) {
          const int t = fdivu(it, w1, inv_w1);
          const int e = lo1 + it - t * w1;
          const ClTerm& c = ct[nt + t];
          if (e >= c.lo && e < c.hi) xs[ct[nt - n2 + t].xo + e] = cl_term<T>(c, sm, xs, e, leg_pack(nd, e));
        }
        __syncthreads();
      }
      pc.lap(P.ctl, 1);
      if (G > 1) {
        for (int it = threadIdx.x; it < G * n_own; it += NT) {
          const int g = fdivu(it, n_own, inv_own);
          const int e = it - g * n_own;
          V a;
          a.x = a.y = (T)0;
          for (int t = g; t < nt; t += G) {
            const V b = cl_term<T>(ct[t], sm, xs, e0 + e, pk[e]);
            a.x += b.x;
            a.y += b.y;
          }
          py[g * S + e] = a;
        }
        __syncthreads();
      }
      const double sj = ks.scale[j], cm = ks.cm;
      double2* W = Ks(j + 1);
      // part[0] = Re <K_j, w>; in mixed precision also part[1] = |w|^2 and part[2] = |K_j|^2, so
      // that one team reduction gives both alpha_j and beta_{j+1}
      double part[3] = {0.0, 0.0, nsq};
      for (int e = threadIdx.x; e < n_own; e += NT) {
        V a;
        if (G > 1) {
          a = py[e];
          for (int g = 1; g < G; ++g) {
            const V b = py[g * S + e];
            a.x += b.x;
            a.y += b.y;
          }
        } else {
          a.x = a.y = (T)0;
          for (int t = 0; t < nt; ++t) {
            const V b = cl_term<T>(ct[t], sm, xs, e0 + e, pk[e]);
            a.x += b.x;
            a.y += b.y;
          }
        }
        double wr = sj * to_f64(a.x), wi = sj * to_f64(a.y);
        const double2 kj = Ks(j)[e];
        if (j > 0) {
          const double2 km = Ks(j - 1)[e];
          wr = fma(-cm, km.x, wr);
          wi = fma(-cm, km.y, wi);
        }
        part[0] = fma(kj.x, wr, fma(kj.y, wi, part[0]));
        if constexpr (kShadow) part[1] = fma(wr, wr, fma(wi, wi, part[1]));
        W[e] = make_double2(wr, wi);
      }
      if constexpr (kShadow)
        team_reduce<3>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0], t[1], t[2]); }, n_own);
      else
        team_reduce<1>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0]); }, n_own);
      pc.lap(P.ctl, 2);
      const double ca = ks.ca;  // alpha_j scale_j
      if (kShadow && ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
      double nrm[1] = {0.0};
      for (int e = threadIdx.x; e < n_own; e += NT) {
        const double2 kj = Ks(j)[e];
        double2 w = W[e];
        w.x = fma(-ca, kj.x, w.x);
        w.y = fma(-ca, kj.y, w.y);
        W[e] = w;
        if constexpr (kShadow) {
          publish(e0 + e, cvt<T>(w));  // every read of the old vector ended at the last barrier
          nrm[0] = fma(w.x, w.x, fma(w.y, w.y, nrm[0]));
        }
      }
      if constexpr (!kShadow) {
        nrm[0] = orth_slices(tm, Ks, n_own, j, ks);
        if (ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
        for (int e = threadIdx.x; e < n_own; e += NT) publish(e0 + e, cvt<T>(W[e]));
      }
      const bool fused = ks.fused != 0;
      nsq = nrm[0];
      if (fused)
        team_sync(tm);  // K_{j+1} is complete on every CTA before the next application
      else
        team_reduce<1>(tm, nrm, [&](const double* t) { krylov_norm(ks, j, t[0], s_rem, P.tol, mmax); }, n_own);
      pc.lap(P.ctl, 3);
      m = j + 1;
      if (ks.check) {
        if (threadIdx.x < 32) krylov_check(ks, m, s_rem, P.tol);
        __syncthreads();
        conv = ks.conv != 0;
        if (ks.conv == 2) set_status(P.ctl, ST_NONFINITE, I.op, I.node);
        pc.lap(P.ctl, 4);
        if (conv || m == mmax) break;
      }
    }
    total_m += m;
    if (threadIdx.x < 32) krylov_exp(ks, m, s_rem, P.tol, !conv && m < N);
    __syncthreads();
    const double s_done = ks.s_done;
    pc.lap(P.ctl, 4);
    double ny[1] = {krylov_combine(ks, Ks, n_own, m)};
    if constexpr (kShadow) {
      // the exact exponential is unitary; FP32-class contractions leave the basis orthonormal
      // only to ~1e-7, so the norm is restored to the input's
      team_reduce<1>(tm, ny, [&](const double* t) { ks.ratio = t[0] > 0.0 ? ks.beta0 / sqrt(t[0]) : 1.0; }, n_own);
      const double ratio = ks.ratio;
      if (fabs(ratio - 1.0) < 1e-3)
        for (int e = threadIdx.x; e < n_own; e += NT) {
          const double2 y = Ks(0)[e];
          Ks(0)[e] = make_double2(y.x * ratio, y.y * ratio);
        }
    }
    __syncthreads();
    pc.lap(P.ctl, 5);
    if (conv || m >= N || s_done == s_rem) break;
    s_rem -= s_done;
    if (chunk == 63 && tm.rank == 0 && threadIdx.x == 0) {
      // 64 Krylov spaces did not cover the time step: the result is incomplete
      atomicAdd(&P.ctl->not_converged, 1ull);
      set_status(P.ctl, ST_NOT_CONVERGED, I.op, I.node);
    }
  }
  for (int e = threadIdx.x; e < n_own; e += NT) x[e0 + e] = Ks(0)[e];
  if (tm.rank == 0 && threadIdx.x == 0) {
    P.mhist[I.hist] = m;
    atomicAdd(&P.ctl->krylov_iters, (unsigned long long)total_m);
    atomicAdd(&P.ctl->applies, (unsigned long long)total_m);
    atomicAdd(&P.ctl->flops, I.flops * total_m);
  }
  team_sync(tm);
  return true;
}

