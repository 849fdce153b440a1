// Householder QR bond step, templated on its arithmetic: FP64 (TTNS_FP64) or double-single
// (the mixed modes).  Included by sweep.cu.
//
// A_v (matricised: rows = all other legs in order, columns = leg I.leg) = Q R with the
// completion rule of the oracle: null sub-columns (norm <= qr_cutoff ||M||_F) get the identity
// reflector and R_jj = 0; Q = H_0 ... H_{n-1} I[:, :n]; R_jj is made real and >= 0; R is
// rescaled to ||R||_F = ||M||_F.
//
// What bounds it: latency.  A column needs one team reduction (the dots of column j with all
// trailing columns), a chain of scalar FP64 operations and a rank-one update of a few thousand
// elements per CTA.  Hence:
//   * the reflector's scalars run on one warp, two square roots at a time, as reciprocal square
//     roots: repeated on every thread they cost more than the update (a square root on all
//     eight warps: 2500 cycles);
//   * a null column leaves the trailing matrix as it is, so after one the next reduction also
//     carries the norms of all later sub-columns and a run of null columns takes one
//     reduction instead of one each (bonds that are not filled yet are mostly null);
//   * everything after the column loop works on the active reflectors only, and Z of the
//     compact form comes from one triangular solve (below) instead of T and T V^H.
// Measured on the 800 x 40 tensors of the 8 x 60 ER tree (double-single, one 16-CTA cluster,
// early in the run): 249 us per QR before, 41 us now; FP64: 354 and 65 us.
//
// The double-single arithmetic issues FP32 operations at about 80 times this part's FP64 rate;
// it keeps every sum and product to about 2^-44 relative, far below the FP32-class error of the
// mixed modes' contractions, and the team reductions and reflectors carry both parts.  A value
// below 2^-126 (about 1.2e-38) is zero there.

struct QrF64 {
  using E = double2;  // complex element
  using S = double;
  struct Acc {
    double s;
    __device__ __forceinline__ void init(S a) { s = a; }
    __device__ __forceinline__ void mac(S x, S y) { s = fma(x, y, s); }
    __device__ __forceinline__ S val() const { return s; }
  };
  static __device__ __forceinline__ S zero() { return 0.0; }
  static __device__ __forceinline__ S one() { return 1.0; }
  static __device__ __forceinline__ S add(S a, S b) { return a + b; }
  static __device__ __forceinline__ S neg(S a) { return -a; }
  static __device__ __forceinline__ S twice(S a) { return 2.0 * a; }
  static __device__ __forceinline__ S re(E z) { return z.x; }
  static __device__ __forceinline__ S im(E z) { return z.y; }
  static __device__ __forceinline__ E c(S r, S i) { return make_double2(r, i); }
  static __device__ __forceinline__ S from(double x) { return x; }
  static __device__ __forceinline__ double to(S x) { return x; }
  static __device__ __forceinline__ E cfrom(double2 z) { return z; }
  static __device__ __forceinline__ double2 cto(E z) { return z; }
  static __device__ __forceinline__ S shfl_xor(S v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
};
struct QrDs {
  using E = float4;
  using S = float2;
  using Acc = DsAcc;
  static __device__ __forceinline__ S zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ S one() { return make_float2(1.f, 0.f); }
  static __device__ __forceinline__ S add(S a, S b) { return ds_add(a, b); }
  static __device__ __forceinline__ S neg(S a) { return ds_neg(a); }
  static __device__ __forceinline__ S twice(S a) { return make_float2(2.f * a.x, 2.f * a.y); }
  static __device__ __forceinline__ S re(E z) { return ds_re(z); }
  static __device__ __forceinline__ S im(E z) { return ds_im(z); }
  static __device__ __forceinline__ E c(S r, S i) { return ds_c(r, i); }
  static __device__ __forceinline__ S from(double x) { return ds_from(x); }
  static __device__ __forceinline__ double to(S x) { return ds_to(x); }
  static __device__ __forceinline__ E cfrom(double2 z) { return ds_cfrom(z); }
  static __device__ __forceinline__ double2 cto(E z) { return ds_cto(z); }
  static __device__ __forceinline__ S shfl_xor(S v, int o) { return shfl_xor_ds(v, o); }
};
static_assert(sizeof(double2) == sizeof(float4) && sizeof(double) == sizeof(float2), "one layout for both");

template <typename A>
__device__ __forceinline__ typename A::E q_neg(typename A::E z) { return A::c(A::neg(A::re(z)), A::neg(A::im(z))); }
// (ar, ai) += conj(v) w, += a b
template <typename A>
__device__ __forceinline__ void q_conj_mac(typename A::Acc& ar, typename A::Acc& ai, typename A::E v, typename A::E w) {
  ar.mac(A::re(v), A::re(w));
  ar.mac(A::im(v), A::im(w));
  ai.mac(A::re(v), A::im(w));
  ai.mac(A::neg(A::im(v)), A::re(w));
}
template <typename A>
__device__ __forceinline__ void q_cmac(typename A::Acc& ar, typename A::Acc& ai, typename A::E a, typename A::E b) {
  ar.mac(A::re(a), A::re(b));
  ar.mac(A::neg(A::im(a)), A::im(b));
  ai.mac(A::re(a), A::im(b));
  ai.mac(A::im(a), A::re(b));
}
// s z for a real s
template <typename A>
__device__ __forceinline__ typename A::E q_scale(typename A::S s, typename A::E z) {
  typename A::Acc r, i;
  r.init(A::zero());
  i.init(A::zero());
  r.mac(s, A::re(z));
  i.mac(s, A::im(z));
  return A::c(r.val(), i.val());
}
// warp_reduce_t for the arithmetic's scalars: lane L returns the total of value warp_reduce_vid<V>(L)
template <typename A, int V>
__device__ __forceinline__ typename A::S q_warp_reduce(typename A::S* v) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int n = V; n > 1; n >>= 1, off >>= 1) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const typename A::S send = hi ? v[i] : v[i + n / 2];
      const typename A::S keep = hi ? v[i + n / 2] : v[i];
      v[i] = A::add(keep, A::shfl_xor(send, off));
    }
  }
  typename A::S t = v[0];
#pragma unroll
  for (; off > 0; off >>= 1) t = A::add(t, A::shfl_xor(t, off));
  return t;
}

// team_reduce_vec for the arithmetic's scalars (the same protocol: callers alternate between two
// `mine` buffers; one cluster barrier per call on cluster teams)
template <typename A>
__device__ __noinline__ void q_team_reduce(Team& tm, const typename A::S* mine, typename A::S* out, int nval) {
  using S = typename A::S;
  __syncthreads();
  cg::cluster_group cl = cg::this_cluster();
  auto sum16 = [&](const S* src, int n) {  // the peers' values loaded together, then a fixed tree
    S a[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) a[r] = r < n ? *cl.map_shared_rank(src, r) : A::zero();
#pragma unroll
    for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
      for (int r = 0; r < w; ++r)
        if (r + w < 16) a[r] = A::add(a[r], a[r + w]);
    return a[0];
  };
  if (tm.kind == TEAM_CLUSTER) {
    if (tm.size > 1) {
      cl.sync();
      for (int k = threadIdx.x; k < nval; k += NT) out[k] = sum16(mine + k, tm.size);
    } else {
      for (int k = threadIdx.x; k < nval; k += NT) out[k] = mine[k];
    }
  } else {
    // per cluster first (the values split over its CTAs), then the cluster totals through global
    // memory, added by every CTA in a fixed order
    const int cs = tm.csize;
    const int crank = (int)cl.block_rank();
    const int cid = tm.rank / cs, ncl = tm.size / cs;
    S* buf = reinterpret_cast<S*>(team_partials(tm));
    cl.sync();
    for (int k = crank * NT + threadIdx.x; k < nval; k += cs * NT) buf[(long long)cid * nval + k] = sum16(mine + k, cs);
    team_sync(tm);
    for (int k = threadIdx.x; k < nval; k += NT) {
      S s = A::zero();
      for (int c = 0; c < ncl; ++c) s = A::add(s, buf[(long long)c * nval + k]);
      out[k] = s;
    }
    tm.parity ^= 1;
  }
  __syncthreads();
}

struct QRShared {
  double shat[TTNS_MAX_D];   // 1 / |v_j| (0 for an identity reflector)
  double2 rdiag[TTNS_MAX_D];
  double2 coef[TTNS_MAX_D];  // (arithmetic's element) tau_j v_j^H W[k] of the trailing columns
  double2 vhead[TTNS_MAX_D]; // (arithmetic's element) heads of the unnormalised reflectors
  double2 ph[TTNS_MAX_D];
  int act[TTNS_MAX_D];       // active columns, ascending
  int na, next;
  double tau, dropped;
  double red[NWARP];
};
__shared__ QRShared s_qs;

__device__ __forceinline__ long long qr_addr(const NodeDesc& nd, int l, long long r, int c) {
  const int st = nd.strides[l];
  const int p = fdivu((int)r, st, nd.inv_strides[l]);
  const int q = (int)r - p * st;
  return (long long)(p * nd.dims[l] * st + c * st + q);
}

// Every CTA of the team owns a contiguous chunk of rows [rb, re).
template <typename A>
__device__ __noinline__ void op_qr(const KernelParams& P, Team& tm, const Instr& I, double2* work) {
  using E = typename A::E;
  using S = typename A::S;
  using Acc = typename A::Acc;
  QRShared& qs = s_qs;
  E* const coef = reinterpret_cast<E*>(qs.coef);
  E* const vhead = reinterpret_cast<E*>(qs.vhead);
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0, tm.kind == TEAM_GRID);
  const NodeDesc nd = P.nodes[I.node];
  const int l = I.leg;
  const int n = nd.dims[l];
  const int rows = nd.size / n;
  double2* Ag = P.pool + nd.off;
  E* W = reinterpret_cast<E*>(work);  // column-major: W[c * rows + r]
  double2* Rout = P.pool + P.trees[I.tree].bond_off;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunk = (rows + tm.size - 1) / tm.size;
  const int rb = min(rows, tm.rank * chunk);
  const int re = min(rows, rb + chunk);
  const int nr = re - rb;
  const float inv_nr = nr > 0 ? 1.0f / (float)nr : 0.0f;
  // shared memory: two partial buffers and the sums (PB scalars each), the own rows of the
  // workspace (column-major, `chunk` rows per column) and Z when they fit, else global memory
  const int PB = (max(2 * n * n, 5 * n + 4) + 1) & ~1;  // (even: the buffers also hold 16-byte elements)
  S* red[2] = {reinterpret_cast<S*>(dyn_smem), reinterpret_cast<S*>(dyn_smem) + PB};
  S* redo = red[1] + PB;
  int rp = 0;
  const long long ws_off = (3LL * PB * (long long)sizeof(S) + 15) & ~15LL;
  const bool in_smem = ws_off + (long long)n * chunk * (long long)sizeof(E) <= P.smem_bytes;
  E* const Wl = in_smem ? reinterpret_cast<E*>(dyn_smem + ws_off) : W;
  const int ldw = in_smem ? chunk : rows;
  const int roff = in_smem ? rb : 0;
  auto WA = [&](int c, int r) -> E& { return Wl[(long long)c * ldw + (r - roff)]; };
  const long long g_off = (ws_off + (in_smem ? (long long)n * chunk * (long long)sizeof(E) : 0) + 15) & ~15LL;
  const bool g_smem = g_off + (long long)n * n * (long long)sizeof(E) <= P.smem_bytes;
  E* Z = g_smem ? reinterpret_cast<E*>(dyn_smem + g_off)
                : reinterpret_cast<E*>(P.cta_scratch + (long long)blockIdx.x * P.cta_scratch_stride);
  for (int c = threadIdx.x; c < n; c += NT) {
    qs.shat[c] = 0.0;
    qs.rdiag[c] = make_double2(0.0, 0.0);
  }
  // copy into the workspace; the Frobenius norm sets the null threshold
  Acc fro;
  fro.init(A::zero());
  for (int idx0 = threadIdx.x; idx0 < n * nr; idx0 += 4 * NT) {  // four loads in flight per thread
    double2 g[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = min(idx0 + u * NT, n * nr - 1);
      const int c = fdivu(idx, nr, inv_nr);
      g[u] = Ag[qr_addr(nd, l, rb + (idx - c * nr), c)];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = idx0 + u * NT;
      if (idx >= n * nr) break;
      const int c = fdivu(idx, nr, inv_nr);
      const E a = A::cfrom(g[u]);
      WA(c, rb + (idx - c * nr)) = a;
      fro.mac(A::re(a), A::re(a));
      fro.mac(A::im(a), A::im(a));
    }
  }
  __syncthreads();
  // This CTA's partials for column jj over its rows r > jj, for the columns c = jj .. n - 1:
  //   slots 4 (c - jj) + {0, 1}: d_c = sum_r conj(W[jj][r]) W[c][r];  {2, 3}: h_c = W[c][jj];
  // with `look` also slot 4 (n - jj) + (c - jj), c > jj: sum_{r >= c} |W[c][r]|^2
  auto prepare = [&](int jj, bool look, S* mine) {
    const int nc = n - jj;
    const int r1 = max(rb, jj + 1);
    S* nu = mine + 4 * nc;
    if (chunk <= 32) {
      // a group of R2 lanes per column, one row per lane
      const int lg = chunk <= 1 ? 0 : 32 - __clz(chunk - 1);
      const int R2 = 1 << lg;
      for (int it0 = 0; it0 < nc * R2; it0 += NT) {
        const int it = it0 + threadIdx.x;
        const int c = it >> lg, r = rb + (it & (R2 - 1));
        S dr = A::zero(), di = A::zero(), nn = A::zero();
        if (c < nc && r < re) {
          const E w = WA(jj + c, r);
          if (r > jj) {
            Acc ar, ai;
            ar.init(A::zero());
            ai.init(A::zero());
            q_conj_mac<A>(ar, ai, WA(jj, r), w);
            dr = ar.val();
            di = ai.val();
          }
          if (look && r >= jj + c) {
            Acc a2;
            a2.init(A::zero());
            a2.mac(A::re(w), A::re(w));
            a2.mac(A::im(w), A::im(w));
            nn = a2.val();
          }
        }
        for (int o = R2 >> 1; o > 0; o >>= 1) {
          dr = A::add(dr, A::shfl_xor(dr, o));
          di = A::add(di, A::shfl_xor(di, o));
          if (look) nn = A::add(nn, A::shfl_xor(nn, o));
        }
        if (c < nc && (it & (R2 - 1)) == 0) {
          mine[4 * c] = dr;
          mine[4 * c + 1] = di;
          if (look) nu[c] = nn;
        }
      }
    } else {
      for (int c0 = 0; c0 < nc; c0 += 4 * NWARP) {  // four columns per warp, lanes over the rows
        Acc acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q].init(A::zero());
        for (int r = r1 + lane; r < re; r += 32) {
          const E vr = WA(jj, r);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = c0 + warp + q * NWARP;
            if (c < nc) q_conj_mac<A>(acc[2 * q], acc[2 * q + 1], vr, WA(jj + c, r));
          }
        }
        S v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = acc[q].val();
        const S t = q_warp_reduce<A, 8>(v);
        if ((lane & 3) == 0) {
          const int vid = warp_reduce_vid<8>(lane);
          const int c = c0 + warp + (vid >> 1) * NWARP;
          if (c < nc) mine[4 * c + (vid & 1)] = t;
        }
        if (look) {
          Acc a2[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) a2[q].init(A::zero());
          for (int r = r1 + lane; r < re; r += 32) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int c = c0 + warp + q * NWARP;
              if (c < nc && r >= jj + c) {
                const E w = WA(jj + c, r);
                a2[q].mac(A::re(w), A::re(w));
                a2[q].mac(A::im(w), A::im(w));
              }
            }
          }
          S u[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) u[q] = a2[q].val();
          const S t2 = q_warp_reduce<A, 4>(u);
          if ((lane & 7) == 0) {
            const int c = c0 + warp + warp_reduce_vid<4>(lane) * NWARP;
            if (c < nc) nu[c] = t2;
          }
        }
      }
    }
    const bool own_row = rb <= jj && jj < re;
    for (int c = threadIdx.x; c < nc; c += NT) {
      const E h = own_row ? WA(jj + c, jj) : A::c(A::zero(), A::zero());
      mine[4 * c + 2] = A::re(h);
      mine[4 * c + 3] = A::im(h);
    }
  };
  {
    S* mine = red[rp];
    rp ^= 1;
    prepare(0, false, mine);
    // the Frobenius norm rides along in the first reduction
    S f = fro.val();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f = A::add(f, A::shfl_xor(f, o));
    S* s_fro = reinterpret_cast<S*>(qs.red);
    if (lane == 0) s_fro[warp] = f;
    __syncthreads();
    if (threadIdx.x == 0) {
      S sum = s_fro[0];
      for (int w = 1; w < NWARP; ++w) sum = A::add(sum, s_fro[w]);
      mine[4 * n] = sum;
      qs.na = 0;
      qs.dropped = 0.0;
    }
    q_team_reduce<A>(tm, mine, redo, 4 * n + 1);
  }
  pc.lap(P.ctl, 8);
  const double fro2 = fmax(A::to(redo[4 * n]), 0.0);  // ||M||_F^2 (redo is reused by the column loop)
  const double thr2 = P.qr_cutoff * P.qr_cutoff * fro2;
  bool look = false;
  for (int j = 0; j < n;) {
    const int nk = n - j - 1;
    // reflector of column j: alpha = -phase(x0) sigma, vh = x0 - alpha = x0 (1 + sigma / |x0|),
    // |vh| = |x0| + sigma, |v|^2 = d_j + |vh|^2, tau = 2 / |v|^2; a head below 1e-145 counts as
    // zero (phase 1; the phase of R_jj is taken out at the end)
    if (warp == 0) {
      const double2 x0 = make_double2(A::to(redo[2]), A::to(redo[3]));
      const double dj = fmax(A::to(redo[0]), 0.0);
      const double ax2 = fma(x0.x, x0.x, x0.y * x0.y);
      const double s2 = ax2 + dj;
      int next = j + 1;
      double drop = s2;  // weight that the null columns leave out of R
      const bool null = !(s2 > thr2);
      if (!null) {
        const double y = rsqrt((lane & 1) ? ax2 : s2);
        const double ys = __shfl_sync(0xffffffffu, y, 0), ya = __shfl_sync(0xffffffffu, y, 1);
        double sigma = s2 * ys;
        sigma = fma(fma(-sigma, sigma, s2), 0.5 * ys, sigma);
        const bool head = ax2 > 1e-290;
        const double f = head ? sigma * ya : 0.0;
        const double hv = head ? fma(ax2, ya, sigma) : sigma;
        const double shat = rsqrt(fma(hv, hv, dj));
        const double2 alpha = head ? make_double2(-f * x0.x, -f * x0.y) : make_double2(-sigma, 0.0);
        const double2 vh = head ? make_double2(fma(f, x0.x, x0.x), fma(f, x0.y, x0.y)) : make_double2(sigma, 0.0);
        if (lane == 0) {
          qs.tau = 2.0 * shat * shat;
          qs.shat[j] = shat;
          qs.rdiag[j] = alpha;
          vhead[j] = A::cfrom(vh);
          qs.act[qs.na] = j;
          qs.na += 1;
        }
      } else if (look) {
        // the first later sub-column above the threshold (norms of this reduction)
        next = n;
        for (int c0 = 1; c0 <= nk; c0 += 32) {
          const int c = c0 + lane;
          const unsigned b = __ballot_sync(0xffffffffu, c <= nk && A::to(redo[4 * (n - j) + min(c, nk)]) > thr2);
          if (b) {
            next = j + c0 + __ffs(b) - 1;
            break;
          }
        }
        double v = 0.0;
        for (int c = 1 + lane; c < next - j; c += 32) v += A::to(redo[4 * (n - j) + c]);
        drop += warp_sum(v);
      }
      if (lane == 0) {
        qs.next = null ? -next : next;
        if (null) qs.dropped += drop;
      }
    }
    __syncthreads();
    const bool null = qs.next < 0;
    const int next = null ? -qs.next : qs.next;
    if (!null && nk > 0) {
      // c_k = tau (d_k + conj(vh) h_k) for the trailing columns
      const E vh = vhead[j];
      const S tau = A::from(qs.tau);
      for (int k = threadIdx.x; k < nk; k += NT) {
        const int sl = 4 * (k + 1);
        Acc ar, ai;
        ar.init(redo[sl]);
        ai.init(redo[sl + 1]);
        q_conj_mac<A>(ar, ai, vh, A::c(redo[sl + 2], redo[sl + 3]));
        coef[k] = q_scale<A>(tau, A::c(ar.val(), ai.val()));
      }
      __syncthreads();
      pc.lap(P.ctl, 13);
      // W[k] -= v c_k on the own rows r >= j, four elements per thread in flight
      const int r0 = max(rb, j);
      const int nrr = max(0, re - r0);
      const float inv_nrr = nrr > 0 ? 1.0f / (float)nrr : 0.0f;
      const int tot = nk * nrr;
      for (int idx0 = threadIdx.x; idx0 < tot; idx0 += 4 * NT) {
        E w[4], vr[4], ck[4];
        E* wp[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int idx = min(idx0 + u * NT, tot - 1);  // clamped: a duplicate is not stored
          const int k = fdivu(idx, nrr, inv_nrr);
          const int r = r0 + (idx - k * nrr);
          vr[u] = (r == j) ? vh : WA(j, r);
          ck[u] = coef[k];
          wp[u] = &WA(j + 1 + k, r);
          w[u] = *wp[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (idx0 + u * NT < tot) {
            Acc ar, ai;
            ar.init(A::re(w[u]));
            ai.init(A::im(w[u]));
            q_cmac<A>(ar, ai, q_neg<A>(vr[u]), ck[u]);
            *wp[u] = A::c(ar.val(), ai.val());
          }
        }
      }
      __syncthreads();
      pc.lap(P.ctl, 14);
    }
    look = null;
    j = next;
    if (j < n) {
      S* mine = red[rp];
      rp ^= 1;
      prepare(j, look, mine);
      pc.lap(P.ctl, 15);
      q_team_reduce<A>(tm, mine, redo, (look ? 5 : 4) * (n - j));
      pc.lap(P.ctl, 9);
    }
  }
  __syncthreads();
  if (in_smem) {  // rows < n to the global workspace (read across CTAs below)
    const int ntop = max(0, min(re, n) - rb);
    for (int idx = threadIdx.x; idx < n * ntop; idx += NT) {
      const int c = idx / ntop;
      const int r = rb + (idx - c * ntop);
      W[(long long)c * rows + r] = WA(c, r);
    }
  }
  pc.lap(P.ctl, 9);
  // Compact form Q = I - Vh T Vh^H of the active unit reflectors vh_a = v_a / |v_a| (a column
  // just above the null threshold has |v| far below |M| and tau far above 1; the unnormalised
  // form would chain such factors and lose orthogonality).  T^{-1} is the strictly upper Gram
  // matrix G plus 1/2 on the diagonal, so Z = T Vh^H[:, :n] solves, from the last row up,
  //   Z_a = 2 (Vh^H)_a - sum_{b > a} 2 G_ab Z_b,
  // by right-looking updates of all earlier rows (independent elements, no dot products).
  const int na = qs.na;
  const int npair = na * (na - 1) / 2;  // pairs a < b, p = b (b - 1) / 2 + a
  {
    S* mine = red[rp];
    rp ^= 1;
    int lg = 0;  // lanes per pair: enough threads when the pairs are few
    while (lg < 5 && (npair << (lg + 1)) <= 2 * NT) ++lg;
    const int g = 1 << lg;
    for (int it0 = 0; it0 < (npair << lg); it0 += NT) {
      const int it = it0 + threadIdx.x;
      const int p = it >> lg;
      const bool on = p < npair;
      Acc g0r, g0i, g1r, g1i;
      g0r.init(A::zero());
      g0i.init(A::zero());
      g1r.init(A::zero());
      g1i.init(A::zero());
      if (on) {
        int b = (int)((1.0f + sqrtf(8.0f * (float)p + 1.0f)) * 0.5f);
        while (b * (b + 1) / 2 <= p) ++b;
        while (b * (b - 1) / 2 > p) --b;
        const int ja = qs.act[p - b * (b - 1) / 2], jb = qs.act[b];
        int r = max(rb, jb) + (it & (g - 1));
        for (; r + g < re; r += 2 * g) {  // r > ja always: a < b
          q_conj_mac<A>(g0r, g0i, WA(ja, r), r == jb ? vhead[jb] : WA(jb, r));
          q_conj_mac<A>(g1r, g1i, WA(ja, r + g), WA(jb, r + g));
        }
        if (r < re) q_conj_mac<A>(g0r, g0i, WA(ja, r), r == jb ? vhead[jb] : WA(jb, r));
      }
      S sr = A::add(g0r.val(), g1r.val()), si = A::add(g0i.val(), g1i.val());
      for (int o = g >> 1; o > 0; o >>= 1) {
        sr = A::add(sr, A::shfl_xor(sr, o));
        si = A::add(si, A::shfl_xor(si, o));
      }
      if (on && (it & (g - 1)) == 0) {
        mine[2 * p] = sr;
        mine[2 * p + 1] = si;
      }
    }
    // (also the barrier after which the top rows of the workspace are read)
    q_team_reduce<A>(tm, mine, redo, 2 * npair);
  }
  pc.lap(P.ctl, 10);
  // G2[p] = -2 shat_a shat_b (sum), Z_a = 2 shat_a conj(V[c][a]); then the solve
  E* G2 = reinterpret_cast<E*>(red[rp]);  // released by the reduction's barrier; npair <= n^2 / 2
  for (int p = threadIdx.x; p < npair; p += NT) {
    int b = (int)((1.0f + sqrtf(8.0f * (float)p + 1.0f)) * 0.5f);
    while (b * (b + 1) / 2 <= p) ++b;
    while (b * (b - 1) / 2 > p) --b;
    const double s = -2.0 * qs.shat[qs.act[p - b * (b - 1) / 2]] * qs.shat[qs.act[b]];
    G2[p] = q_scale<A>(A::from(s), A::c(redo[2 * p], redo[2 * p + 1]));
  }
  for (int idx = threadIdx.x; idx < na * n; idx += NT) {
    const int a = idx / n, c = idx - a * n;
    const int ja = qs.act[a];
    E z = A::c(A::zero(), A::zero());
    if (c >= ja) {
      const E v = c == ja ? vhead[ja] : W[(long long)ja * rows + c];
      z = q_scale<A>(A::from(2.0 * qs.shat[ja]), A::c(A::re(v), A::neg(A::im(v))));
    }
    Z[idx] = z;
  }
  __syncthreads();
  for (int b = na - 1; b > 0; --b) {
    const int jb = qs.act[b], w = n - jb;  // Z_b is zero before column jb
    const float inv_w = 1.0f / (float)w;
    for (int idx = threadIdx.x; idx < b * w; idx += NT) {
      const int a = fdivu(idx, w, inv_w);
      const int c = jb + idx - a * w;
      Acc zr, zi;
      const E z = Z[a * n + c];
      zr.init(A::re(z));
      zi.init(A::im(z));
      q_cmac<A>(zr, zi, G2[b * (b - 1) / 2 + a], Z[b * n + c]);
      Z[a * n + c] = A::c(zr.val(), zi.val());
    }
    __syncthreads();
  }
  // Q = I - V Z with the unnormalised V of the workspace
  for (int idx = threadIdx.x; idx < na * n; idx += NT) {
    const int ja = qs.act[idx / n];
    Z[idx] = q_scale<A>(A::from(qs.shat[ja]), Z[idx]);
  }
  // phases of the diagonal of R
  for (int j = threadIdx.x; j < n; j += NT) {
    const double2 a = qs.rdiag[j];
    const double a2 = fma(a.x, a.x, a.y * a.y);
    const double y = a2 > 0.0 ? rsqrt(a2) : 0.0;
    qs.ph[j] = a2 > 0.0 ? make_double2(a.x * y, a.y * y) : make_double2(1.0, 0.0);
  }
  if (threadIdx.x == NT - 32) {
    const double rn2 = fro2 - qs.dropped;
    qs.tau = rn2 > 0.0 ? sqrt(fro2 / rn2) : 1.0;
  }
  __syncthreads();
  pc.lap(P.ctl, 11);
  // R (row j scaled by conj(ph_j)) into the bond buffer: R[j][k] = W[k][j] (k > j), diag alpha_j,
  // rescaled to ||R||_F = ||M||_F (the weight of dropped sub-columns returns to the kept content).
  // The reflectors keep every column's norm, so ||R||_F^2 = ||M||_F^2 - the dropped weight; the
  // entries are spread over the team (one CTA took 6 us for them, most of it FP64 instructions)
  for (int idx = tm.gtid(); idx < n * n; idx += tm.nthr()) {
    const int j = idx / n, k = idx % n;
    double2 r = make_double2(0, 0);
    if (k > j) r = A::cto(W[(long long)k * rows + j]);
    else if (k == j) r = qs.rdiag[j];
    const double2 p = qs.ph[j];
    const double scale = qs.tau;
    Rout[idx] = make_double2(scale * (r.x * p.x + r.y * p.y), scale * (r.y * p.x - r.x * p.y));
  }
  // Q[r][c] = (delta_rc - sum_a V[r][a] Z[a][c]) ph_c over the own rows, active columns a with
  // j_a <= min(r, c); a thread takes the columns c0 and c0 + 1 of one row (V loaded once)
  const int ncp = (n + 1) / 2;
  for (int idx = threadIdx.x; idx < ncp * nr; idx += NT) {
    const int cp = fdivu(idx, nr, inv_nr);
    const int r = rb + (idx - cp * nr);
    const int c0 = 2 * cp, c1 = min(c0 + 1, n - 1);
    const int jmax = min(r, c1);
    Acc q0r, q0i, q1r, q1i;
    q0r.init(r == c0 ? A::one() : A::zero());
    q0i.init(A::zero());
    q1r.init(r == c1 ? A::one() : A::zero());
    q1i.init(A::zero());
    for (int a = 0; a < na; ++a) {
      const int ja = qs.act[a];
      if (ja > jmax) break;
      const E nv = q_neg<A>((r == ja) ? vhead[ja] : WA(ja, r));
      q_cmac<A>(q0r, q0i, nv, Z[a * n + c0]);
      q_cmac<A>(q1r, q1i, nv, Z[a * n + c1]);
    }
    auto put = [&](int c, S qr, S qi) {
      E v = A::c(qr, qi);
      if (qs.shat[c] != 0.0) {  // an active column: times its phase (1 otherwise)
        Acc o_r, o_i;
        o_r.init(A::zero());
        o_i.init(A::zero());
        q_cmac<A>(o_r, o_i, v, A::cfrom(qs.ph[c]));
        v = A::c(o_r.val(), o_i.val());
      }
      const long long at = qr_addr(nd, l, r, c);
      Ag[at] = A::cto(v);
      // the mixed modes' environment updates read Q from the FP32 mirror (the heads of v)
      if constexpr (std::is_same<A, QrDs>::value) P.pool32[nd.off + at] = make_float2(A::re(v).x, A::im(v).x);
    };
    put(c0, q0r.val(), q0i.val());
    if (c1 > c0) put(c1, q1r.val(), q1i.val());
  }
  team_sync(tm);
  pc.lap(P.ctl, 12);
}
