// Krylov exponential and environment update of "site" tensors (included by sweep.cu): two or
// three legs, every dense factor on a leg A or C, every row-sparse factor on the remaining leg P
// (a chain site: parent and child bonds, and the Fock leg with its ladder operators; the root of
// a single chain).  Both work slice by slice: a slice is the tensor at one index of P, and a term
// is a dense product inside a slice followed by the few entries that the sparse factor has per
// row.  A CTA owns the rows [a0, a1) of A, all of C, for a range of P indices; the team's CTAs
// cover the tensor.
//
// Why: the products are D x D matrices times slices of D x D (D <= 64), a few hundred
// kFLOP per CTA, so their time is operand traffic and latency.  The element-wise form read two
// shared-memory words per multiply-add and walked through one term after another; here a thread
// forms a 2 x 2 tile of one (term, slice) product, and the tensor-core form's operand splitting and
// layout (20 us of every 35 us application on 40 x 40 x 20 tensors) has nothing to amortise it.
// The Krylov vectors' own parts stay in shared memory as far as they fit; an updated vector goes
// to the CTAs that read its slices, through distributed shared memory (cluster teams) or a
// slice-major copy in global memory (the grid team).
// Forward exponential of a 40 x 40 x 20 tensor, whole grid, about four applications: 190 us per
// operation before, 103 now (BF16X3 mode); FP64, about eight applications: 1500 and 660.
//
// The plan (legs, jobs, split, layout: SitePlan) comes from the host: worked out by one thread of
// every CTA it took 6 us per operation.

__device__ __forceinline__ int site_slot(unsigned long long need, int s) { return __popcll(need & ((1ull << s) - 1ull)); }

// One CTA's part: unit = rank; ranks beyond the units own nothing.
struct SiteUnit {
  int a0, A, s0, S;   // rows and P indices
  int n;              // own elements, index o = (s_l * A + a_l) * Dc + c
  int off;            // position of the own elements in a unit-ordered vector of N elements
  int nsl;
  unsigned long long need;
  float inv_ac, inv_c;
};
__device__ __forceinline__ SiteUnit site_unit(const SitePlan& sp, int rank) {
  SiteUnit u;
  const int sbi = rank % sp.ns, ai = rank / sp.ns;
  const bool on = ai < sp.na;
  u.s0 = sbi * sp.sb;
  u.S = min(sp.sb, sp.dp - u.s0);
  u.a0 = on ? ai * sp.Ab : 0;
  u.A = on ? min(sp.Ab, sp.Da - u.a0) : 0;
  u.n = u.A * sp.Dc * u.S;
  u.off = (u.s0 * sp.Da + u.a0 * u.S) * sp.Dc;
  u.need = on ? sp.need[sbi] : 0ull;
  u.nsl = __popcll(u.need);
  u.inv_ac = u.A > 0 ? 1.0f / (float)(u.A * sp.Dc) : 0.0f;
  u.inv_c = 1.0f / (float)sp.Dc;
  return u;
}
struct SiteAt {
  int s, a, c;  // P index, A row, C index
};
__device__ __forceinline__ SiteAt site_at(const SitePlan& sp, const SiteUnit& u, int o) {
  const int sl = fdivu(o, u.A * sp.Dc, u.inv_ac);
  const int r = o - sl * u.A * sp.Dc;
  const int al = fdivu(r, sp.Dc, u.inv_c);
  return SiteAt{u.s0 + sl, u.a0 + al, r - al * sp.Dc};
}
// The plan into shared memory, and the unit's tables: value of every job at every P index, and
// the position in xs of the slice that it reads (own P indices only).  Ends with a block barrier.
template <typename T>
__device__ __forceinline__ SiteUnit site_begin(const KernelParams& P, const Team& tm, const Instr& I) {
  using V = typename C2<T>::t;
  SitePlan& sp = *reinterpret_cast<SitePlan*>(dyn_smem);
  const int4* g = reinterpret_cast<const int4*>(P.sites + I.site);
  static_assert(sizeof(SitePlan) % 16 == 0, "plans are copied 16 bytes at a time");
  __syncthreads();
  for (int k = threadIdx.x; k < (int)(sizeof(SitePlan) / 16); k += NT) reinterpret_cast<int4*>(dyn_smem)[k] = g[k];
  __syncthreads();
  const SiteUnit u = site_unit(sp, tm.rank);
  V* vals = reinterpret_cast<V*>(dyn_smem + sp.vals);
  int* cols = reinterpret_cast<int*>(dyn_smem + sp.cols);
  const V* src = ops<T>(P) + I.rega_off;
  for (int it = threadIdx.x; it < sp.nj * u.S; it += NT) {
    const int j = it / u.S, s = u.s0 + it - j * u.S;
    const SiteJob& jb = sp.job[j];
    V v;
    v.x = (T)1;
    v.y = (T)0;
    int col = s;
    if (jb.nnz > 0) {
      v = src[jb.sp + (long long)s * jb.nnz + jb.q];
      col = (int)src[jb.sp + (long long)sp.dp * jb.nnz + (long long)s * jb.nnz + jb.q].x;
    }
    vals[j * sp.dp + s] = v;
    cols[j * sp.dp + s] = site_slot(u.need, col) * sp.Da * sp.Cp;
  }
  return u;
}

// Staged matrices: the own rows of an A matrix, a C matrix transposed (k-major, so that
// consecutive outputs are contiguous).  The caller waits for the copies.
template <typename T>
__device__ void site_stage(const KernelParams& P, const Instr& I, const SitePlan& sp, const SiteUnit& u) {
  using V = typename C2<T>::t;
  V* sm = reinterpret_cast<V*>(dyn_smem + sp.mats);
  const V* src = ops<T>(P) + I.rega_off;
  const int Cq = sp.Dc + (sp.Dc & 1);
  auto cp = [&](V* d, const V* s) {
    if constexpr (sizeof(V) == 16)
      cp_async16(d, s);
    else
      cp_async8(d, s);
  };
  for (int j = 0; j < sp.nd; ++j) {
    const SiteJob jb = sp.job[j];
    if (jb.q > 0) continue;
    V* d = sm + jb.moff;
    if (jb.type == 0) {
      const V* s = src + jb.mat + (long long)u.a0 * sp.Da;
      for (int k = threadIdx.x; k < u.A * sp.Da; k += NT) cp(d + k, s + k);
    } else {
      const V* s = src + jb.mat;
      const float inv = 1.0f / (float)sp.Dc;
      for (int k = threadIdx.x; k < sp.Dc * sp.Dc; k += NT) {
        const int i = fdivu(k, sp.Dc, inv), kk = k - i * sp.Dc;
        cp(d + kk * Cq + i, s + k);
      }
    }
  }
}

// two adjacent values (16-byte aligned for floats)
__device__ __forceinline__ void ld_pair(const float2* p, float2& a, float2& b) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld_pair(const double2* p, double2& a, double2& b) {
  a = p[0];
  b = p[1];
}

// Dense jobs on the own rows and P indices: results v * (dense product at the job's
// column) to dbuf[job * stride + o], a TA x TC tile per thread.  xs: slices [slot][a][c], rows of
// Cp.
template <typename T, int TA, int TC>
__device__ __noinline__ void site_tiles(const SitePlan& sp, const SiteUnit& u, const typename C2<T>::t* xs,
                                        typename C2<T>::t* dbuf, int stride) {
  using V = typename C2<T>::t;
  const V* sm = reinterpret_cast<const V*>(dyn_smem + sp.mats);
  const V* vals = reinterpret_cast<const V*>(dyn_smem + sp.vals);
  const int* cols = reinterpret_cast<const int*>(dyn_smem + sp.cols);
  const int na2 = (u.A + TA - 1) / TA, nc2 = (sp.Dc + TC - 1) / TC, Cq = sp.Dc + (sp.Dc & 1);
  const int tiles = na2 * nc2;
  const float inv_t = tiles > 0 ? 1.0f / (float)tiles : 0.0f, inv_c2 = 1.0f / (float)nc2;
  const float inv_S = u.S > 0 ? 1.0f / (float)u.S : 0.0f;
  const int total = sp.nd * u.S * tiles;
  for (int it = threadIdx.x; it < total; it += NT) {
    const int js = fdivu(it, tiles, inv_t), r = it - js * tiles;
    const int j = fdivu(js, u.S, inv_S), sl = js - j * u.S;
    const int at = fdivu(r, nc2, inv_c2);
    const int al0 = TA * at, al1 = min(al0 + 1, u.A - 1), c0 = TC * (r - at * nc2);
    const V w = vals[j * sp.dp + u.s0 + sl];
    V x[TA][TC];
#pragma unroll
    for (int i = 0; i < TA; ++i)
#pragma unroll
      for (int q = 0; q < TC; ++q) x[i][q].x = x[i][q].y = (T)0;
    const SiteJob& jb = sp.job[j];
    if (w.x != (T)0 || w.y != (T)0) {
      const V* slice = xs + cols[j * sp.dp + u.s0 + sl];
      const V *p0, *b;
      int ps, bs;  // the second row's distance, and b's row length
      if (jb.type == 0) {
        p0 = sm + jb.moff + al0 * sp.Da;
        ps = sp.Da;
        b = slice + c0;
        bs = sp.Cp;
      } else {
        b = sm + jb.moff + c0;
        bs = Cq;
        p0 = slice + (u.a0 + al0) * sp.Cp;
        ps = sp.Cp;
      }
      const V* p1 = p0 + (al1 - al0) * ps;
      const int K = jb.K;
      constexpr int U = std::is_same<T, double>::value ? 1 : 4;
      V acc[TA][TC][U];
#pragma unroll
      for (int i = 0; i < TA; ++i)
#pragma unroll
        for (int e = 0; e < TC; ++e)
#pragma unroll
          for (int u4 = 0; u4 < U; ++u4) acc[i][e][u4].x = acc[i][e][u4].y = (T)0;
      auto step = [&](int k, int u4) {
        V q[TA], g[TC];
        q[0] = p0[k];
        if (TA > 1) q[TA - 1] = p1[k];
        if constexpr (TC > 1)
          ld_pair(b + k * bs, g[0], g[TC - 1]);
        else
          g[0] = b[k * bs];
#pragma unroll
        for (int i = 0; i < TA; ++i)
#pragma unroll
          for (int e = 0; e < TC; ++e) cmac<T>(acc[i][e][u4], q[i], g[e]);
      };
      int k = 0;
      for (; k + 3 < K; k += 4) {
#pragma unroll
        for (int u4 = 0; u4 < 4; ++u4) step(k + u4, u4 % U);
      }
      for (; k < K; ++k) step(k, 0);
#pragma unroll
      for (int i = 0; i < TA; ++i)
#pragma unroll
        for (int e = 0; e < TC; ++e) x[i][e] = sum_parts<U>(acc[i][e]);
      if (jb.nnz > 0) {
#pragma unroll
        for (int i = 0; i < TA; ++i)
#pragma unroll
          for (int e = 0; e < TC; ++e) {
            V y;
            y.x = w.x * x[i][e].x - w.y * x[i][e].y;
            y.y = w.x * x[i][e].y + w.y * x[i][e].x;
            x[i][e] = y;
          }
      }
    }
    V* o = dbuf + j * stride + (sl * u.A + al0) * sp.Dc + c0;
#pragma unroll
    for (int i = 0; i < TA; ++i)
#pragma unroll
      for (int e = 0; e < TC; ++e)
        if (al0 + i < u.A && c0 + e < sp.Dc) o[i * sp.Dc + e] = x[i][e];
  }
}
// The tile: in FP32 2 x 2 (its operand loads are the bound) unless that leaves threads without
// work, then 1 x 2 or single elements; in FP64 single elements (the FP64 pipe is the bound, and
// tiles over odd edges waste it).
template <typename T>
__device__ __forceinline__ void site_products(const SitePlan& sp, const SiteUnit& u, const typename C2<T>::t* xs,
                                              typename C2<T>::t* dbuf, int stride) {
  if constexpr (std::is_same<T, double>::value) {
    site_tiles<T, 1, 1>(sp, u, xs, dbuf, stride);
  } else {
    const int rows = sp.nd * u.S, nc2 = (sp.Dc + 1) / 2;
    if (rows * ((u.A + 1) / 2) * nc2 >= NT)
      site_tiles<T, 2, 2>(sp, u, xs, dbuf, stride);
    else if (rows * u.A * nc2 >= NT)
      site_tiles<T, 1, 2>(sp, u, xs, dbuf, stride);
    else
      site_tiles<T, 1, 1>(sp, u, xs, dbuf, stride);
  }
}
// Sum of block blk's jobs at own element o: dense results and sparse-only terms
template <typename T>
__device__ __forceinline__ typename C2<T>::t site_sum(const SitePlan& sp, const typename C2<T>::t* xs,
                                                      const typename C2<T>::t* dbuf, int stride, int o,
                                                      const SiteAt& at, int blk) {
  using V = typename C2<T>::t;
  const V* vals = reinterpret_cast<const V*>(dyn_smem + sp.vals) + at.s;
  const int* cols = reinterpret_cast<const int*>(dyn_smem + sp.cols) + at.s;
  V y;
  y.x = y.y = (T)0;
#pragma unroll 4
  for (int j = 0; j < sp.nd; ++j) {
    if (sp.job[j].blk != blk) continue;
    const V d = dbuf[j * stride + o];
    y.x += d.x;
    y.y += d.y;
  }
  const int row = at.a * sp.Cp + at.c;
  for (int j = sp.nd; j < sp.nj; ++j)
    if (sp.job[j].blk == blk) {
      const V w = vals[j * sp.dp];
      if (w.x != (T)0 || w.y != (T)0) cmac<T>(y, w, xs[cols[j * sp.dp] + row]);
    }
  return y;
}

template <typename T>
__device__ __noinline__ bool op_expm_site(const KernelParams& P, Team& tm, const Instr& I, double2* work, double tau) {
  using V = typename C2<T>::t;
  KrylovShared& ks = s_ks;
  if (I.site < 0) return false;
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0, tm.kind == TEAM_GRID);
  const long long node_off = P.nodes[I.node].off;
  const SiteUnit u = site_begin<T>(P, tm, I);
  const SitePlan& sp = *reinterpret_cast<const SitePlan*>(dyn_smem);
  const int N = sp.Da * sp.Dc * sp.dp;
  const bool grid = tm.kind == TEAM_GRID;
  const int T_ = tm.size;
  const int mmax = min(P.mmax, min(N, TTNS_KMAX));
  constexpr bool kShadow = !std::is_same<T, double>::value;  // mixed modes: FP64 basis, FP32 operand
  const int S_max = sp.Ab * sp.Dc * sp.sb;
  V* xs = reinterpret_cast<V*>(dyn_smem + sp.xs);
  V* dbuf = reinterpret_cast<V*>(dyn_smem + sp.dbuf);
  double2* basis = reinterpret_cast<double2*>(dyn_smem + sp.rest);
  const int cap = (int)min((long long)mmax + 1, (P.smem_bytes - sp.rest) / ((long long)S_max * (long long)sizeof(double2)));
  site_stage<T>(P, I, sp, u);
  cg::cluster_group cl = cg::this_cluster();
  auto Ks = [&](int j) -> double2* {
    return j < cap ? basis + (long long)j * S_max : work + (long long)(j - cap) * P.kvec + u.off;
  };
  // the grid team's copy of the input vector: slice-major, rows of Cp (behind the Krylov slots)
  V* xg = reinterpret_cast<V*>(work + (long long)(P.mmax + P.n_tmp) * P.kvec);
  auto publish = [&](const SiteAt& at, V v) {
    if (grid) {
      xg[(at.s * sp.Da + at.a) * sp.Cp + at.c] = v;
    } else if (T_ == 1) {
      xs[(site_slot(u.need, at.s) * sp.Da + at.a) * sp.Cp + at.c] = v;
    } else {
      const int row = at.a * sp.Cp + at.c;
      for (int sbi = 0; sbi < sp.ns; ++sbi) {
        const unsigned long long need = sp.need[sbi];
        if (!((need >> at.s) & 1ull)) continue;
        V* dst = xs + site_slot(need, at.s) * sp.Da * sp.Cp + row;
        for (int ai = 0; ai < sp.na; ++ai) *cl.map_shared_rank(dst, sbi + ai * sp.ns) = v;
      }
    }
  };
  // grid team: the slices that this unit reads, after the barrier that completes the vector
  auto gather = [&]() {
    if (!grid) return;
    const int len = sp.Da * sp.Cp;  // an even number of elements: 16-byte copies
    unsigned long long m = u.need;
    for (int slot = 0; slot < u.nsl; ++slot) {
      const int s = __ffsll((long long)m) - 1;
      m &= m - 1;
      const V* src = xg + (long long)s * len;
      V* dst = xs + slot * len;
      const int n16 = len * (int)sizeof(V) / 16;
      for (int k = threadIdx.x; k < n16; k += NT)
        cp_async16(reinterpret_cast<char*>(dst) + 16 * k, reinterpret_cast<const char*>(src) + 16 * k);
    }
    cp_async_wait_all();
    __syncthreads();
  };
  double2* x = P.pool + node_off;
  const int sA = sp.sA, sC = sp.sC, sP = sp.sP;
  double s_rem = I.sign * tau / HBAR_EVFS;
  int total_m = 0, m = 0;
  const SiteAt at_tid = site_at(sp, u, min((int)threadIdx.x, max(u.n - 1, 0)));
  auto pos = [&](int o) { return o == (int)threadIdx.x ? at_tid : site_at(sp, u, o); };
  for (int o = threadIdx.x; o < u.n; o += NT) {
    const SiteAt at = pos(o);
    Ks(0)[o] = x[at.a * sA + at.c * sC + at.s * sP];
  }
  cp_async_wait_all();
  __syncthreads();
  pc.lap(P.ctl, 0);
  for (int chunk = 0; chunk < 64; ++chunk) {
    double v[1] = {0.0};
    for (int o = threadIdx.x; o < u.n; o += NT) {
      const double2 a = Ks(0)[o];
      v[0] = fma(a.x, a.x, fma(a.y, a.y, v[0]));
      publish(pos(o), cvt<T>(a));
    }
    team_reduce<1>(tm, v, [&](const double* t) { krylov_begin(ks, t[0]); }, u.n);
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
      gather();
      pc.lap(P.ctl, 1);
      site_products<T>(sp, u, xs, dbuf, S_max);
      __syncthreads();
      pc.lap(P.ctl, 7);
      const double sj = ks.scale[j], cm = ks.cm;
      double2* W = Ks(j + 1);
      double part[3] = {0.0, 0.0, nsq};
      for (int o = threadIdx.x; o < u.n; o += NT) {
        const V a = site_sum<T>(sp, xs, dbuf, S_max, o, pos(o), 0);
        double wr = sj * to_f64(a.x), wi = sj * to_f64(a.y);
        const double2 kj = Ks(j)[o];
        if (j > 0) {
          const double2 km = Ks(j - 1)[o];
          wr = fma(-cm, km.x, wr);
          wi = fma(-cm, km.y, wi);
        }
        part[0] = fma(kj.x, wr, fma(kj.y, wi, part[0]));
        if constexpr (kShadow) part[1] = fma(wr, wr, fma(wi, wi, part[1]));
        W[o] = make_double2(wr, wi);
      }
      if constexpr (kShadow)
        team_reduce<3>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0], t[1], t[2]); }, u.n);
      else
        team_reduce<1>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0]); }, u.n);
      pc.lap(P.ctl, 2);
      const double ca = ks.ca;  // alpha_j scale_j
      if (kShadow && ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
      double nrm[1] = {0.0};
      for (int o = threadIdx.x; o < u.n; o += NT) {
        const double2 kj = Ks(j)[o];
        double2 w = W[o];
        w.x = fma(-ca, kj.x, w.x);
        w.y = fma(-ca, kj.y, w.y);
        W[o] = w;
        if constexpr (kShadow) {
          publish(pos(o), cvt<T>(w));  // every read of the old vector ended at the last barrier
          nrm[0] = fma(w.x, w.x, fma(w.y, w.y, nrm[0]));
        }
      }
      if constexpr (!kShadow) {
        nrm[0] = orth_slices(tm, Ks, u.n, j, ks);
        if (ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
        for (int o = threadIdx.x; o < u.n; o += NT) publish(pos(o), cvt<T>(W[o]));
      }
      const bool fused = ks.fused != 0;
      nsq = nrm[0];
      if (fused)
        team_sync(tm);  // K_{j+1} is complete for every CTA before the next application
      else
        team_reduce<1>(tm, nrm, [&](const double* t) { krylov_norm(ks, j, t[0], s_rem, P.tol, mmax); }, u.n);
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
    const double ny = krylov_combine(ks, Ks, u.n, m);
    if constexpr (kShadow) {
      // the exact exponential is unitary; FP32-class contractions leave the basis orthonormal
      // only to ~1e-7, so the norm is restored to the input's
      double nv[1] = {ny};
      team_reduce<1>(tm, nv, [&](const double* t) { ks.ratio = t[0] > 0.0 ? ks.beta0 / sqrt(t[0]) : 1.0; }, u.n);
      const double ratio = ks.ratio;
      if (fabs(ratio - 1.0) < 1e-3)
        for (int o = threadIdx.x; o < u.n; o += NT) {
          const double2 y = Ks(0)[o];
          Ks(0)[o] = make_double2(y.x * ratio, y.y * ratio);
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
  for (int o = threadIdx.x; o < u.n; o += NT) {
    const SiteAt at = pos(o);
    x[at.a * sA + at.c * sC + at.s * sP] = Ks(0)[o];
  }
  if (tm.rank == 0 && threadIdx.x == 0) {
    P.mhist[I.hist] = m;
    atomicAdd(&P.ctl->krylov_iters, (unsigned long long)total_m);
    atomicAdd(&P.ctl->applies, (unsigned long long)total_m);
    atomicAdd(&P.ctl->flops, I.flops * total_m);
  }
  team_sync(tm);
  return true;
}

// env(u -> v) of a site tensor toward leg A: block 0 = Q^H (H-terms without v) Q, block 1 + b = Q^H
// (channel b) Q, over all C and P indices.  A CTA forms the results of its rows a' and P indices and
// the partial blocks E[b][a][a'] = sum_{s, c} conj(Q[a][c][s]) Y_b[a'][c][s] for all a, so a partial
// holds only D x Ab values per block and only the few CTAs of the same rows are added up.  A
// channel whose operator is the adjoint of the one before it (the two halves of a hopping term)
// takes that block's adjoint.  Sums: FP32 over one slice, then double-single (mixed modes); FP64.
template <typename T>
__device__ __noinline__ bool op_env_site(const KernelParams& P, Team& tm, const Instr& I) {
  using V = typename C2<T>::t;
  using A = typename EnvArith<T>::A;
  using E = typename A::E;
  constexpr bool kMixed = !std::is_same<T, double>::value;
  if (I.site < 0) return false;
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0, tm.kind == TEAM_GRID);
  const int nch = I.nchan, nb = 1 + nch;
  const long long node_off = P.nodes[I.node].off;
  const SiteUnit u = site_begin<T>(P, tm, I);
  const SitePlan& sp = *reinterpret_cast<const SitePlan*>(dyn_smem);
  const int S_max = sp.Ab * sp.Dc * sp.sb;
  const int Yrow = sp.Cp, Yblk = sp.sb * sp.Ab * Yrow;
  V* xs = reinterpret_cast<V*>(dyn_smem + sp.xs);
  V* dbuf = reinterpret_cast<V*>(dyn_smem + sp.dbuf);
  V* Y = dbuf + (long long)sp.nd * S_max;
  site_stage<T>(P, I, sp, u);
  {
    // slices of Q (mixed modes: from the FP32 mirror)
    const V* src = ops<T>(P) + node_off;
    const int per = sp.Da * sp.Dc;
    const float inv_per = 1.0f / (float)per;
    for (int it = threadIdx.x; it < u.nsl * per; it += NT) {
      const int slot = fdivu(it, per, inv_per), r = it - slot * per;
      const int a = fdivu(r, sp.Dc, u.inv_c), c = r - a * sp.Dc;
      unsigned long long m = u.need;
      for (int k = 0; k < slot; ++k) m &= m - 1;
      const int s = __ffsll((long long)m) - 1;
      const V* g = src + a * sp.sA + c * sp.sC + s * sp.sP;
      V* d = xs + (slot * sp.Da + a) * sp.Cp + c;
      if constexpr (sizeof(V) == 16)
        cp_async16(d, g);
      else
        cp_async8(d, g);
    }
    cp_async_wait_all();
  }
  __syncthreads();
  pc.lap(P.ctl, 16);
  site_products<T>(sp, u, xs, dbuf, S_max);
  __syncthreads();
  for (int it = threadIdx.x; it < nb * u.n; it += NT) {
    const int b = it / max(u.n, 1), o = it - b * u.n;
    if (b > 0 && ((I.adj >> (b - 1)) & 1u)) continue;
    const SiteAt at = site_at(sp, u, o);
    Y[b * Yblk + ((at.s - u.s0) * u.A + at.a - u.a0) * Yrow + at.c] = site_sum<T>(sp, xs, dbuf, S_max, o, at, b);
  }
  __syncthreads();
  pc.lap(P.ctl, 17);
  const int D = sp.Da, D2 = D * D, nval = nb * D2;
  const bool sum = sp.ns > 1;
  double2* out = P.pool + I.env_out;
  E* buf = reinterpret_cast<E*>(team_partials(tm));
  auto emit = [&](int k, E v) {
    out[k] = A::cto(v);
    if constexpr (kMixed) P.pool32[I.env_out + k] = make_float2(A::re(v).x, A::im(v).x);
  };
  auto done = [&](int b, int a, int a2, E v) {  // final value, and the adjoint channel's
    emit(b * D2 + a * D + a2, v);
    if (b > 0 && b < nch && ((I.adj >> b) & 1u)) emit((b + 1) * D2 + a2 * D + a, A::c(A::re(v), A::neg(A::im(v))));
  };
  {
    // 2 x 2 tiles (a, a'), few tiles split over up to eight lanes each along C
    const int da2 = (D + 1) / 2, ua2 = (u.A + 1) / 2, tiles = da2 * ua2;
    const int total = tiles * nb;
    int lg = 0;
    while (lg < 3 && (total << (lg + 1)) <= NT && (2 << lg) <= sp.Dc) ++lg;
    const int ksp = 1 << lg;
    const float inv_t = tiles > 0 ? 1.0f / (float)tiles : 0.0f, inv_u2 = ua2 > 0 ? 1.0f / (float)ua2 : 0.0f;
    const int sbi = u.s0 / sp.sb;
    for (int it0 = 0; it0 < (total << lg); it0 += NT) {
      const int it = (it0 + threadIdx.x) >> lg, sub = threadIdx.x & (ksp - 1);
      const bool in = it < total;
      const int b = in ? fdivu(it, tiles, inv_t) : 0, r = in ? it - b * tiles : 0;
      const int ta = in ? fdivu(r, ua2, inv_u2) : 0;
      const int a0 = 2 * ta, a1 = min(a0 + 1, D - 1), p0 = 2 * (r - ta * ua2), p1 = min(p0 + 1, u.A - 1);
      const bool on = in && !(b > 0 && ((I.adj >> (b - 1)) & 1u));
      E acc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = A::c(A::zero(), A::zero());
      if (on)
        for (int sl = 0; sl < u.S; ++sl) {
          const V* qs = xs + site_slot(u.need, u.s0 + sl) * D * sp.Cp;
          const V *q0 = qs + a0 * sp.Cp, *q1 = qs + a1 * sp.Cp;
          const V* ys = Y + b * Yblk + sl * u.A * Yrow;
          const V *y0 = ys + p0 * Yrow, *y1 = ys + p1 * Yrow;
          constexpr int U = kMixed ? 4 : 1;
          V s[4][U];
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u4 = 0; u4 < U; ++u4) s[q][u4].x = s[q][u4].y = (T)0;
          auto cj = [](V& s, V q, V y) {  // s += conj(q) y
            s.x = fma(q.x, y.x, fma(q.y, y.y, s.x));
            s.y = fma(q.x, y.y, fma(-q.y, y.x, s.y));
          };
          auto step = [&](int c, int u4) {
            const V u0 = q0[c], u1 = q1[c], w0 = y0[c], w1 = y1[c];
            cj(s[0][u4], u0, w0);
            cj(s[1][u4], u0, w1);
            cj(s[2][u4], u1, w0);
            cj(s[3][u4], u1, w1);
          };
          int c = sub;
          for (; c + 3 * ksp < sp.Dc; c += 4 * ksp) {
#pragma unroll
            for (int u4 = 0; u4 < 4; ++u4) step(c + u4 * ksp, u4 % U);
          }
          for (; c < sp.Dc; c += ksp) step(c, 0);
          auto add = [&](E& e, V t) {
            if constexpr (kMixed)
              e = A::c(A::add(A::re(e), make_float2(t.x, 0.f)), A::add(A::im(e), make_float2(t.y, 0.f)));
            else
              e = A::c(A::add(A::re(e), t.x), A::add(A::im(e), t.y));
          };
#pragma unroll
          for (int q = 0; q < 4; ++q) add(acc[q], sum_parts<U>(s[q]));
        }
      for (int o = ksp >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          acc[q] = A::c(A::add(A::re(acc[q]), A::shfl_xor(A::re(acc[q]), o)),
                        A::add(A::im(acc[q]), A::shfl_xor(A::im(acc[q]), o)));
      if (on && sub == 0) {
        auto put = [&](int a, int p, E v) {
          if (sum)
            buf[(long long)sbi * nval + b * D2 + a * D + u.a0 + p] = v;
          else
            done(b, a, u.a0 + p, v);
        };
        put(a0, p0, acc[0]);
        if (p1 > p0) put(a0, p1, acc[1]);
        if (a1 > a0) {
          put(a1, p0, acc[2]);
          if (p1 > p0) put(a1, p1, acc[3]);
        }
      }
    }
  }
  pc.lap(P.ctl, 18);
  if (sum) {
    team_sync(tm);
    const float inv_d2 = 1.0f / (float)D2, inv_d = 1.0f / (float)D;
    for (int k = tm.gtid(); k < nval; k += tm.nthr()) {
      const int b = fdivu(k, D2, inv_d2), r = k - b * D2;
      if (b > 0 && ((I.adj >> (b - 1)) & 1u)) continue;
      typename A::S re = A::zero(), im = A::zero();
#pragma unroll 4
      for (int q = 0; q < sp.ns; ++q) {
        const E v = buf[(long long)q * nval + k];
        re = A::add(re, A::re(v));
        im = A::add(im, A::im(v));
      }
      const int a = fdivu(r, D, inv_d);
      done(b, a, r - a * D, A::c(re, im));
    }
    tm.parity ^= 1;
  }
  team_sync(tm);
  pc.lap(P.ctl, 19);
  if (tm.rank == 0 && threadIdx.x == 0) {
    atomicAdd(&P.ctl->applies, 1ull);
    atomicAdd(&P.ctl->flops, I.flops);
  }
  return true;
}

