// Gauge absorb (included by sweep.cu).
//
// A_u <- R applied on leg I.leg, in FP64 (TTNS_FP64) or double-single (the mixed modes).  Along
// the leg the tensor falls into independent fibres of D elements; every CTA owns a range of
// them, so the product is done in place: no second copy of the tensor and no barrier between
// reading and writing.  The fibres are converted once into shared memory (k-major), R too, and
// few outputs per CTA are split over two or four lanes each.  (40 x 40 x 20 tensors of the ER
// tree on the whole grid: 24 us per absorb with a converted global copy before, 15 us now.)
template <typename A>
__device__ __noinline__ void op_absorb(const KernelParams& P, Team& tm, const Instr& I) {
  using E = typename A::E;
  using Acc = typename A::Acc;
  const NodeDesc nd = P.nodes[I.node];
  const int l = I.leg;
  const int D = nd.dims[l], st = nd.strides[l];
  const int F = nd.size / D;
  const float inv_st = nd.inv_strides[l], inv_D = nd.inv_dims[l];
  double2* Ag = P.pool + nd.off;
  const double2* R = P.pool + P.trees[I.tree].bond_off;
  E* Rs = reinterpret_cast<E*>(dyn_smem);
  E* xs = Rs + D * D;
  const int chunk = (F + tm.size - 1) / tm.size;
  const int fb = min(F, tm.rank * chunk), fe = min(F, fb + chunk);
  const int cap = max(1, (int)((P.smem_bytes / (long long)sizeof(E) - D * D) / D));  // fibres per pass
  __syncthreads();
  for (int k = threadIdx.x; k < D * D; k += NT) Rs[k] = A::cfrom(R[k]);
  for (int f0 = fb; f0 < fe; f0 += cap) {
    const int nf = min(cap, fe - f0);
    const float inv_nf = 1.0f / (float)nf;
    auto addr = [&](int f, int k) {  // element k of fibre f0 + f
      const int q = fdivu(f0 + f, st, inv_st);
      return (long long)q * D * st + (f0 + f - q * st) + (long long)k * st;
    };
    __syncthreads();
    for (int it = threadIdx.x; it < nf * D; it += NT) {
      int f, k;
      if (st == 1) {  // consecutive threads along contiguous memory
        f = fdivu(it, D, inv_D);
        k = it - f * D;
      } else {
        k = fdivu(it, nf, inv_nf);
        f = it - k * nf;
      }
      xs[k * nf + f] = A::cfrom(Ag[addr(f, k)]);
    }
    __syncthreads();
    const int items = nf * D;
    const int lg = 4 * items <= NT ? 2 : (2 * items <= NT ? 1 : 0);  // lanes per output
    const int ks = 1 << lg;
    for (int it0 = 0; it0 < (items << lg); it0 += NT) {
      const int it = (it0 + threadIdx.x) >> lg, sub = threadIdx.x & (ks - 1);
      const bool on = it < items;
      const int i = on ? fdivu(it, nf, inv_nf) : 0;
      const int f = on ? it - i * nf : 0;
      Acc ar, ai, br, bi;
      ar.init(A::zero());
      ai.init(A::zero());
      br.init(A::zero());
      bi.init(A::zero());
      const E* row = Rs + i * D;
      int k = sub;
      for (; k + ks < D; k += 2 * ks) {
        q_cmac<A>(ar, ai, row[k], xs[k * nf + f]);
        q_cmac<A>(br, bi, row[k + ks], xs[(k + ks) * nf + f]);
      }
      if (k < D) q_cmac<A>(ar, ai, row[k], xs[k * nf + f]);
      typename A::S r = A::add(ar.val(), br.val()), m = A::add(ai.val(), bi.val());
      for (int o = ks >> 1; o > 0; o >>= 1) {
        r = A::add(r, A::shfl_xor(r, o));
        m = A::add(m, A::shfl_xor(m, o));
      }
      if (on && sub == 0) Ag[addr(f, i)] = A::cto(A::c(r, m));
    }
  }
  team_sync(tm);
}

// the arithmetic of sums over rows in the given compute type
template <typename T> struct EnvArith;
template <> struct EnvArith<double> { using A = QrF64; };
template <> struct EnvArith<float> { using A = QrDs; };
