// Observables beyond the populations: the energy surfaces of Eq. 3-4 and the bond entropies.
//
// Energy surfaces (Results, section on dynamic energy surfaces).  With the orthogonality
// centre at the root, the root tensor A[r][s] (r = the bond indices, s = the electronic state)
// has the Schmidt form A = sum_k sigma_k phi_k(r) u_k(s) for the bipartition electronic |
// environment: u_k are the eigenvectors of rho_S = A^T conj(A) and phi_k = A conj(u_k) / sigma_k.
// In the basis |phi_k>|l> (bath-major) the effective Hamiltonian is
//   H_eff[(i j), (k l)] = <phi_i, j| H |phi_k, l> = sum_r conj(phi_i(r)) (H_root X_kl)[r][j],
// X_kl[r][s] = phi_k(r) delta_sl, H_root the root's local effective Hamiltonian (its
// environment blocks project H onto the bond basis); V_eff = H_eff - T_eff with T the chains'
// kinetic energy, whose environment blocks come from its own environment pass.
//
// Bond entropies (Results, ER section; Methods): S_e = -sum_a lambda_a ln lambda_a over the
// eigenvalues of the density matrix of bond e (the downward pass of bond densities).
//
// Eigenvalues and eigenvectors of the small Hermitian matrices come from a cyclic Jacobi
// method for complex Hermitian matrices (Golub & Van Loan, "Matrix Computations", the
// symmetric Jacobi method with parallel ordering, complex rotations): one CTA per matrix, FP64.
#include <cuda_runtime.h>

#include <algorithm>

#include "index.cuh"
#include "internal.h"

namespace ttns {

namespace {
constexpr int kJT = 256;
}

// Batched complex Hermitian Jacobi.  Matrix b (n_b = ns[b] <= 64) starts at base + offs[b],
// row-major with leading dimension ld[b]; eigenvalues (ascending) go to evals + b * 64, and
// when evecs != nullptr the eigenvectors (columns, in the same order) to evecs + b * 64 * 64
// (leading dimension 64).  Dynamic shared memory: n_max^2 complex, twice with vectors.
//
// Bound by latency (the rotation's scalars and the barriers), so a sweep takes n - 1 rounds of
// n / 2 disjoint pivots (round-robin ordering) instead of n (n - 1) / 2 pivots one after another:
// every pair's scalars on its own thread (two reciprocal square roots), then every 2 x 2 block of
// A rotated from both sides by one thread, two barriers per round: 0.27 ms for 37 bond spectra
// with n <= 12.
struct JacobiRot {
  double c;
  double2 s;  // p' = c p - conj(s) q, q' = s p + c q (columns)
};
__global__ void __launch_bounds__(kJT) k_herm_jacobi(const double2* base, const long long* offs, const int* ns,
                                                     const int* lds, double* evals, double2* evecs, int n_max,
                                                     int max_sweeps) {
  extern __shared__ double2 jsm[];
  const int b = blockIdx.x;
  const int n = ns[b];
  const int ld = lds[b];
  const double2* Ain = base + offs[b];
  double2* A = jsm;
  double2* V = jsm + n_max * n_max;
  const bool vecs = evecs != nullptr;
  __shared__ double s_off[kJT / 32], s_diag[kJT / 32];
  __shared__ JacobiRot s_rot[32];
  __shared__ int s_p[32], s_q[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int idx = threadIdx.x; idx < n * n; idx += kJT) {
    const int r = idx / n, c = idx % n;
    A[r * n_max + c] = Ain[(long long)r * ld + c];
    if (vecs) V[r * n_max + c] = make_double2(r == c ? 1.0 : 0.0, 0.0);
  }
  const int m = n + (n & 1), np = m / 2;  // players and pairs (an odd n has a pair with index n: no rotation)
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    __syncthreads();
    double off = 0.0, dg = 0.0;
    for (int idx = threadIdx.x; idx < n * n; idx += kJT) {
      const int r = idx / n, c = idx - r * n;
      const double2 a = A[r * n_max + c];
      if (r == c)
        dg = fma(a.x, a.x, dg);
      else
        off = fma(a.x, a.x, fma(a.y, a.y, off));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      dg += __shfl_xor_sync(0xffffffffu, dg, o);
    }
    if (lane == 0) {
      s_off[warp] = off;
      s_diag[warp] = dg;
    }
    __syncthreads();
    off = dg = 0.0;
    for (int w = 0; w < kJT / 32; ++w) {
      off += s_off[w];
      dg += s_diag[w];
    }
    if (!(off > 1e-30 * (dg + off))) break;
    for (int round = 0; round < m - 1; ++round) {
      __syncthreads();  // the last round's blocks are written
      if (threadIdx.x < np) {
        const int i = threadIdx.x;
        int p = i == 0 ? m - 1 : (round + i) % (m - 1);
        int q = i == 0 ? round : (round - i + m - 1) % (m - 1);
        if (p > q) {
          const int x = p;
          p = q;
          q = x;
        }
        JacobiRot r{1.0, make_double2(0.0, 0.0)};
        if (q < n) {
          // t = tan of the rotation: with d = A_qq - A_pp, h = sqrt(d^2 + 4 |A_pq|^2),
          // c^2 = (1 + |d| / h) / 2 and s = sign(d) A_pq / (h c)
          const double2 apq = A[p * n_max + q];
          const double d = A[q * n_max + q].x - A[p * n_max + p].x;
          const double r2 = fma(apq.x, apq.x, apq.y * apq.y);
          const double h2 = fma(d, d, 4.0 * r2);
          if (r2 > 0.0 && h2 > 1e-300) {
            const double y = rsqrt(h2);
            const double c2 = fma(0.5 * fabs(d), y, 0.5);
            const double rc = rsqrt(c2);
            const double k = (d >= 0.0 ? y : -y) * rc;
            r.c = c2 * rc;
            r.s = make_double2(k * apq.x, k * apq.y);
          }
        }
        s_rot[i] = r;
        s_p[i] = p;
        s_q[i] = q;
      }
      __syncthreads();
      // block (i, j), i <= j: B <- J_i^H B J_j, and its mirror image
      for (int idx = threadIdx.x; idx < np * np; idx += kJT) {
        const int i = idx / np, j = idx - i * np;
        if (i > j) continue;
        const int p1 = s_p[i], q1 = s_q[i], p2 = s_p[j], q2 = s_q[j];
        const JacobiRot ri = s_rot[i], rj = s_rot[j];
        const bool oi = q1 < n, oj = q2 < n;
        const double2 z = make_double2(0.0, 0.0);
        double2 pp = A[p1 * n_max + p2], pq = oj ? A[p1 * n_max + q2] : z, qp = oi ? A[q1 * n_max + p2] : z,
                qq = oi && oj ? A[q1 * n_max + q2] : z;
        auto lin = [](double c, double2 a, double2 s, double2 b) {  // c a + s b
          return make_double2(fma(c, a.x, fma(s.x, b.x, -s.y * b.y)), fma(c, a.y, fma(s.x, b.y, s.y * b.x)));
        };
        auto neg = [](double2 a) { return make_double2(-a.x, -a.y); };
        auto conj = [](double2 a) { return make_double2(a.x, -a.y); };
        // columns: p' = c p - conj(s) q, q' = s p + c q
        const double2 pp1 = lin(rj.c, pp, neg(conj(rj.s)), pq), pq1 = lin(rj.c, pq, rj.s, pp);
        const double2 qp1 = lin(rj.c, qp, neg(conj(rj.s)), qq), qq1 = lin(rj.c, qq, rj.s, qp);
        // rows (the conjugate): p' = c p - s q, q' = conj(s) p + c q
        pp = lin(ri.c, pp1, neg(ri.s), qp1);
        pq = lin(ri.c, pq1, neg(ri.s), qq1);
        qp = lin(ri.c, qp1, conj(ri.s), pp1);
        qq = lin(ri.c, qq1, conj(ri.s), pq1);
        if (i == j) {
          A[p1 * n_max + p1] = make_double2(pp.x, 0.0);
          if (oi) {
            A[q1 * n_max + q1] = make_double2(qq.x, 0.0);
            A[p1 * n_max + q1] = z;
            A[q1 * n_max + p1] = z;
          }
          continue;
        }
        A[p1 * n_max + p2] = pp;
        A[p2 * n_max + p1] = conj(pp);
        if (oj) {
          A[p1 * n_max + q2] = pq;
          A[q2 * n_max + p1] = conj(pq);
        }
        if (oi) {
          A[q1 * n_max + p2] = qp;
          A[p2 * n_max + q1] = conj(qp);
        }
        if (oi && oj) {
          A[q1 * n_max + q2] = qq;
          A[q2 * n_max + q1] = conj(qq);
        }
      }
      if (vecs) {
        for (int idx = threadIdx.x; idx < n * np; idx += kJT) {
          const int k = idx / np, i = idx - k * np;
          const int p = s_p[i], q = s_q[i];
          if (q >= n) continue;
          const JacobiRot r = s_rot[i];
          const double2 vp = V[k * n_max + p], vq = V[k * n_max + q];
          V[k * n_max + p] = make_double2(fma(r.c, vp.x, fma(-r.s.x, vq.x, -r.s.y * vq.y)),
                                          fma(r.c, vp.y, fma(-r.s.x, vq.y, r.s.y * vq.x)));
          V[k * n_max + q] = make_double2(fma(r.c, vq.x, fma(r.s.x, vp.x, -r.s.y * vp.y)),
                                          fma(r.c, vq.y, fma(r.s.x, vp.y, r.s.y * vp.x)));
        }
      }
    }
  }
  __syncthreads();
  // ascending order (selection by rank: the count of smaller values, ties by index)
  for (int i = threadIdx.x; i < n; i += kJT) {
    const double di = A[i * n_max + i].x;
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double dj = A[j * n_max + j].x;
      rank += (dj < di) || (dj == di && j < i);
    }
    evals[(long long)b * 64 + rank] = di;
    if (vecs)
      for (int k = 0; k < n; ++k) evecs[(long long)b * 64 * 64 + (long long)k * 64 + rank] = V[k * n_max + i];
  }
}

// ------------------------------------------------------------------ downward pass
// Bond densities and occupations of one level of the tree (all nodes of equal depth), three
// launches per level instead of three or four per density: a chain's levels depend on one
// another, but its siblings do not, and the launches were the time.  FP64.
//
// X = rho_in on leg 0 of every node's tensor, X[idx] = sum_a' rho_in[a'][a] A[.., a', ..] with a
// the leg-0 index of idx, and the partial sums of <n> = sum s Re(X conj(A)) over the block's
// elements (s = the physical leg's index, the last leg).  Grid: (blocks, nodes).
constexpr int kDT = 256;
__global__ void __launch_bounds__(kDT) k_down_x(const double2* pool, const NodeDesc* nodes, DownBatch b,
                                                const double* obs, double2* X, long long kvec, double* occ_part) {
  extern __shared__ double2 s_rho[];
  const DownNode dn = b.node[blockIdx.y];
  if (dn.rho_in < 0) return;  // the root: X is the tensor itself, and it has no occupation here
  const NodeDesc nd = nodes[dn.node];
  const double2* A = pool + nd.off;
  double2* Xv = X + (long long)blockIdx.y * kvec;
  const double2* rho = reinterpret_cast<const double2*>(obs + dn.rho_in);
  const int Dp = nd.dims[0], stp = nd.strides[0];
  for (int k = threadIdx.x; k < Dp * Dp; k += kDT) s_rho[k] = rho[k];
  __syncthreads();
  const int d = nd.dims[nd.nl - 1];
  double occ = 0.0;
  for (int idx = blockIdx.x * kDT + threadIdx.x; idx < nd.size; idx += gridDim.x * kDT) {
    const int a = fdivu(idx, stp, nd.inv_strides[0]);
    const double2* x = A + (idx - a * stp);
    double r0 = 0.0, i0 = 0.0, r1 = 0.0, i1 = 0.0;
    int a2 = 0;
    for (; a2 + 1 < Dp; a2 += 2) {
      const double2 w0 = s_rho[a2 * Dp + a], w1 = s_rho[(a2 + 1) * Dp + a];
      const double2 v0 = x[(long long)a2 * stp], v1 = x[(long long)(a2 + 1) * stp];
      r0 = fma(w0.x, v0.x, fma(-w0.y, v0.y, r0));
      i0 = fma(w0.x, v0.y, fma(w0.y, v0.x, i0));
      r1 = fma(w1.x, v1.x, fma(-w1.y, v1.y, r1));
      i1 = fma(w1.x, v1.y, fma(w1.y, v1.x, i1));
    }
    if (a2 < Dp) {
      const double2 w0 = s_rho[a2 * Dp + a], v0 = x[(long long)a2 * stp];
      r0 = fma(w0.x, v0.x, fma(-w0.y, v0.y, r0));
      i0 = fma(w0.x, v0.y, fma(w0.y, v0.x, i0));
    }
    r0 += r1;
    i0 += i1;
    Xv[idx] = make_double2(r0, i0);
    if (dn.occ >= 0) {
      const int s = idx - fdivu(idx, d, nd.inv_dims[nd.nl - 1]) * d;
      const double2 v = A[idx];
      occ = fma((double)s, fma(r0, v.x, i0 * v.y), occ);
    }
  }
  if (dn.occ < 0) return;
  __shared__ double s_occ[kDT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) occ += __shfl_xor_sync(0xffffffffu, occ, o);
  if ((threadIdx.x & 31) == 0) s_occ[threadIdx.x >> 5] = occ;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kDT / 32; ++w) s += s_occ[w];
    occ_part[blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

// Partials of rho[c][c2] = sum_rows X[row, c] conj(A[row, c2]), c <= c2 (Hermitian), along the
// density's leg, rows split over the blocks.  Grid: (blocks, densities).
__global__ void __launch_bounds__(kDT) k_down_density(const double2* pool, const NodeDesc* nodes, DownBatch b,
                                                      const double2* X, long long kvec, double* part,
                                                      long long part_stride) {
  const DownDens dd = b.dens[blockIdx.y];
  const DownNode dn = b.node[dd.item];
  const NodeDesc nd = nodes[dn.node];
  const double2* A = pool + nd.off;
  const double2* Xv = dn.rho_in < 0 ? A : X + (long long)dd.item * kvec;
  const int D = dd.D, st = nd.strides[dd.leg];
  const int rows = nd.size / D, chunk = (rows + gridDim.x - 1) / gridDim.x;
  const int r0 = min(rows, (int)blockIdx.x * chunk), r1 = min(rows, r0 + chunk);
  double* out = part + (long long)(blockIdx.y * gridDim.x + blockIdx.x) * part_stride;
  const int np = D * (D + 1) / 2;
  for (int p = threadIdx.x; p < np; p += kDT) {  // pair p = c2 (c2 + 1) / 2 + c
    int c2 = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((c2 + 1) * (c2 + 2) / 2 <= p) ++c2;
    while (c2 * (c2 + 1) / 2 > p) --c2;
    const int c = p - c2 * (c2 + 1) / 2;
    double re = 0.0, im = 0.0;
    for (int r = r0; r < r1; ++r) {
      const int q = fdivu(r, st, nd.inv_strides[dd.leg]);
      const long long base = (long long)q * D * st + (r - q * st);
      const double2 x = Xv[base + (long long)c * st], y = A[base + (long long)c2 * st];
      re = fma(x.x, y.x, fma(x.y, y.y, re));
      im = fma(x.y, y.x, fma(-x.x, y.y, im));
    }
    out[2 * p] = re;
    out[2 * p + 1] = im;
  }
}

// Fixed-order sums of both kinds of partials, one warp per value (lanes over the blocks, then a
// butterfly: one thread per value walked through up to a hundred dependent FP64 additions).
// Grid: (blocks, densities + nodes).
__global__ void __launch_bounds__(kDT) k_down_sum(DownBatch b, const double* part, long long part_stride, int nblk_d,
                                                  const double* occ_part, int nblk_x, double* obs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((int)blockIdx.y < b.n_dens) {
    const DownDens dd = b.dens[blockIdx.y];
    const int D = dd.D, np = D * (D + 1) / 2;
    double2* out = reinterpret_cast<double2*>(obs + dd.out);
    const double* src = part + (long long)blockIdx.y * nblk_d * part_stride;
    for (int p = blockIdx.x * (kDT / 32) + warp; p < np; p += gridDim.x * (kDT / 32)) {
      double re = 0.0, im = 0.0;
      for (int k = lane; k < nblk_d; k += 32) {
        const double2 v = *reinterpret_cast<const double2*>(src + k * part_stride + 2 * p);
        re += v.x;
        im += v.y;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) {
        int c2 = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
        while ((c2 + 1) * (c2 + 2) / 2 <= p) ++c2;
        while (c2 * (c2 + 1) / 2 > p) --c2;
        const int c = p - c2 * (c2 + 1) / 2;
        out[c * D + c2] = make_double2(re, im);
        out[c2 * D + c] = make_double2(re, -im);
      }
    }
    return;
  }
  const DownNode dn = b.node[blockIdx.y - b.n_dens];
  if (dn.occ < 0 || blockIdx.x != 0 || warp != 0) return;
  double s = 0.0;
  for (int k = lane; k < nblk_x; k += 32) s += occ_part[(blockIdx.y - b.n_dens) * nblk_x + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) obs[dn.occ] = s;
}

// partials: 1024 slots of 2 maxD^2 doubles at the front of the observables buffer; the
// occupation partials take the last ones
cudaError_t launch_down(const double2* pool, const NodeDesc* d_nodes, const DownBatch& b, double* obs, double2* xbuf,
                        long long kvec, double* partials, cudaStream_t st) {
  int max_size = 1, max_rho = 1, max_D = 1;
  bool any_x = false;
  for (int k = 0; k < b.n_nodes; ++k) {
    max_size = std::max(max_size, b.node[k].size);
    any_x = any_x || b.node[k].rho_in >= 0;
  }
  for (int k = 0; k < b.n_dens; ++k) max_D = std::max(max_D, b.dens[k].D);
  max_rho = 64 * 64 * (int)sizeof(double2);
  // about two waves of blocks over the level, one element (or a few rows) per thread at least
  const int nblk_x = std::max(1, std::min({(max_size + kDT - 1) / kDT, 304 / std::max(1, b.n_nodes) + 1, 128}));
  const long long stride = (long long)max_D * (max_D + 1);
  const int nblk_d =
      b.n_dens ? std::max(1, std::min({max_size / max_D / 4, 608 / b.n_dens + 1, 960 / b.n_dens})) : 1;
  double* occ_part = partials + 960LL * stride;
  if (any_x) {
    cudaError_t e = cudaFuncSetAttribute(k_down_x, cudaFuncAttributeMaxDynamicSharedMemorySize, max_rho);
    if (e != cudaSuccess) return e;
    k_down_x<<<dim3(nblk_x, b.n_nodes), kDT, max_rho, st>>>(pool, d_nodes, b, obs, xbuf, kvec, occ_part);
  }
  if (b.n_dens) k_down_density<<<dim3(nblk_d, b.n_dens), kDT, 0, st>>>(pool, d_nodes, b, xbuf, kvec, partials, stride);
  k_down_sum<<<dim3(std::max(1, std::min(32, (int)(stride / 2 + kDT / 32 - 1) / (kDT / 32))), b.n_dens + b.n_nodes), kDT,
               0, st>>>(
      b, partials, stride, nblk_d, occ_part, nblk_x, obs);
  return cudaGetLastError();
}

// Populations of every tree in tree order, one block per tree: sum_r |A[r][s]|^2 of its root
// tensor (the physical leg is the last one).
__global__ void __launch_bounds__(kDT) k_populations(const double2* pool, const NodeDesc* nodes, const TreeDesc* trees,
                                                     double* out) {
  const TreeDesc td = trees[blockIdx.x];
  const NodeDesc nd = nodes[td.node0];
  const double2* A = pool + nd.off;
  const int ne = td.n_el, rows = nd.size / ne;
  int off = 0;
  for (int k = 0; k < (int)blockIdx.x; ++k) off += trees[k].n_el;
  __shared__ double s_sum[kDT / 32];
  for (int s = 0; s < ne; ++s) {
    double v = 0.0;
    for (int r = threadIdx.x; r < rows; r += kDT) {
      const double2 a = A[(long long)r * ne + s];
      v = fma(a.x, a.x, fma(a.y, a.y, v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < kDT / 32; ++w) t += s_sum[w];
      out[off + s] = t;
    }
    __syncthreads();
  }
}

cudaError_t launch_populations(const double2* pool, const NodeDesc* d_nodes, const TreeDesc* d_trees, int n_trees,
                               double* out, cudaStream_t st) {
  k_populations<<<n_trees, kDT, 0, st>>>(pool, d_nodes, d_trees, out);
  return cudaGetLastError();
}

// phi_k(r) = sum_s A[r][s] conj(U[s][k]) / sig[k] for the kept bath states k < nb
__global__ void k_bath_states(const double2* A, long long R, int n_el, const double2* U, const double* sig, int nb,
                              double2* Phi) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < R * nb;
       idx += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(idx / R);
    const long long r = idx - (long long)k * R;
    double re = 0.0, im = 0.0;
    for (int s = 0; s < n_el; ++s) {
      const double2 a = A[r * n_el + s], u = U[s * nb + k];
      re += a.x * u.x + a.y * u.y;
      im += a.y * u.x - a.x * u.y;
    }
    Phi[(long long)k * R + r] = make_double2(re / sig[k], im / sig[k]);
  }
}

// The columns of the projected operators go through in batches (blockIdx.y; vector b of a batch at
// kvec b): one column after another left most of the chip idle.
//
// X[r][s] = phi_k(r) delta_{s l} for column c0 + b = k n_el + l
__global__ void k_build_x(const double2* Phi, int c0, long long R, int n_el, double2* X, long long kvec) {
  const int k = (c0 + (int)blockIdx.y) / n_el, l = (c0 + (int)blockIdx.y) % n_el;
  X += blockIdx.y * kvec;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < R * n_el;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long r = idx / n_el;
    const int s = (int)(idx - r * n_el);
    X[idx] = s == l ? Phi[(long long)k * R + r] : make_double2(0.0, 0.0);
  }
}

// per-block partials of out[(i j)] = sum_r conj(phi_i(r)) y[r][j], as (re, im) pairs
__global__ void k_project_partial(const double2* y, const double2* Phi, long long R, int n_el, int nb,
                                  double* partials, long long kvec) {
  const int nv = nb * n_el;
  y += blockIdx.y * kvec;
  partials += (long long)blockIdx.y * gridDim.x * 2 * nv;
  const long long chunk = (R + gridDim.x - 1) / gridDim.x;
  const long long r0 = blockIdx.x * chunk, r1 = min(R, r0 + chunk);
  for (int o = threadIdx.x; o < nv; o += blockDim.x) {
    const int i = o / n_el, j = o % n_el;
    double re = 0.0, im = 0.0;
    for (long long r = r0; r < r1; ++r) {
      const double2 p = Phi[(long long)i * R + r], v = y[r * n_el + j];
      re += p.x * v.x + p.y * v.y;
      im += p.x * v.y - p.y * v.x;
    }
    partials[(long long)blockIdx.x * 2 * nv + 2 * o] = re;
    partials[(long long)blockIdx.x * 2 * nv + 2 * o + 1] = im;
  }
}

// out[k] = sum over blocks of partials (fixed order, one warp per value); blockIdx.y: column of a
// column-major matrix
__global__ void k_reduce_to(const double* partials, int nblocks, int nval, double* out) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  partials += (long long)blockIdx.y * nblocks * nval;
  out += (long long)blockIdx.y * nval;
  for (int k = blockIdx.x * nw + (threadIdx.x >> 5); k < nval; k += gridDim.x * nw) {
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partials[(long long)b * nval + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[k] = s;
  }
}

__global__ void k_sub(const double* a, const double* b, double* c, int n) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) c[k] = a[k] - b[k];
}

cudaError_t launch_herm_jacobi(const double2* base, const long long* offs, const int* ns, const int* lds, int count,
                               int n_max, double* evals, double2* evecs, cudaStream_t st) {
  const size_t smem = (size_t)n_max * n_max * sizeof(double2) * (evecs ? 2 : 1);
  cudaError_t e = cudaFuncSetAttribute(k_herm_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_herm_jacobi<<<count, kJT, smem, st>>>(base, offs, ns, lds, evals, evecs, n_max, 60);
  return cudaGetLastError();
}

cudaError_t launch_bath_states(const double2* A, long long R, int n_el, const double2* U, const double* sig, int nb,
                               double2* Phi, cudaStream_t st) {
  const int blocks = (int)std::min<long long>(1024, (R * nb + 255) / 256);
  k_bath_states<<<blocks, 256, 0, st>>>(A, R, n_el, U, sig, nb, Phi);
  return cudaGetLastError();
}

cudaError_t launch_build_x(const double2* Phi, int c0, int count, long long R, int n_el, double2* X, long long kvec,
                           cudaStream_t st) {
  const int blocks = (int)std::min<long long>(256, (R * n_el + 255) / 256);
  k_build_x<<<dim3(blocks, count), 256, 0, st>>>(Phi, c0, R, n_el, X, kvec);
  return cudaGetLastError();
}

cudaError_t launch_project(const double2* y, const double2* Phi, long long R, int n_el, int nb, double* partials,
                           int nblocks, double* out, int count, long long kvec, cudaStream_t st) {
  k_project_partial<<<dim3(nblocks, count), 128, 0, st>>>(y, Phi, R, n_el, nb, partials, kvec);
  const int nval = 2 * nb * n_el;
  k_reduce_to<<<dim3((nval + 7) / 8, count), 256, 0, st>>>(partials, nblocks, nval, out);
  return cudaGetLastError();
}

cudaError_t launch_sub(const double* a, const double* b, double* c, int n, cudaStream_t st) {
  k_sub<<<(n + 255) / 256, 256, 0, st>>>(a, b, c, n);
  return cudaGetLastError();
}

}  // namespace ttns
