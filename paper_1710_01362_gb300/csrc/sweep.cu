// Device side of the TTNS sweep: one persistent cooperative kernel that runs the
// compiled one-site TDVP step (Results, "TTNS for vibronic quantum dynamics":
// every tensor evolved in turn with its local effective Hamiltonian) for n steps.
//
// Execution model (GB300: 152 SMs, FP64 at about 1/80 of the FP32 rate with a long
// dependent latency, and the FP64 <-> FP32 conversions on the same narrow pipe; hardware
// cluster barriers ~0.2 us; the software grid barrier meets at the cluster barrier first):
//   * a "team" executes one instruction: either one thread-block cluster (hardware
//     barrier; small tensors, and every QR below the QR threshold) or the whole grid
//     (software barrier; Krylov exponentials, environment updates and absorbs of tensors
//     above the grid threshold);
//   * in batched mode every cluster advances its own trees independently;
//   * reductions are deterministic: per-CTA partials, then a fixed-order sum
//     that every CTA computes identically (no floating-point atomics);
//   * every spin-wait is bounded and reports TTNS_E_TIMEOUT instead of hanging.
//
// Two instances of the kernel are compiled from this file: one CTA per SM with all of its
// registers and shared memory, and (SWEEP_PAIR, from sweep_pair.cu) two CTAs per SM for sets of
// many small trees.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <type_traits>

#include "internal.h"
#include "ds.cuh"
#include "index.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

#ifdef SWEEP_PAIR
#define SWEEP_CTAS 2
#else
#define SWEEP_CTAS 1
#endif

namespace ttns {
#ifdef SWEEP_PAIR
namespace pair {
#endif

#define NT 256
#define NWARP (NT / 32)
#define HBAR_EVFS 0.6582119569

// status codes mirrored from ttns.h
#define ST_TIMEOUT 5
#define ST_NOT_CONVERGED 4
#define ST_NONFINITE 6
#define ST_LAUNCH 3       // the launch did not have the cluster shape / shared memory it was planned for

__constant__ double c_inv[256];       // 1/n, c_inv[0] = 0

// ------------------------------------------------------------------ complex helpers
template <typename T> struct C2;
template <> struct C2<double> { using t = double2; };
template <> struct C2<float> { using t = float2; };

template <typename T>
__device__ __forceinline__ typename C2<T>::t ld(const double2* p) {
  double2 v = *p;
  typename C2<T>::t r;
  r.x = (T)v.x;
  r.y = (T)v.y;
  return r;
}
template <typename T>
__device__ __forceinline__ typename C2<T>::t cvt(double2 v) {
  typename C2<T>::t r;
  r.x = (T)v.x;
  r.y = (T)v.y;
  return r;
}
template <>
__device__ __forceinline__ float2 cvt<float>(double2 v) {  // no conversion on the narrow FP64 pipe
  return make_float2(d2f_bits(v.x), d2f_bits(v.y));
}
template <typename T>
__device__ __forceinline__ typename C2<T>::t cvt(float2 v) {
  typename C2<T>::t r;
  r.x = (T)v.x;
  r.y = (T)v.y;
  return r;
}

template <typename T>
__device__ __forceinline__ void cmac(typename C2<T>::t& acc, typename C2<T>::t a, typename C2<T>::t b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
// Sum of U partial sums.  In FP32 the products of a leg and the projections keep four accumulators
// per output (every fourth term each), as mode_dot does: with one, the rounding of a chain of 16 to
// 64 additions made the errors against FP64 references 1.1 to 1.4 times as large (one step of 4 x 3
// stars of D 16 and 20, two steps of 8-site chains of D 24; geometric means over 24 to 64 seeds;
// 0.8 to 1.07 now).  They cost 0.4 to 3.4 %: 25-site chain 44.2 -> 45.7 ms, 4 x 20 star 56.1 ->
// 57.1, 8 x 60 ER tree 348.3 -> 349.7.
template <int U, typename V>
__device__ __forceinline__ V sum_parts(const V* a) {
  V r = a[0];
  if constexpr (U == 2) {
    r.x += a[1].x;
    r.y += a[1].y;
  } else if constexpr (U == 4) {
    r.x += a[1].x + (a[2].x + a[3].x);
    r.y += a[1].y + (a[2].y + a[3].y);
  }
  return r;
}

// ------------------------------------------------------------------ teams
struct Team {
  int kind;      // TEAM_GRID / TEAM_CLUSTER
  int rank;      // CTA rank in the team
  int size;      // CTAs in the team
  double* red;   // two partial buffers, red_stride doubles each
  long long red_stride;
  int parity;
  Ctl* ctl;
  long long spin_limit;
  int csize;     // CTAs per thread-block cluster (the grid team reduces per cluster first)
  __device__ int nthr() const { return size * NT; }
  __device__ int gtid() const { return rank * NT + (int)threadIdx.x; }
};

__device__ __forceinline__ int ld_volatile_int(const int* p) { return *(volatile const int*)p; }

__device__ void set_status(Ctl* ctl, int st, int where, int node) {
  if (atomicCAS(&ctl->status, 0, st) == 0) {
    ctl->err_where = where;
    ctl->err_node = node;
  }
}

// software barrier over all CTAs of the grid; bounded.  Hierarchical: the CTAs of each
// thread-block cluster meet at the hardware cluster barrier, one thread per cluster arrives
// at the global counter and waits for the generation to change, and a second cluster barrier
// releases its cluster.  The cluster barriers' release/acquire and the global release/acquire
// pair order every CTA's writes before the barrier with every CTA's reads after it.  A launch
// without clusters is a grid of one-CTA clusters.
//
// The counter only grows (64 bits), and a cluster waits for it to reach the next multiple of the
// number of clusters: the last arrival is at once the release (a counter reset and a separate
// generation word cost the others a fence and another round trip).  An environment update, which has
// two: 35 us before, 30 now.
__device__ void grid_sync(Ctl* ctl, long long spin_limit) {
  cg::cluster_group cl = cg::this_cluster();
  const unsigned csz = cl.num_blocks();
  if (csz > 1) cl.sync(); else __syncthreads();
  if (cl.block_rank() == 0 && threadIdx.x == 0) {
    const unsigned nclu = gridDim.x / csz;
    unsigned long long prev;
    asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], 1;" : "=l"(prev) : "l"(&ctl->bar_count) : "memory");
    const unsigned long long target = prev - prev % nclu + nclu;
    if (prev + 1 != target) {
      // bounded wait; the bound applies to time without progress of the working cluster
      long long t0 = clock64();
      unsigned seen = *(volatile unsigned*)&ctl->progress;
      for (;;) {
        unsigned long long now;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(now) : "l"(&ctl->bar_count) : "memory");
        if (now >= target) break;
        if (ld_volatile_int(&ctl->status) != 0) break;
        const unsigned pr = *(volatile unsigned*)&ctl->progress;
        if (pr != seen) {
          seen = pr;
          t0 = clock64();
        }
        if (clock64() - t0 > spin_limit) {
          set_status(ctl, ST_TIMEOUT, 100, -1);
          break;
        }
      }
    }
  }
  if (csz > 1) cl.sync(); else __syncthreads();
}

__device__ __forceinline__ void team_sync(Team& tm) {
  if (tm.kind == TEAM_CLUSTER) {
    if (tm.size > 1)
      cg::this_cluster().sync();
    else
      __syncthreads();  // a cluster barrier costs 450 cycles even for one CTA
  } else {
    grid_sync(tm.ctl, tm.spin_limit);
  }
}

// warp sum with a fixed order; every lane returns lane 0's value
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return __shfl_sync(0xffffffffu, v, 0);
}

// Sum of V values (a power of two <= 16) over a warp with V - 1 + 5 - log2(V) additions per
// lane instead of 5 V: the first log2(V) butterfly levels exchange half of the remaining
// values, the rest are plain.  Lane L returns the total of value warp_reduce_vid<V>(L); the
// FP64 pipe, which also runs these additions, is the narrow one on this part.
template <int V>
__device__ __forceinline__ int warp_reduce_vid(int lane) {
  int vid = 0;
#pragma unroll
  for (int n = V, off = 16; n > 1; n >>= 1, off >>= 1)
    if (lane & off) vid += n / 2;
  return vid;
}
template <int V>
__device__ __forceinline__ double warp_reduce_t(double* v) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int n = V; n > 1; n >>= 1, off >>= 1) {
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const double send = hi ? v[i] : v[i + n / 2];
      const double keep = hi ? v[i + n / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  double t = v[0];
#pragma unroll
  for (; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  return t;
}

// All-reduce of NV <= 4 per-thread values over the team.  Deterministic and identical on every
// CTA.  Inside a CTA the 256 values go through shared memory to warp 0, which adds them in a
// fixed tree (7 additions per lane, then one transposing butterfly for all values, instead of a
// butterfly per value on every warp: a warp's FP64 addition holds the SM's FP64 unit for about
// 20 cycles whatever its lanes do).  Cluster teams push each CTA's totals into every peer's
// shared memory before the cluster barrier, so that after it the sums come from local shared
// memory; the grid team goes through global memory.  `fin` runs on thread 0 with the totals
// before the last block barrier (`nact`: the first threads that hold values; the others' are not
// read): scalars derived from them are computed once and read from
// shared memory (a square root that all eight warps repeat costs 2500 cycles).
static_assert(NT == 256, "team_reduce assumes 256 threads per CTA");
__shared__ double s_all[4][NT];
__shared__ double s_recv[2][16][4];  // [parity][source rank][value] (cluster teams, <= 16 CTAs)
template <int NV>
__device__ __noinline__ void team_total(Team& tm, const double* v, double* tot, int nact) {  // totals on warp 0
  static_assert(NV <= 4, "up to four values");
  constexpr int NB = NV == 1 ? 1 : (NV == 2 ? 2 : 4);  // values of the butterfly
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rows = (min(nact, NT) + 31) >> 5;  // warps with values: four or all of them are added
  if (warp < (rows <= 4 ? 4 : 8))
#pragma unroll
    for (int i = 0; i < NV; ++i) s_all[i][threadIdx.x] = v[i];
  __syncthreads();
  double t[NB];
#pragma unroll
  for (int i = 0; i < NB; ++i) t[i] = 0.0;
  if (warp == 0) {  // this CTA's totals
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const double* a = s_all[i];
      if (rows <= 1)
        t[i] = a[lane];
      else if (rows <= 2)
        t[i] = a[lane] + a[lane + 32];
      else
        t[i] = (a[lane] + a[lane + 32]) + (a[lane + 64] + a[lane + 96]);
      if (rows > 4) t[i] += (a[lane + 128] + a[lane + 160]) + (a[lane + 192] + a[lane + 224]);
    }
    const double r = warp_reduce_t<NB>(t);
#pragma unroll
    for (int i = 0; i < NV; ++i) tot[i] = __shfl_sync(0xffffffffu, r, i * (32 / NB));
  }
  if (tm.kind == TEAM_CLUSTER) {
    if (tm.size > 1) {
      cg::cluster_group cl = cg::this_cluster();
      if (warp == 0 && lane < tm.size) {
        double* dst = cl.map_shared_rank(&s_recv[tm.parity][tm.rank][0], lane);
#pragma unroll
        for (int i = 0; i < NV; ++i) dst[i] = tot[i];
      }
      cl.sync();
      if (warp == 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) t[i] = lane < tm.size ? s_recv[tm.parity][lane][i] : 0.0;
        const double r = warp_reduce_t<NB>(t);
#pragma unroll
        for (int i = 0; i < NV; ++i) tot[i] = __shfl_sync(0xffffffffu, r, i * (32 / NB));
      }
    }
  } else {
    double* buf = tm.red + (long long)tm.parity * tm.red_stride;
    if (threadIdx.x == 0)
#pragma unroll
      for (int i = 0; i < NV; ++i) buf[tm.rank * 4 + i] = tot[i];
    team_sync(tm);
    if (warp == 0) {
#pragma unroll
      for (int i = 0; i < NB; ++i) t[i] = 0.0;
      for (int r = lane; r < tm.size; r += 32)
#pragma unroll
        for (int i = 0; i < NV; ++i) t[i] += buf[r * 4 + i];
      const double r = warp_reduce_t<NB>(t);
#pragma unroll
      for (int i = 0; i < NV; ++i) tot[i] = __shfl_sync(0xffffffffu, r, i * (32 / NB));
    }
  }
  tm.parity ^= 1;
}
template <int NV, typename F>
__device__ __forceinline__ void team_reduce(Team& tm, const double* v, F&& fin, int nact = NT) {
  double tot[NV];
  team_total<NV>(tm, v, tot, nact);
  if (threadIdx.x == 0) fin(tot);
  __syncthreads();
}

// Multi-value all-reduce: every CTA has written nval partial doubles at
// part[rank * nval ...] (in the current parity buffer); after the call out[k]
// holds the fixed-order sum over CTAs, written by exactly one thread of the team.
// The caller must team_sync before reading `out` from other CTAs.
__device__ double* team_partials(Team& tm) { return tm.red + (long long)tm.parity * tm.red_stride; }

__device__ void team_finish_multi(Team& tm, int nval, double* out, double scale) {
  team_sync(tm);
  double* buf = team_partials(tm);
  for (int k = tm.gtid(); k < nval; k += tm.nthr()) {
    double s = 0;
    for (int r = 0; r < tm.size; ++r) s += buf[(long long)r * nval + k];
    out[k] = s * scale;
  }
  tm.parity ^= 1;
  team_sync(tm);
}

// ------------------------------------------------------------------ sum-of-products apply
// Position decomposition of flat index idx along leg l.
struct LegPos {
  long long base;  // idx - i * stride
  int i;
};
__device__ __forceinline__ LegPos leg_pos(const NodeDesc& nd, int l, long long idx) {
  const int st = nd.strides[l], D = nd.dims[l];
  const int n = (int)idx;
  const int q = fdivu(n, st, nd.inv_strides[l]);
  const int i = q - fdivu(q, D, nd.inv_dims[l]) * D;
  return LegPos{(long long)(n - i * st), i};
}

// y_i = sum_k M[i][k] x[base + k*stride] with four independent accumulators.  M is a row
// of a dims x dims matrix, either staged in shared memory (compute type) or in the pool.
template <typename T, typename MT, typename XT>
__device__ __forceinline__ typename C2<T>::t mode_dot(const MT* row, int D, const XT* x, long long base, int stride) {
  using V = typename C2<T>::t;
  V a0, a1, a2, a3;
  a0.x = a0.y = a1.x = a1.y = a2.x = a2.y = a3.x = a3.y = (T)0;
  const XT* xp = x + base;
  int k = 0;
  for (; k + 3 < D; k += 4) {
    const V m0 = cvt<T>(row[k]), m1 = cvt<T>(row[k + 1]), m2 = cvt<T>(row[k + 2]), m3 = cvt<T>(row[k + 3]);
    const V x0 = cvt<T>(xp[(long long)k * stride]), x1 = cvt<T>(xp[(long long)(k + 1) * stride]);
    const V x2 = cvt<T>(xp[(long long)(k + 2) * stride]), x3 = cvt<T>(xp[(long long)(k + 3) * stride]);
    cmac<T>(a0, m0, x0);
    cmac<T>(a1, m1, x1);
    cmac<T>(a2, m2, x2);
    cmac<T>(a3, m3, x3);
  }
  for (; k < D; ++k) cmac<T>(a0, cvt<T>(row[k]), cvt<T>(xp[(long long)k * stride]));
  a0.x += a1.x + (a2.x + a3.x);
  a0.y += a1.y + (a2.y + a3.y);
  return a0;
}

// Staging of one op's operands in shared memory.  Every node's operators (the
// environment blocks flowing into it and its constant operators) are contiguous in the
// pool, so an op stages one or two regions with asynchronous copies (cp.async), plus its
// term list; a factor's shared-memory slot is its offset inside the staged regions.  The
// matrices are staged in the compute type: FP64 from the pool, or FP32 from its mirror.
extern __shared__ __align__(16) unsigned char dyn_smem[];

// operator data in the compute type: the FP64 pool, or its FP32 mirror
template <typename T>
__device__ __forceinline__ const typename C2<T>::t* ops(const KernelParams& P);
template <>
__device__ __forceinline__ const double2* ops<double>(const KernelParams& P) { return P.pool; }
template <>
__device__ __forceinline__ const float2* ops<float>(const KernelParams& P) { return P.pool32; }

struct OpStage {
  Term terms[TTNS_MAX_TERMS];
  Factor chans[16];
  long long a_off, b_off;  // pool offsets of the staged regions
  int a_n, b_n;            // staged elements of each (a prefix when the region is larger)
  int end;                 // first free double2 of the dynamic shared memory
};

// one staging record per CTA, shared by every op (ops run one at a time)
__shared__ OpStage s_os;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T>
__device__ void stage_op(const KernelParams& P, const Instr& I, const TermList& L, const Factor* chans, int nchan,
                         OpStage& os) {
  // half of the dynamic shared memory for matrices (in the compute type), half for vectors
  using V = typename C2<T>::t;
  const long long cap = P.smem_bytes / (long long)sizeof(V) / 2;
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long an = I.rega_len < cap ? I.rega_len : cap;
    const long long rest = cap - an;
    const long long bn = I.regb_len < rest ? I.regb_len : rest;
    os.a_off = I.rega_off;
    os.b_off = I.regb_off;
    os.a_n = (int)an;
    os.b_n = (int)bn;
    // end of the staged matrices in 16-byte units, rounded up to 32 bytes
    const long long bytes = (an + bn) * (long long)sizeof(V);
    os.end = (int)((((bytes + 15) / 16) + 1) & ~1LL);
  }
  const int nt = L.count < TTNS_MAX_TERMS ? L.count : TTNS_MAX_TERMS;
  for (int t = threadIdx.x; t < nt; t += NT) os.terms[t] = P.terms[L.first + t];
  for (int b = threadIdx.x; b < nchan && b < 16; b += NT) os.chans[b] = chans[b];
  __syncthreads();
  if constexpr (std::is_same<T, double>::value) {
    double2* sm = reinterpret_cast<double2*>(dyn_smem);
    for (int k = threadIdx.x; k < os.a_n; k += NT) cp_async16(sm + k, P.pool + os.a_off + k);
    for (int k = threadIdx.x; k < os.b_n; k += NT) cp_async16(sm + os.a_n + k, P.pool + os.b_off + k);
    cp_async_wait_all();
  } else {
    // from the FP32 mirror (a double -> float conversion per element would run on the FP64
    // pipe) with asynchronous 8-byte copies: every copy of a thread is in flight at once
    float2* sm = reinterpret_cast<float2*>(dyn_smem);
    for (int k = threadIdx.x; k < os.a_n; k += NT) cp_async8(sm + k, P.pool32 + os.a_off + k);
    for (int k = threadIdx.x; k < os.b_n; k += NT) cp_async8(sm + os.a_n + k, P.pool32 + os.b_off + k);
    cp_async_wait_all();
  }
  __syncthreads();
}

// shared-memory position of n pool elements starting at pool offset off, or -1
__device__ __forceinline__ int staged_at(const OpStage& os, long long off, long long n) {
  long long e = off - os.a_off;
  if (e >= 0 && e + n <= os.a_n) return (int)e;
  e = off - os.b_off;
  if (e >= 0 && e + n <= os.b_n) return os.a_n + (int)e;
  return -1;
}

__device__ __forceinline__ int fslot(const OpStage& os, const Factor& f, int D) {
  const long long need = (long long)D * D;
  long long e = f.mat - os.a_off;
  if (e >= 0 && e + need <= os.a_n) return (int)e;
  e = f.mat - os.b_off;
  if (e >= 0 && e + need <= os.b_n) return os.a_n + (int)e;
  return -1;
}

// Input vector staged in shared memory (compute type) after the matrices, when it fits.
template <typename T>
__device__ typename C2<T>::t* vec_smem(const KernelParams& P, const OpStage& os, long long N) {
  using V = typename C2<T>::t;
  const long long avail = P.smem_bytes - (long long)os.end * (long long)sizeof(double2);
  if (N * (long long)sizeof(V) > avail) return nullptr;
  return reinterpret_cast<V*>(dyn_smem + (long long)os.end * sizeof(double2));
}

template <typename T>
__device__ void stage_vector(typename C2<T>::t* dst, const double2* src, long long N) {
  __syncthreads();
  long long k = threadIdx.x;
  for (; k + 3 * NT < N; k += 4 * NT) {  // four independent loads in flight per thread
    const double2 a = src[k], b = src[k + NT], c = src[k + 2 * NT], d = src[k + 3 * NT];
    dst[k] = cvt<T>(a);
    dst[k + NT] = cvt<T>(b);
    dst[k + 2 * NT] = cvt<T>(c);
    dst[k + 3 * NT] = cvt<T>(d);
  }
  for (; k < N; k += NT) dst[k] = cvt<T>(src[k]);
  __syncthreads();
}

// A compute-type vector copied into shared memory with asynchronous copies.
__device__ void stage_copy(float2* dst, const float2* src, long long N) {
  __syncthreads();
  for (long long k = threadIdx.x; k < N; k += NT) cp_async8(dst + k, src + k);
  cp_async_wait_all();
  __syncthreads();
}

// One factor applied at output idx: sum_k M[i][k] x[idx + (k - i) * stride] along the factor's leg.
template <typename T, typename XT>
__device__ __forceinline__ typename C2<T>::t factor_dot(const KernelParams& P, const NodeDesc& nd, const Factor& f,
                                                        const OpStage& os, const XT* x, long long idx) {
  const LegPos lp = leg_pos(nd, f.leg, idx);
  const int D = nd.dims[f.leg];
  if (f.nnz > 0) {
    using V = typename C2<T>::t;
    V acc;
    acc.x = acc.y = (T)0;
    const int sl = staged_at(os, f.sp, 2LL * D * f.nnz);
    if (sl >= 0) {  // the table staged with the node's operators, in the compute type
      const V* tab = reinterpret_cast<const V*>(dyn_smem) + sl;
      const V* vals = tab + lp.i * f.nnz;
      const V* cols = tab + D * f.nnz + lp.i * f.nnz;
      for (int e = 0; e < f.nnz; ++e) {
        const int k = (int)cols[e].x;
        cmac<T>(acc, vals[e], cvt<T>(x[lp.base + (long long)k * nd.strides[f.leg]]));
      }
      return acc;
    }
    const V* vals = ops<T>(P) + f.sp + (long long)lp.i * f.nnz;
    const V* cols = ops<T>(P) + f.sp + (long long)D * f.nnz + (long long)lp.i * f.nnz;
    for (int e = 0; e < f.nnz; ++e) {
      const int k = (int)cols[e].x;
      cmac<T>(acc, vals[e], cvt<T>(x[lp.base + (long long)k * nd.strides[f.leg]]));
    }
    return acc;
  }
  const int slot = fslot(os, f, D);
  if (slot >= 0) {  // staged in the compute type
    const typename C2<T>::t* sm = reinterpret_cast<const typename C2<T>::t*>(dyn_smem) + slot;
    return mode_dot<T>(sm + lp.i * D, D, x, lp.base, nd.strides[f.leg]);
  }
  return mode_dot<T>(ops<T>(P) + f.mat + (long long)lp.i * D, D, x, lp.base, nd.strides[f.leg]);
}

// Direct two-factor term at idx: the sparse factor's few entries, each times the dense
// factor applied at the shifted position.
template <typename T, typename XT>
__device__ __forceinline__ typename C2<T>::t direct_dot(const KernelParams& P, const NodeDesc& nd, const Term& T_,
                                                        const OpStage& os, const XT* x, long long idx) {
  using V = typename C2<T>::t;
  const Factor& sf = T_.f[T_.sparse_f];
  const Factor& df = T_.f[1 - T_.sparse_f];
  const LegPos lp = leg_pos(nd, sf.leg, idx);
  const int Ds = nd.dims[sf.leg];
  V acc;
  acc.x = acc.y = (T)0;
  const int sl = staged_at(os, sf.sp, 2LL * Ds * sf.nnz);
  if (sl >= 0) {  // staged table (compute type)
    const V* tab = reinterpret_cast<const V*>(dyn_smem) + sl;
    const V* vals = tab + lp.i * sf.nnz;
    const V* cols = tab + Ds * sf.nnz + lp.i * sf.nnz;
    for (int e = 0; e < sf.nnz; ++e) {
      const V v = vals[e];
      if (v.x == (T)0 && v.y == (T)0) continue;
      const long long idx2 = lp.base + (long long)((int)cols[e].x) * nd.strides[sf.leg];
      const V d = factor_dot<T>(P, nd, df, os, x, idx2);
      cmac<T>(acc, v, d);
    }
    return acc;
  }
  const V* vals = ops<T>(P) + sf.sp + (long long)lp.i * sf.nnz;
  const V* cols = ops<T>(P) + sf.sp + (long long)Ds * sf.nnz + (long long)lp.i * sf.nnz;
  for (int e = 0; e < sf.nnz; ++e) {
    const V v = vals[e];
    if (v.x == (T)0 && v.y == (T)0) continue;
    const long long idx2 = lp.base + (long long)((int)cols[e].x) * nd.strides[sf.leg];
    const V d = factor_dot<T>(P, nd, df, os, x, idx2);
    cmac<T>(acc, v, d);
  }
  return acc;
}

// Stage 1: tmp[t] = first factor of two-stage term t applied to x (tmp in the compute type)
template <typename T, typename XT>
__device__ void apply_stage1(const KernelParams& P, Team& tm, const NodeDesc& nd, const XT* x, const TermList& L,
                             typename C2<T>::t* tmp, long long tstride, const OpStage& os) {
  const int t0 = L.count - L.n2;
  const long long N = nd.size;
  for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
    for (int t = 0; t < L.n2; ++t) tmp[t * tstride + idx] = factor_dot<T>(P, nd, os.terms[t0 + t].f[0], os, x, idx);
  }
}

// Stage 2 value at idx: one-factor and direct terms on x, second factors on tmp
template <typename T, typename XT>
__device__ __forceinline__ typename C2<T>::t apply_stage2_at(const KernelParams& P, const NodeDesc& nd, const XT* x,
                                                            const TermList& L, const typename C2<T>::t* tmp,
                                                            long long tstride, long long idx, const OpStage& os) {
  typename C2<T>::t acc;
  acc.x = 0;
  acc.y = 0;
  const int n1 = L.count - L.n2 - L.nd;
  for (int t = 0; t < n1; ++t) {
    const auto a = factor_dot<T>(P, nd, os.terms[t].f[0], os, x, idx);
    acc.x += a.x;
    acc.y += a.y;
  }
  for (int t = n1; t < n1 + L.nd; ++t) {
    const auto a = direct_dot<T>(P, nd, os.terms[t], os, x, idx);
    acc.x += a.x;
    acc.y += a.y;
  }
  const int t0 = L.count - L.n2;
  for (int t = 0; t < L.n2; ++t) {
    const auto a = factor_dot<T>(P, nd, os.terms[t0 + t].f[1], os, tmp + t * tstride, idx);
    acc.x += a.x;
    acc.y += a.y;
  }
  return acc;
}

// Sum of nval doubles over the team, in a fixed order, identical on every CTA.  `mine`
// holds this CTA's partials in shared memory; store(k, sum) runs on one thread of every CTA.
// Cluster teams read the other CTAs' partials through distributed shared memory: callers
// alternate between two `mine` buffers, so that one cluster barrier per call suffices (a
// buffer is rewritten only after the next call's barrier, which every reader has passed).
// Grid teams go through the global partial buffers.
template <typename F>
__device__ __forceinline__ void team_reduce_vec(Team& tm, const double* mine, int nval, F&& store) {
  __syncthreads();
  if (tm.kind == TEAM_CLUSTER) {
    cg::cluster_group cl = cg::this_cluster();
    if (tm.size > 1) cl.sync();
    for (int k = threadIdx.x; k < nval; k += NT) {
      // the 16 peers' values loaded together, then added in a fixed tree (depth 4)
      double a[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) a[r] = r < tm.size ? *cl.map_shared_rank(mine + k, r) : 0.0;
#pragma unroll
      for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
        for (int r = 0; r < w; ++r) a[r] += a[r + w];
      store(k, a[0]);
    }
  } else {
    // grid team: each cluster first sums its CTAs' partials through distributed shared memory
    // (the values split over the cluster's CTAs, each value added in a fixed tree), the cluster
    // totals go to global memory, and after the grid barrier every CTA adds the few cluster
    // totals in a fixed order.  Every CTA computes the same sums.
    cg::cluster_group cl = cg::this_cluster();
    const int cs = tm.csize;
    const int crank = (int)cl.block_rank();
    const int cid = tm.rank / cs;
    const int ncl = tm.size / cs;
    double* buf = team_partials(tm);
    cl.sync();
    for (int k = crank * NT + threadIdx.x; k < nval; k += cs * NT) {
      double a[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) a[r] = r < cs ? *cl.map_shared_rank(mine + k, r) : 0.0;
#pragma unroll
      for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
        for (int r = 0; r < w; ++r) a[r] += a[r + w];
      buf[(long long)cid * nval + k] = a[0];
    }
    team_sync(tm);
    for (int k = threadIdx.x; k < nval; k += NT) {
      double s = 0.0;
      for (int c = 0; c < ncl; ++c) s += buf[(long long)c * nval + k];
      store(k, s);
    }
    tm.parity ^= 1;
  }
  __syncthreads();
}

#include "krylov.cuh"

// Tiled apply for grid-team nodes too large for shared memory.  The node (legs 0..nl-1, the
// last one physical) is covered twice by tiles:
//   pass A: tiles over legs h..nl-1 (contiguous blocks), one per index of legs 0..h-1;
//   pass B: tiles over legs 0..h-1 and nl-1, one per index of legs h..nl-2;
// with h = (nl - 1) / 2.  A term is computed in the pass whose tile holds all its legs, from
// the tile of the input vector staged in shared memory (every element of a tile is read by
// D of its neighbours along a leg: this replaces strided L2 reads).  Pass A writes its sum,
// pass B adds its terms to it.  A term with legs in neither tile keeps the element-wise apply.
//
// In FP32 a dense factor is a product over the fibres of its leg in the tile, a block of rows and
// fibres per thread (tile_product), and a two-factor term is that product followed by the other
// factor on its result: element by element the operand loads are the bound (two shared-memory
// or L2 words per multiply-add).  Root of a star of four chains (20^4 x 5, two of the couplings
// with three entries a row, which kept it from being tiled), whole grid, TF32X3 mode: 5760 us per
// exponential before, 3500 now (3250 with one accumulator).  In FP64 the FP64 pipe is the bound in
// either form (18.9 ms element by element, 20.5 by products), so there, and where three tiles
// (input, sum, product) do not fit in shared memory, a tile's terms are taken element by element,
// without two-stage terms.
struct TiledApply {
  NodeDesc ta, tb;                  // the tile tensors of the two passes
  int h;
  int lmapA[TTNS_MAX_LEGS], lmapB[TTNS_MAX_LEGS];  // tile leg of each node leg (-1: none)
  int nst[TTNS_MAX_LEGS];           // node strides of the tile-B legs 0..h-1
  int bdims[TTNS_MAX_LEGS], bst[TTNS_MAX_LEGS];    // legs h..nl-2: dims and node strides
  int nb;                           // number of such legs
  int nta, ntb;
  unsigned long long inB;           // bit t: term t is computed in pass B
  int ok;
};
__shared__ TiledApply s_tp;

__device__ void tiled_plan(const NodeDesc& nd, const OpStage& os, const TermList& L, TiledApply& tp) {
  const int nl = nd.nl, h = (nl - 1) / 2;
  tp.ok = 0;
  if (nl < 3 || h < 1 || L.count > 64) return;
  bool ok = true;
  tp.h = h;
  NodeDesc& a = tp.ta;
  a.nl = nl - h;
  for (int q = 0; q < a.nl; ++q) {
    a.dims[q] = nd.dims[h + q];
    a.strides[q] = nd.strides[h + q];
  }
  a.size = nd.strides[h - 1];
  NodeDesc& b = tp.tb;
  b.nl = h + 1;
  for (int q = 0; q < h; ++q) b.dims[q] = nd.dims[q];
  b.dims[h] = nd.dims[nl - 1];
  b.strides[h] = 1;
  for (int q = h - 1; q >= 0; --q) b.strides[q] = b.strides[q + 1] * b.dims[q + 1];
  b.size = b.strides[0] * b.dims[0];
  for (int q = 0; q < a.nl; ++q) {
    a.inv_dims[q] = 1.0f / (float)a.dims[q];
    a.inv_strides[q] = 1.0f / (float)a.strides[q];
  }
  for (int q = 0; q < b.nl; ++q) {
    b.inv_dims[q] = 1.0f / (float)b.dims[q];
    b.inv_strides[q] = 1.0f / (float)b.strides[q];
  }
  for (int l = 0; l < TTNS_MAX_LEGS; ++l) {
    tp.lmapA[l] = (l >= h && l < nl) ? l - h : -1;
    tp.lmapB[l] = l < h ? l : (l == nl - 1 ? h : -1);
  }
  for (int q = 0; q < h; ++q) tp.nst[q] = nd.strides[q];
  tp.nb = nl - 1 - h;
  for (int q = 0; q < tp.nb; ++q) {
    tp.bdims[q] = nd.dims[h + q];
    tp.bst[q] = nd.strides[h + q];
  }
  tp.nta = (int)(nd.size / a.size);
  tp.ntb = (int)(nd.size / b.size);
  tp.inB = 0ull;
  for (int t = 0; t < L.count; ++t) {
    const Term& tt = os.terms[t];
    bool allA = true, allB = true;
    for (int k = 0; k < tt.nf; ++k) {
      allA = allA && tp.lmapA[tt.f[k].leg] >= 0;
      allB = allB && tp.lmapB[tt.f[k].leg] >= 0;
    }
    if (!allA) {
      if (allB) tp.inB |= 1ull << t;
      else ok = false;
    }
    if (tt.nf == 2 && tt.f[0].nnz > 0 && tt.f[1].nnz > 0) ok = false;
  }
  tp.ok = ok;
}

// out (+)= M x along one leg of a tile of TT elements: dimension D, stride st; TA rows times TC
// fibres per thread.
template <typename T, int TA, int TC>
__device__ __forceinline__ void tile_rows(const typename C2<T>::t* M, int D, int st, float inv_st, int TT,
                                          const typename C2<T>::t* x, typename C2<T>::t* out, bool add) {
  using V = typename C2<T>::t;
  const int nc = TT / D, ncg = (nc + TC - 1) / TC, nrg = (D + TA - 1) / TA;
  const float inv_g = 1.0f / (float)ncg;
  for (int it = threadIdx.x; it < nrg * ncg; it += NT) {
    const int rg = fdivu(it, ncg, inv_g), c0 = it - rg * ncg, i0 = rg * TA;
    int base[TC];
    constexpr int U = TA * TC > 4 ? 2 : 4;  // (more would spill)
    const V* row[TA];
    V acc[TA][TC][U];
#pragma unroll
    for (int q = 0; q < TC; ++q) {
      const int c = min(c0 + q * ncg, nc - 1), hi = fdivu(c, st, inv_st);
      base[q] = hi * D * st + c - hi * st;
    }
#pragma unroll
    for (int i = 0; i < TA; ++i) {
      row[i] = M + min(i0 + i, D - 1) * D;
#pragma unroll
      for (int q = 0; q < TC; ++q)
#pragma unroll
        for (int u = 0; u < U; ++u) acc[i][q][u].x = acc[i][q][u].y = (T)0;
    }
    auto step = [&](int k, int u) {
      V m[TA], v[TC];
#pragma unroll
      for (int i = 0; i < TA; ++i) m[i] = row[i][k];
#pragma unroll
      for (int q = 0; q < TC; ++q) v[q] = x[base[q] + k * st];
#pragma unroll
      for (int i = 0; i < TA; ++i)
#pragma unroll
        for (int q = 0; q < TC; ++q) cmac<T>(acc[i][q][u], m[i], v[q]);
    };
    int k = 0;
    for (; k + 3 < D; k += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) step(k + u, u % U);
    }
    for (; k < D; ++k) step(k, 0);
#pragma unroll
    for (int i = 0; i < TA; ++i)
#pragma unroll
      for (int q = 0; q < TC; ++q)
        if (i0 + i < D && c0 + q * ncg < nc) {
          V* o = out + base[q] + (i0 + i) * st;
          V r = sum_parts<U>(acc[i][q]);
          if (add) {
            r.x += o->x;
            r.y += o->y;
          }
          *o = r;
        }
  }
}
// The block with the fewest operand loads per thread (rounds x (rows + fibres)): 4 x 2 at D 20 and
// 5 D^2 elements, 2 x 2 at D 14 (one round instead of four of single elements).
template <typename T>
__device__ __noinline__ void tile_product(const KernelParams& P, const NodeDesc& td, const OpStage& os, const Factor& f,
                                          int leg, const typename C2<T>::t* x, typename C2<T>::t* out, bool add) {
  using V = typename C2<T>::t;
  const int D = td.dims[leg], st = td.strides[leg], TT = td.size;
  const int slot = fslot(os, f, D);
  const V* M = slot >= 0 ? reinterpret_cast<const V*>(dyn_smem) + slot : ops<T>(P) + f.mat;
  const float inv_st = td.inv_strides[leg];
  const int nc = TT / D, nc2 = (nc + 1) / 2;
  auto loads = [](int items, int per) { return (items + NT - 1) / NT * per; };
  const int l1 = loads(TT, 2), l2 = loads((D + 1) / 2 * nc2, 4), l4 = loads((D + 3) / 4 * nc2, 6);
  if (l4 < l2 && l4 < l1)
    tile_rows<T, 4, 2>(M, D, st, inv_st, TT, x, out, add);
  else if (l2 < l1)
    tile_rows<T, 2, 2>(M, D, st, inv_st, TT, x, out, add);
  else
    tile_rows<T, 1, 1>(M, D, st, inv_st, TT, x, out, add);
}

// Shared memory of the tiled apply, or nullptr: three tiles (fibres), or the input tile alone
// for lists without two-stage terms.  The same on every CTA.  any: with fewer tiles than CTAs too.
// The plan is shared: the barrier before it waits for the readers of an earlier one (an
// exponential may ask twice), and a caller that changes `os` afterwards needs one of its own.
template <typename T>
__device__ typename C2<T>::t* tiled_begin(const KernelParams& P, const Team& tm, const NodeDesc& nd, const OpStage& os,
                                          const TermList& L, bool any, bool& tiled, bool& fibres) {
  TiledApply& tp = s_tp;
  __syncthreads();
  if (threadIdx.x == 0) tiled_plan(nd, os, L, tp);
  __syncthreads();
  tiled = fibres = false;
  if (!tp.ok || (!any && (std::is_same<T, double>::value || min(tp.nta, tp.ntb) < tm.size))) return nullptr;
  const int TT = tp.ta.size > tp.tb.size ? tp.ta.size : tp.tb.size;
  typename C2<T>::t* xt = nullptr;
  if constexpr (!std::is_same<T, double>::value) xt = vec_smem<T>(P, os, 3LL * TT);
  fibres = xt != nullptr;
  if (!fibres && L.n2 == 0) xt = vec_smem<T>(P, os, TT);
  tiled = xt != nullptr;
  return xt;
}

// One pass over this CTA's tiles; emit(global index, sum of the pass's terms at it).  xt: the
// input tile, with `fibres` followed by the tile's sum and a factor's result.
template <typename T, typename F>
__device__ void tiled_pass(const KernelParams& P, Team& tm, const TiledApply& tp, const OpStage& os,
                           const TermList& L, const typename C2<T>::t* xin, typename C2<T>::t* xt, bool fibres,
                           int pass, F&& emit) {
  using V = typename C2<T>::t;
  const NodeDesc& td = pass ? tp.tb : tp.ta;
  const int* lmap = pass ? tp.lmapB : tp.lmapA;
  const int ntiles = pass ? tp.ntb : tp.nta;
  const int TT = td.size;
  const int h = tp.h;
  auto gidx = [&](long long base, int e) -> long long {
    if (!pass) return base + e;
    long long g = base;
    int rem = e;
    for (int q = 0; q < h; ++q) {
      const int iq = fdivu(rem, td.strides[q], td.inv_strides[q]);
      rem -= iq * td.strides[q];
      g += (long long)iq * tp.nst[q];
    }
    return g + rem;  // the physical leg has node stride 1
  };
  for (int tile = tm.rank; tile < ntiles; tile += tm.size) {
    long long base;
    if (!pass) {
      base = (long long)tile * TT;
    } else {
      base = 0;
      int rem = tile;
      for (int q = tp.nb - 1; q >= 0; --q) {
        const int iq = rem % tp.bdims[q];
        rem /= tp.bdims[q];
        base += (long long)iq * tp.bst[q];
      }
    }
    __syncthreads();  // the previous tile's reads are done
    for (int e = threadIdx.x; e < TT; e += NT) {
      if constexpr (sizeof(V) == 16)
        cp_async16(xt + e, xin + gidx(base, e));
      else
        cp_async8(xt + e, xin + gidx(base, e));
    }
    cp_async_wait_all();
    __syncthreads();
    if constexpr (!std::is_same<T, double>::value) if (fibres) {
      V* y = xt + TT;
      V* z = y + TT;
      for (int e = threadIdx.x; e < TT; e += NT) {  // terms of one sparse factor
        V acc;
        acc.x = acc.y = (T)0;
        for (int t = 0; t < L.count; ++t) {
          if ((int)((tp.inB >> t) & 1ull) != pass || os.terms[t].nf != 1 || os.terms[t].f[0].nnz == 0) continue;
          Factor f = os.terms[t].f[0];
          f.leg = lmap[f.leg];
          const V a = factor_dot<T>(P, td, f, os, xt, e);
          acc.x += a.x;
          acc.y += a.y;
        }
        y[e] = acc;
      }
      __syncthreads();
      for (int t = 0; t < L.count; ++t) {
        const Term& tt = os.terms[t];
        if ((int)((tp.inB >> t) & 1ull) != pass) continue;
        if (tt.nf == 1) {
          if (tt.f[0].nnz > 0) continue;
          tile_product<T>(P, td, os, tt.f[0], lmap[tt.f[0].leg], xt, y, true);
          __syncthreads();
          continue;
        }
        const int d = tt.f[0].nnz == 0 ? 0 : 1;  // a dense factor first (tiled_plan: there is one)
        tile_product<T>(P, td, os, tt.f[d], lmap[tt.f[d].leg], xt, z, false);
        __syncthreads();
        Factor f = tt.f[1 - d];
        f.leg = lmap[f.leg];
        if (f.nnz == 0)
          tile_product<T>(P, td, os, f, f.leg, z, y, true);
        else
          for (int e = threadIdx.x; e < TT; e += NT) {
            const V a = factor_dot<T>(P, td, f, os, z, e);
            y[e].x += a.x;
            y[e].y += a.y;
          }
        __syncthreads();
      }
      for (int e = threadIdx.x; e < TT; e += NT) emit(gidx(base, e), y[e]);
      continue;
    }
    for (int e = threadIdx.x; e < TT; e += NT) {
      V acc;
      acc.x = acc.y = (T)0;
      for (int t = 0; t < L.count; ++t) {
        if ((int)((tp.inB >> t) & 1ull) != pass) continue;
        Term tt = os.terms[t];
        tt.f[0].leg = lmap[tt.f[0].leg];
        if (tt.nf == 2) tt.f[1].leg = lmap[tt.f[1].leg];
        const V a = tt.nf == 1 ? factor_dot<T>(P, td, tt.f[0], os, xt, e) : direct_dot<T>(P, td, tt, os, xt, e);
        acc.x += a.x;
        acc.y += a.y;
      }
      emit(gidx(base, e), acc);
    }
  }
}

// ------------------------------------------------------------------ tensor-core apply
// H_eff v for a node whose terms have at most one dense factor each (no dense x dense term):
// the terms are grouped by the leg l their dense factor acts on, and every group is one complex
// GEMM on the tensor cores,
//   Y_l[r][i] = sum_{t in group, k} z_t[r][k] M_t[i][k],
// with rows r = the node index with leg l removed, k the index of leg l, z_t = x with the
// term's row-sparse factor (a, a^+, a diagonal or sparse pattern on another leg) applied while
// the operand is staged, and M_t the term's dense matrix (an environment block or a dense
// constant operator).  A task is one group and one tile of 128 rows; K is taken in chunks of at
// most 32 complex values (64 real), so any leg dimension up to 64 fits the shared memory.  The
// result of group g goes to its own compute-type buffer; the terms outside every group (a
// row-sparse factor alone, or a dense factor on a leg below 8) stay on the SIMT path in the pass
// that sums the groups (tc_sum_at).
struct TcPlan {
  int ok;
  int ngroups;
  int gleg[TTNS_MAX_LEGS];
  int gfirst[TTNS_MAX_LEGS + 1];   // terms of group g: gterm[gfirst[g] .. gfirst[g + 1])
  int gterm[TTNS_MAX_TERMS];
  int gdense[TTNS_MAX_TERMS];      // index of the dense factor of each grouped term
  int nsimt;
  int simt[TTNS_MAX_TERMS];        // terms evaluated element-wise
  int gtask0[TTNS_MAX_LEGS + 1];   // first task of group g (tasks of g: K parts x row tiles)
  int gtiles[TTNS_MAX_LEGS];       // row tiles of group g
  int gkpart[TTNS_MAX_LEGS];       // complex K per part (whole chunks)
  int gslot0[TTNS_MAX_LEGS + 1];   // first result slot of group g (one slot per K part)
  float inv_st[TTNS_MAX_LEGS];
};
__shared__ TcPlan s_tcp;

struct TcState {
  uint64_t mbar;
  uint32_t tmem;
  uint32_t phase;
  int on;
};
__shared__ TcState s_tc;

constexpr int kTcRows = 128;   // rows per task (the MMA's M)
constexpr int kTcTmemCols = 512;  // all of an SM's tensor memory (one CTA per SM)
constexpr int kTcSlots = 16;      // compute-type result vectors in the workspace

// Groups, and each group's K (term, leg index) split into parts of whole chunks, one result
// slot per part, so that the tasks (group, part, row tile) run on more CTAs and each runs
// fewer chunks one after another.  ksc: complex K per MMA K step of the precision in use.
__device__ void tc_plan(const NodeDesc& nd, const OpStage& os, const TermList& L, int ksc, TcPlan& tp) {
  tp.ok = 0;
  if (L.n2 > 0 || L.count > TTNS_MAX_TERMS) return;
  int dleg[TTNS_MAX_TERMS], dfac[TTNS_MAX_TERMS];
  for (int t = 0; t < L.count; ++t) {
    const Term& T = os.terms[t];
    dleg[t] = -1;
    dfac[t] = -1;
    if (T.nf == 1) {
      if (T.f[0].nnz == 0 && nd.dims[T.f[0].leg] >= 8) { dleg[t] = T.f[0].leg; dfac[t] = 0; }
    } else if (T.sparse_f >= 0) {
      const int d = 1 - T.sparse_f;
      if (T.f[d].nnz == 0 && nd.dims[T.f[d].leg] >= 8) { dleg[t] = T.f[d].leg; dfac[t] = d; }
    }
  }
  tp.ngroups = 0;
  tp.nsimt = 0;
  int nt = 0;
  for (int l = 0; l < nd.nl; ++l) {
    int c = 0;
    for (int t = 0; t < L.count; ++t) c += dleg[t] == l;
    if (c == 0) continue;
    const int g = tp.ngroups++;
    tp.gleg[g] = l;
    tp.gfirst[g] = nt;
    tp.inv_st[g] = 1.0f / (float)nd.strides[l];
    for (int t = 0; t < L.count; ++t)
      if (dleg[t] == l) { tp.gterm[nt] = t; tp.gdense[nt] = dfac[t]; ++nt; }
  }
  tp.gfirst[tp.ngroups] = nt;
  int ntask = 0, nslot = 0;
  const int cap = tp.ngroups > 0 ? max(1, kTcSlots / tp.ngroups) : 1;
  for (int g = 0; g < tp.ngroups; ++g) {
    const int D = nd.dims[tp.gleg[g]];
    const int Npad = ((2 * D + 15) / 16) * 16;
    const int chunk_kc = min(8, kTcTmemCols / Npad) * ksc;
    const int nterm = tp.gfirst[g + 1] - tp.gfirst[g];
    const int ktot = ((nterm * D + ksc - 1) / ksc) * ksc;
    const int nchunk = (ktot + chunk_kc - 1) / chunk_kc;
    int parts = min(nchunk, cap);
    const int cpp = (nchunk + parts - 1) / parts;  // chunks per part
    parts = (nchunk + cpp - 1) / cpp;
    tp.gkpart[g] = cpp * chunk_kc;
    tp.gtiles[g] = (nd.size / D + kTcRows - 1) / kTcRows;
    tp.gtask0[g] = ntask;
    tp.gslot0[g] = nslot;
    ntask += parts * tp.gtiles[g];
    nslot += parts;
  }
  tp.gtask0[tp.ngroups] = ntask;
  tp.gslot0[tp.ngroups] = nslot;
  for (int t = 0; t < L.count; ++t)
    if (dleg[t] < 0) tp.simt[tp.nsimt++] = t;
  tp.ok = tp.ngroups > 0;
}

// value of z = (row-sparse factor fs, if any) x at idx, in the compute type
template <typename T, typename XT>
__device__ __forceinline__ typename C2<T>::t tc_z(const KernelParams& P, const NodeDesc& nd, const Factor* fs,
                                                  const XT* x, long long idx) {
  if (!fs) return cvt<T>(x[idx]);
  using V = typename C2<T>::t;
  const LegPos lp = leg_pos(nd, fs->leg, idx);
  const int D = nd.dims[fs->leg];
  const V* vals = ops<T>(P) + fs->sp + (long long)lp.i * fs->nnz;
  const V* cols = ops<T>(P) + fs->sp + (long long)D * fs->nnz + (long long)lp.i * fs->nnz;
  V acc;
  acc.x = acc.y = (T)0;
  for (int e = 0; e < fs->nnz; ++e) {
    const int k = (int)cols[e].x;
    cmac<T>(acc, vals[e], cvt<T>(x[lp.base + (long long)k * nd.strides[fs->leg]]));
  }
  return acc;
}

// One task (group g, row tile rt).  K runs over (term, leg index) of the group's terms back to
// back; it is staged in chunks of n_acc MMA K steps, every K step accumulates into its own TMEM
// columns (the tensor core's accumulation rounds toward zero, so a long accumulation drifts),
// and the steps are summed in shared memory in FP32 round-to-nearest, in a fixed order.  The
// operand loads of a thread are issued together (four items at a time) before any is
// converted, so their latencies overlap.  Returns false if a completion wait gave up (the
// status word is set).
template <int KIND, typename T, typename XT>
__device__ __noinline__ bool tc_task(const KernelParams& P, const NodeDesc& nd, const OpStage& os, const TcPlan& tp, int g,
                        int part, int rt, const XT* x, typename C2<T>::t* yg, bool prof) {
  PhaseClock pc;  // phases 20-23 (grid counters): operand staging, MMA completion, read-back, write
  pc.start(prof && threadIdx.x == 0, true);
  using S = tc::Split<KIND>;
  using V = typename C2<T>::t;
  TcState& ts = s_tc;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l = tp.gleg[g];
  const int D = nd.dims[l];
  const int st = nd.strides[l];
  const int rows = nd.size / D;
  const int r0 = rt * kTcRows;
  const int Npad = ((2 * D + 15) / 16) * 16;
  const int nterm = tp.gfirst[g + 1] - tp.gfirst[g];
  constexpr int G = 8 / S::esize;                // complex values per 16-byte core row
  constexpr int KSC = S::kstep / 2;              // complex K per MMA K step
  const int n_acc = min(8, kTcTmemCols / Npad);   // K steps per chunk, one TMEM slot each
  const int chunk_kc = n_acc * KSC;
  const int ktot = ((nterm * D + KSC - 1) / KSC) * KSC;
  const int ldsum = Npad + 1;
  float* sums = reinterpret_cast<float*>(dyn_smem);
  const uint32_t a_plane = (uint32_t)kTcRows * 2 * chunk_kc * S::esize;
  const uint32_t b_plane = (uint32_t)Npad * 2 * chunk_kc * S::esize;
  const uint32_t sum_bytes = ((uint32_t)kTcRows * ldsum * 4u + 1023u) & ~1023u;
  unsigned char* A = dyn_smem + sum_bytes;
  unsigned char* B = A + S::parts * a_plane;
  // this thread's share of the accumulator: row (TMEM lane) and half of the columns
  const int q4 = warp & 3, half = warp >> 2;
  const int my_row = q4 * 32 + lane;
  const int c_lo = half * (Npad / 2), c_hi = c_lo + Npad / 2;
  for (int c = c_lo; c < c_hi; ++c) sums[my_row * ldsum + c] = 0.0f;
  // Sparse factors with one entry per row (a, a^+, a diagonal): their tables go to shared
  // memory after the operand planes, so that every z of a batch is one independent load of x
  // (else each z would chain a table load and an x load).  Other groups keep tc_z.
  struct SpHdr {
    int sp, leg, st, D;
    float inv_st, inv_D;
    int off, pad;
  };
  unsigned char* tail = B + S::parts * b_plane;
  SpHdr* hdr = reinterpret_cast<SpHdr*>(tail);
  const long long tail_off = (long long)(tail - dyn_smem);
  bool fast = nterm <= TTNS_MAX_TERMS;
  int ntab = 0;
  for (int tl = 0; tl < nterm && fast; ++tl) {
    const int q = tp.gfirst[g] + tl;
    const Term& T_ = os.terms[tp.gterm[q]];
    if (T_.nf == 2) {
      const Factor& f = T_.f[1 - tp.gdense[q]];
      if (f.nnz != 1) fast = false;
      ntab += nd.dims[f.leg];
    }
  }
  const long long hdr_bytes = ((long long)nterm * sizeof(SpHdr) + 15) & ~15LL;
  float2* tvals = reinterpret_cast<float2*>(tail + hdr_bytes);
  int* tcols = reinterpret_cast<int*>(tvals + ntab);
  fast = fast && tail_off + hdr_bytes + (long long)ntab * 12 <= P.smem_bytes;
  if (fast) {
    int off = 0;
    for (int tl = 0; tl < nterm; ++tl) {  // every thread walks the same terms
      const int q = tp.gfirst[g] + tl;
      const Term& T_ = os.terms[tp.gterm[q]];
      SpHdr h{};
      if (T_.nf == 2) {
        const Factor& f = T_.f[1 - tp.gdense[q]];
        h.sp = 1;
        h.leg = f.leg;
        h.st = nd.strides[f.leg];
        h.D = nd.dims[f.leg];
        h.inv_st = nd.inv_strides[f.leg];
        h.inv_D = nd.inv_dims[f.leg];
        h.off = off;
        for (int i = tid; i < h.D; i += NT) {
          tvals[off + i] = P.pool32[f.sp + i];
          tcols[off + i] = (int)P.pool32[f.sp + h.D + i].x;
        }
        off += h.D;
      }
      if (tid == 0) hdr[tl] = h;
    }
    __syncthreads();
  }
  bool ok = true;
  const int kbeg = part * tp.gkpart[g];
  const int kend = min(ktot, kbeg + tp.gkpart[g]);
  for (int kc0 = kbeg; kc0 < kend && ok; kc0 += chunk_kc) {
    const int nk = min(chunk_kc, kend - kc0);   // a multiple of KSC
    const int Kr = 2 * nk;
    // A: rows of the tile x (term, k) of the chunk
    if (fast) {
      const int per_row = nk / G;
      const int nitems = kTcRows * per_row;
      for (int it0 = tid; it0 < nitems; it0 += 4 * NT) {
        long long xi[4][G];
        V cv[4][G];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int item = it0 + u * NT;
          const int row = item % kTcRows, kq = item / kTcRows;
          const int R = r0 + row;
          const bool in = item < nitems && R < rows;
          long long base = 0;
          if (in) {
            const int outer = fdivu(R, st, tp.inv_st[g]);
            base = (long long)outer * D * st + (R - outer * st);
          }
#pragma unroll
          for (int j = 0; j < G; ++j) {
            const int kg = kc0 + kq * G + j;
            xi[u][j] = -1;
            cv[u][j].x = (T)1;
            cv[u][j].y = (T)0;
            if (in && kg < nterm * D) {
              const int tl = kg / D, kk = kg - tl * D;
              const int el = (int)(base + (long long)kk * st);
              const SpHdr h = hdr[tl];
              if (h.sp) {
                const int qq = fdivu(el, h.st, h.inv_st);
                const int i = qq - fdivu(qq, h.D, h.inv_D) * h.D;
                xi[u][j] = (long long)(el - i * h.st) + (long long)tcols[h.off + i] * h.st;
                const float2 v = tvals[h.off + i];
                cv[u][j].x = (T)v.x;
                cv[u][j].y = (T)v.y;
              } else {
                xi[u][j] = el;
              }
            }
          }
        }
        V xv[4][G];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int j = 0; j < G; ++j) {
            if (xi[u][j] >= 0) {
              xv[u][j] = cvt<T>(x[xi[u][j]]);
            } else {
              xv[u][j].x = (T)0;
              xv[u][j].y = (T)0;
            }
          }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int item = it0 + u * NT;
          if (item >= nitems) break;
          const int row = item % kTcRows, kq = item / kTcRows;
#pragma unroll
          for (int j = 0; j < G; ++j) {
            V z;
            z.x = z.y = (T)0;
            cmac<T>(z, cv[u][j], xv[u][j]);
            tc::put_split_f<KIND>(A, a_plane, row, 2 * (kq * G + j), Kr, (float)z.x);
            tc::put_split_f<KIND>(A, a_plane, row, 2 * (kq * G + j) + 1, Kr, (float)z.y);
          }
        }
      }
    } else {
      const int per_row = nk / G;
      const int nitems = kTcRows * per_row;
      for (int it0 = tid; it0 < nitems; it0 += 4 * NT) {
        float re[4][G], im[4][G];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int item = it0 + u * NT;
          const int row = item % kTcRows, kq = item / kTcRows;
          const int R = r0 + row;
          const bool in = item < nitems && R < rows;
          long long base = 0;
          if (in) {
            const int outer = fdivu(R, st, tp.inv_st[g]);
            base = (long long)outer * D * st + (R - outer * st);
          }
#pragma unroll
          for (int j = 0; j < G; ++j) {
            const int kg = kc0 + kq * G + j;   // global K index: term kg / D, leg index kg % D
            V z;
            z.x = z.y = (T)0;
            if (in && kg < nterm * D) {
              const int tl = kg / D, kk = kg - tl * D;
              const int q = tp.gfirst[g] + tl;
              const Term& T_ = os.terms[tp.gterm[q]];
              const Factor* fs = T_.nf == 2 ? &T_.f[1 - tp.gdense[q]] : nullptr;
              z = tc_z<T>(P, nd, fs, x, base + (long long)kk * st);
            }
            re[u][j] = (float)z.x;
            im[u][j] = (float)z.y;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int item = it0 + u * NT;
          if (item >= nitems) break;
          const int row = item % kTcRows, kq = item / kTcRows;
#pragma unroll
          for (int j = 0; j < G; ++j) {
            tc::put_split_f<KIND>(A, a_plane, row, 2 * (kq * G + j), Kr, re[u][j]);
            tc::put_split_f<KIND>(A, a_plane, row, 2 * (kq * G + j) + 1, Kr, im[u][j]);
          }
        }
      }
    }
    // B: the 2 x 2 real blocks of M_t[i][k]: rows 2i (a, -b) and 2i + 1 (b, a)
    {
      const int per_i = nk / G;
      const int nitems = (Npad / 2) * per_i;
      for (int item = tid; item < nitems; item += NT) {
        const int kq = item % per_i, i = item / per_i;
        float2 m[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int kg = kc0 + kq * G + j;
          m[j] = make_float2(0.f, 0.f);
          if (i < D && kg < nterm * D) {
            const int tl = kg / D, kk = kg - tl * D;
            const int q = tp.gfirst[g] + tl;
            const Factor& fd = os.terms[tp.gterm[q]].f[tp.gdense[q]];
            m[j] = P.pool32[fd.mat + (long long)i * D + kk];
          }
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const int k = kq * G + j;
          tc::put_split_f<KIND>(B, b_plane, 2 * i, 2 * k, Kr, m[j].x);
          tc::put_split_f<KIND>(B, b_plane, 2 * i, 2 * k + 1, Kr, -m[j].y);
          tc::put_split_f<KIND>(B, b_plane, 2 * i + 1, 2 * k, Kr, m[j].y);
          tc::put_split_f<KIND>(B, b_plane, 2 * i + 1, 2 * k + 1, Kr, m[j].x);
        }
      }
    }
    tc::fence_proxy_async();
    __syncthreads();
    pc.lap(P.ctl, 20);
    const int nsteps = nk / KSC;
    if (tid == 0) {
      tc::fence_after();
      for (int ks = 0; ks < nsteps; ++ks)
        tc::issue_kstep<KIND>(ts.tmem + (uint32_t)(ks * Npad), A, a_plane, B, b_plane, Npad, Kr, ks);
      tc::commit(&ts.mbar);
    }
    const bool w = tc::mbar_wait(&ts.mbar, ts.phase, P.spin_limit);
    tc::fence_after();
    ok = __syncthreads_and(w) != 0;  // the same decision on every thread
    if (!ok) break;
    if (tid == 0) ts.phase ^= 1u;
    pc.lap(P.ctl, 21);
    // the K steps' partial products, summed in a fixed order into the shared FP32 sums; the
    // loads of all K steps of a column group are issued before one wait
    const uint32_t lane_base = ts.tmem + ((uint32_t)(q4 * 32) << 16);
    for (int c = c_lo; c < c_hi; c += 8) {
      uint32_t r[8][8];
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        if (ks < nsteps) tc::tmem_ld8_nowait(lane_base + (uint32_t)(ks * Npad + c), r[ks]);
      tc::tmem_wait_ld();
      float acc[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        if (ks < nsteps) {
          tc::tmem_pin8(r[ks]);
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] += __uint_as_float(r[ks][j]);
        }
#pragma unroll
      for (int j = 0; j < 8; ++j) sums[my_row * ldsum + c + j] += acc[j];
    }
    tc::fence_before();
    __syncthreads();
    pc.lap(P.ctl, 22);
  }
  if (!ok) {
    // a completion wait gave up: report it, give the MMAs in flight a last bounded wait, and
    // leave the tensor cores alone in this CTA for the rest of the launch
    if (tid == 0) set_status(P.ctl, ST_TIMEOUT, 400, -1);
    tc::mbar_wait(&ts.mbar, ts.phase, P.spin_limit);
    __syncthreads();
    if (tid == 0) ts.on = 0;
    __syncthreads();
    return false;
  }
  // the tile's rows of Y_g: row R = (outer, inner) of leg l, column pair (2i, 2i + 1) = y[.., i, ..]
  const int R = r0 + my_row;
  if (R < rows) {
    const int outer = fdivu(R, st, tp.inv_st[g]);
    const long long base = (long long)outer * D * st + (R - outer * st);
    for (int c = c_lo; c < c_hi; c += 2) {
      const int i = c >> 1;
      if (i < D) {
        V y;
        y.x = (T)sums[my_row * ldsum + c];
        y.y = (T)sums[my_row * ldsum + c + 1];
        yg[base + (long long)i * st] = y;
      }
    }
  }
  __syncthreads();
  pc.lap(P.ctl, 23);
  return true;
}

// All tasks of the plan over the team's CTAs (task k on rank k mod size).  The result of
// part p of group g goes to slot gslot0[g] + p at ybuf + slot * ystride.  The caller
// synchronises the team before reading the slots.
template <typename T, typename XT>
__device__ void tc_apply(const KernelParams& P, Team& tm, const NodeDesc& nd, const OpStage& os, const TcPlan& tp,
                         const XT* x, typename C2<T>::t* ybuf, long long ystride) {
  const int ntask = tp.gtask0[tp.ngroups];
  for (int task = tm.rank; task < ntask; task += tm.size) {
    int g = 0;
    while (task >= tp.gtask0[g + 1]) ++g;
    const int local = task - tp.gtask0[g];
    const int part = local / tp.gtiles[g], rt = local - part * tp.gtiles[g];
    auto* yg = ybuf + (long long)(tp.gslot0[g] + part) * ystride;
    const bool prof = P.profile && tm.rank == 0;
    const bool ok = P.precision == 2 ? tc_task<tc::KIND_BF16X3, T>(P, nd, os, tp, g, part, rt, x, yg, prof)
                                     : tc_task<tc::KIND_TF32X3, T>(P, nd, os, tp, g, part, rt, x, yg, prof);
    if (!ok) break;
  }
}

// H_eff x at idx from the group results and the terms left to the SIMT path
template <typename T, typename XT>
__device__ __forceinline__ typename C2<T>::t tc_sum_at(const KernelParams& P, const NodeDesc& nd, const OpStage& os,
                                                      const TcPlan& tp, const XT* x,
                                                      const typename C2<T>::t* ybuf, long long ystride,
                                                      long long idx) {
  typename C2<T>::t acc;
  acc.x = acc.y = (T)0;
  const int nslot = tp.gslot0[tp.ngroups];
  for (int sl = 0; sl < nslot; ++sl) {
    const auto y = ybuf[sl * ystride + idx];
    acc.x += y.x;
    acc.y += y.y;
  }
  for (int q = 0; q < tp.nsimt; ++q) {
    const Term& T_ = os.terms[tp.simt[q]];
    const auto a = T_.nf == 1 ? factor_dot<T>(P, nd, T_.f[0], os, x, idx) : direct_dot<T>(P, nd, T_, os, x, idx);
    acc.x += a.x;
    acc.y += a.y;
  }
  return acc;
}

template <typename T>
__device__ __noinline__ void op_expm(const KernelParams& P, Team& tm, const Instr& I, double2* work, double tau) {
  KrylovShared& ks = s_ks;
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0, tm.kind == TEAM_GRID);
  const NodeDesc nd = P.nodes[I.node];
  const TermList L = P.lists[I.terms];
  const long long N = nd.size;
  const long long kv = P.kvec;
  double2* x = P.pool + nd.off;
  double2* Kb = work;                           // K_1..K_mmax at Kb + (j-1)*kv
  auto* tmp = reinterpret_cast<typename C2<T>::t*>(work + (long long)P.mmax * kv);  // n_tmp temporaries
  auto Kp = [&](int j) -> double2* { return j == 0 ? x : Kb + (long long)(j - 1) * kv; };
  const int mmax = min(P.mmax, (int)(N < (long long)TTNS_KMAX ? N : (long long)TTNS_KMAX));
  OpStage& os = s_os;
  stage_op<T>(P, I, L, nullptr, 0, os);
  using V = typename C2<T>::t;
  constexpr bool kShadow = !std::is_same<T, double>::value;
  // tensor-core apply (split precision) for nodes whose terms have one dense factor each; its
  // operand tiles take the dynamic shared memory, so nothing staged there is used
  // (a large root's tiles first: 2980 us per exponential at 20^4 x 5, 8 % more since their products
  // keep several accumulators; the tensor cores 4210 in TF32X3 and 3550 in BF16X3, where splitting
  // the operands is the bound; at 14^4 x 5 980 us, there 980 and 1030.  With fewer tiles than CTAs
  // the tensor cores are ahead: 400 us at 20^3 x 5, by tiles 580)
  V* xt = nullptr;
  bool tiled = false, fibres = false, use_tc = false;
  if constexpr (kShadow)
    if (tm.kind == TEAM_GRID && vec_smem<T>(P, os, N) == nullptr) {
      xt = tiled_begin<T>(P, tm, nd, os, L, false, tiled, fibres);
      tiled = fibres;
      __syncthreads();  // every thread has placed its tiles by os.end, which the plan below clears
    }
  if (SWEEP_CTAS == 1 && !fibres && s_tc.on && (P.precision == 1 || P.precision == 2) && N >= 4096) {
    if (threadIdx.x == 0) {
      tc_plan(nd, os, L, P.precision == 2 ? tc::Split<tc::KIND_BF16X3>::kstep / 2 : tc::Split<tc::KIND_TF32X3>::kstep / 2,
              s_tcp);
      if (s_tcp.ok) {
        os.a_n = os.b_n = 0;
        os.end = 0;
      }
    }
    __syncthreads();
    use_tc = s_tcp.ok != 0;
  }
  V* ybuf = reinterpret_cast<V*>(work + (long long)(P.mmax + P.n_tmp + 2) * kv);  // group results (TC)
  V* xs = use_tc || fibres ? nullptr : vec_smem<T>(P, os, N);  // input vector in shared memory when it fits
  // otherwise, in mixed precision, a compute-type copy of the input vector in the workspace,
  // written by the pass that produces the vector (FP64 Krylov basis, FP32 operand)
  // (kept in the mixed modes whether or not the vector is staged: staging then copies it
  // instead of converting the FP64 vector on every CTA)
  V* xf = reinterpret_cast<V*>(work + (long long)(P.mmax + P.n_tmp) * kv);
  const bool shadow = kShadow;
  // tiled apply for a grid-team node that does not fit in shared memory
  TiledApply& tp = s_tp;
  if (tm.kind == TEAM_GRID && xs == nullptr && !use_tc && !fibres) xt = tiled_begin<T>(P, tm, nd, os, L, L.n2 == 0, tiled, fibres);
  pc.lap(P.ctl, 0);
  // exp(-i s H): s = time / hbar with the op's sign.  If the Krylov space of dimension
  // mmax does not reach the tolerance for the remaining time, the largest s / 2^k that
  // does is taken on the same space and a new space is built for the rest.
  double s_rem = I.sign * tau / HBAR_EVFS;
  int total_m = 0;
  int m = 0;
  for (int chunk = 0; chunk < 64; ++chunk) {
    double v[1];
    v[0] = 0;
    for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
      const double2 a = x[idx];
      v[0] = fma(a.x, a.x, fma(a.y, a.y, v[0]));
      if constexpr (kShadow) xf[idx] = cvt<T>(a);
    }
    team_reduce<1>(tm, v, [&](const double* t) { krylov_begin(ks, t[0]); });
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
      double2* Kj = Kp(j);
      double2* Kjm = j > 0 ? Kp(j - 1) : x;
      double2* W = Kb + (long long)j * kv;  // slot of K_{j+1}
      const double sj = ks.scale[j];
      const double cm = ks.cm;  // beta_j scale_{j-1}
      if (xs) {
        if constexpr (kShadow)
          stage_copy(xs, xf, N);
        else
          stage_vector<T>(xs, Kj, N);
      }
      // operand of this application: shared memory, the FP32 shadow, or K_j itself (FP64)
      const V* xin = xs ? xs : (shadow ? xf : reinterpret_cast<const V*>(Kj));
      if (L.n2 > 0 && !tiled) {
        apply_stage1<T>(P, tm, nd, xin, L, tmp, kv, os);
        team_sync(tm);
      }
      pc.lap(P.ctl, 1);
      // part[0] = Re <K_j, w>; in mixed precision also part[1] = |w|^2 and part[2] = |K_j|^2
      // (one reduction for alpha_j and beta_{j+1}, as in the cluster-resident form)
      double part[3] = {0.0, 0.0, nsq};
      // w = s_j H K_j - beta_j q_{j-1} at idx, and the dots
      auto recur = [&](long long idx, V a) {
        double wr = sj * to_f64(a.x), wi = sj * to_f64(a.y);
        const double2 kj = Kj[idx];
        if (j > 0) {
          const double2 km = Kjm[idx];
          wr = fma(-cm, km.x, wr);
          wi = fma(-cm, km.y, wi);
        }
        part[0] = fma(kj.x, wr, fma(kj.y, wi, part[0]));  // Re(conj(K_j) w)
        if constexpr (kShadow) part[1] = fma(wr, wr, fma(wi, wi, part[1]));
        W[idx] = make_double2(wr, wi);
      };
      if (use_tc) {
        tc_apply<T>(P, tm, nd, os, s_tcp, xin, ybuf, kv);
        team_sync(tm);
        pc.lap(P.ctl, 7);
        for (long long idx = tm.gtid(); idx < N; idx += tm.nthr())
          recur(idx, tc_sum_at<T>(P, nd, os, s_tcp, xin, ybuf, kv, idx));
      } else if (tiled) {
        V* y = tmp;  // pass A sums (the temporaries of two-stage terms are not used here)
        tiled_pass<T>(P, tm, tp, os, L, xin, xt, fibres, 0, [&](long long g, V acc) { y[g] = acc; });
        team_sync(tm);
        tiled_pass<T>(P, tm, tp, os, L, xin, xt, fibres, 1, [&](long long g, V acc) {
          V a = y[g];
          a.x += acc.x;
          a.y += acc.y;
          recur(g, a);
        });
      } else {
        for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) recur(idx, apply_stage2_at<T>(P, nd, xin, L, tmp, kv, idx, os));
      }
      if constexpr (kShadow)
        team_reduce<3>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0], t[1], t[2]); });
      else
        team_reduce<1>(tm, part, [&](const double* t) { krylov_alpha(ks, j, t[0]); });
      pc.lap(P.ctl, 2);
      const double ca = ks.ca;  // alpha_j scale_j
      if (kShadow && ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
      double nrm[1] = {0.0};
      for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
        const double2 kj = Kj[idx];
        double2 w = W[idx];
        w.x = fma(-ca, kj.x, w.x);
        w.y = fma(-ca, kj.y, w.y);
        W[idx] = w;
        if constexpr (kShadow) {
          xf[idx] = cvt<T>(w);  // every read of the old shadow ended at the last barrier
          nrm[0] = fma(w.x, w.x, fma(w.y, w.y, nrm[0]));
        }
      }
      if constexpr (!kShadow) {
        nrm[0] = orth_strided(tm, N, x, Kb, kv, W, j, ks);
        if (ks.fused && threadIdx.x == NT - 32) krylov_norm(ks, j, ks.b2, s_rem, P.tol, mmax);
      }
      const bool fused = ks.fused != 0;
      nsq = nrm[0];
      if (fused)
        team_sync(tm);  // K_{j+1} and its shadow are complete before the next application
      else
        team_reduce<1>(tm, nrm, [&](const double* t) { krylov_norm(ks, j, t[0], s_rem, P.tol, mmax); });
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
    // y = beta0 * sum_k u_k q_k written over x (each thread reads its own K_0 = x entries first)
    double ny[1] = {0.0};
    for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
      double yr = 0.0, yi = 0.0;
      for (int k = 0; k < m; ++k) {
        const double2 q = Kp(k)[idx];
        const double cr = ks.ure[k], ci = ks.uim[k];
        yr = fma(cr, q.x, fma(-ci, q.y, yr));
        yi = fma(cr, q.y, fma(ci, q.x, yi));
      }
      x[idx] = make_double2(yr, yi);
      ny[0] = fma(yr, yr, fma(yi, yi, ny[0]));
    }
    if constexpr (kShadow) {
      // The exact exponential is unitary.  FP32-class contractions leave the Krylov basis
      // orthonormal only to ~1e-7, so the combination's norm is restored to the input's.
      team_reduce<1>(tm, ny, [&](const double* t) { ks.ratio = t[0] > 0.0 ? ks.beta0 / sqrt(t[0]) : 1.0; });
      const double ratio = ks.ratio;
      if (fabs(ratio - 1.0) < 1e-3) {
        for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
          double2 y = x[idx];
          x[idx] = make_double2(y.x * ratio, y.y * ratio);
        }
      }
    }
    team_sync(tm);
    pc.lap(P.ctl, 5);
    if (conv || m >= N || s_done == s_rem) break;
    s_rem -= s_done;
    if (chunk == 63 && tm.rank == 0 && threadIdx.x == 0) {
      // 64 Krylov spaces did not cover the time step: the result is incomplete
      atomicAdd(&P.ctl->not_converged, 1ull);
      set_status(P.ctl, ST_NOT_CONVERGED, I.op, I.node);
    }
  }
  if (tm.rank == 0 && threadIdx.x == 0) {
    P.mhist[I.hist] = m;
    atomicAdd(&P.ctl->krylov_iters, (unsigned long long)total_m);
    atomicAdd(&P.ctl->applies, (unsigned long long)total_m);
    atomicAdd(&P.ctl->flops, I.flops * total_m);
  }
}

#include "qr.cuh"

#include "absorb.cuh"
#include "site.cuh"

// ------------------------------------------------------------------ environment update
// env(u -> v): block 0 = Q^H (H-terms of u without v) Q, block 1+b = Q^H (channel factor b) Q,
// contracted over every leg of Q except the leg toward v.  This form takes the tensors that are
// not sites (ER nodes, roots of several chains, OBB sites): results of all rows in global memory,
// every output value summed over all rows by one CTA.
// Projection of the grid team: out[b][a][a'] = sum_rows conj(Q[row, a]) Y_b[row, a'].  Every CTA
// sums over its own rows, in blocks of kProjRows staged in shared memory with a 2 x 2 tile of
// outputs per thread, in runs of one block in the compute type and between blocks in FP64 or
// double-single; the CTAs' partials are added in order.  With outputs split over the CTAs instead
// (below) every CTA reads all rows, a word per multiply-add from L2: 417 us at 40000 rows, D 20, in
// FP32 and 780 in FP64; 70 and 434 now.  From a block of rows per CTA on; with fewer the partials
// and their sum cost as much as the products.
constexpr int kProjRows = 64;
template <typename T>
__device__ __noinline__ bool project_rows(const KernelParams& P, Team& tm, const Instr& I, const NodeDesc& nd,
                                          const typename C2<T>::t* xq, const typename C2<T>::t* Y) {
  using V = typename C2<T>::t;
  using A = typename EnvArith<T>::A;
  using E = typename A::E;
  const int l = I.leg, D = I.D, nch = I.nchan, nb = 1 + nch, lst = nd.strides[l];
  const int rows = nd.size / D, chunk = (rows + tm.size - 1) / tm.size;
  const long long kv = P.kvec;
  constexpr int RP = kProjRows + 1;  // odd: lanes on different columns read different banks
  if (tm.kind != TEAM_GRID || rows < kProjRows * tm.size || 2LL * D * RP * (long long)sizeof(V) > P.smem_bytes) return false;
  V* Qs = reinterpret_cast<V*>(dyn_smem);
  V* Ys = Qs + D * RP;
  const int rb = min(rows, tm.rank * chunk), re = min(rows, rb + chunk);
  const int D2 = D * D, nval = nb * D2, h = (D + 1) / 2;
  const float inv_h = 1.0f / (float)h, inv_D = nd.inv_dims[l], inv_l = nd.inv_strides[l];
  E* buf = reinterpret_cast<E*>(team_partials(tm));
  E* mine = buf + (long long)tm.rank * nval;
  auto load = [&](V* dst, const V* src, int r0, int nr) {  // dst[a][r]
    const float inv_n = 1.0f / (float)nr;
    for (int it = threadIdx.x; it < D * nr; it += NT) {
      int a, r;
      if (lst == 1) {
        r = fdivu(it, D, inv_D);
        a = it - r * D;
      } else {
        a = fdivu(it, nr, inv_n);
        r = it - a * nr;
      }
      const int p = fdivu(r0 + r, lst, inv_l);
      const V* g = src + (long long)p * D * lst + (r0 + r - p * lst) + (long long)a * lst;
      if constexpr (sizeof(V) == 16)
        cp_async16(dst + a * RP + r, g);
      else
        cp_async8(dst + a * RP + r, g);
    }
  };
  auto skip = [&](int b) { return b > 0 && ((I.adj >> (b - 1)) & 1u); };  // adjoint of the channel before
  for (int r0 = rb; r0 < re || r0 == rb; r0 += kProjRows) {
    const int nr = max(0, min(kProjRows, re - r0));
    for (int b = 0; b < nb; ++b) {
      if (skip(b)) continue;
      __syncthreads();
      if (nr > 0) {
        if (b == 0) load(Qs, xq, r0, nr);
        load(Ys, Y + b * kv, r0, nr);
      }
      cp_async_wait_all();
      __syncthreads();
      for (int it = threadIdx.x; it < h * h; it += NT) {
        const int ta = fdivu(it, h, inv_h);
        const int a0 = 2 * ta, a1 = min(a0 + 1, D - 1), p0 = 2 * (it - ta * h), p1 = min(p0 + 1, D - 1);
        const V *q0 = Qs + a0 * RP, *q1 = Qs + a1 * RP, *y0 = Ys + p0 * RP, *y1 = Ys + p1 * RP;
        constexpr int U = std::is_same<T, double>::value ? 1 : 4;
        V s[4][U];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int u = 0; u < U; ++u) s[q][u].x = s[q][u].y = (T)0;
        auto cj = [](V& e, V q, V y) {  // e += conj(q) y
          e.x = fma(q.x, y.x, fma(q.y, y.y, e.x));
          e.y = fma(q.x, y.y, fma(-q.y, y.x, e.y));
        };
        auto step = [&](int r, int u) {
          const V u0 = q0[r], u1 = q1[r], w0 = y0[r], w1 = y1[r];
          cj(s[0][u], u0, w0);
          cj(s[1][u], u0, w1);
          cj(s[2][u], u1, w0);
          cj(s[3][u], u1, w1);
        };
        int r = 0;
        for (; r + 3 < nr; r += 4) {
#pragma unroll
          for (int u = 0; u < 4; ++u) step(r + u, u % U);
        }
        for (; r < nr; ++r) step(r, 0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int a = a0 + (q >> 1), p = p0 + (q & 1);
          if (a >= D || p >= D) continue;
          E& e = mine[b * D2 + a * D + p];
          E o = r0 == rb ? A::c(A::zero(), A::zero()) : e;
          const V t = sum_parts<U>(s[q]);
          if constexpr (std::is_same<T, double>::value)
            o = A::c(A::add(A::re(o), t.x), A::add(A::im(o), t.y));
          else
            o = A::c(A::add(A::re(o), make_float2(t.x, 0.f)), A::add(A::im(o), make_float2(t.y, 0.f)));
          e = o;
        }
      }
    }
  }
  team_sync(tm);
  double2* out = P.pool + I.env_out;
  auto emit = [&](int k, E v) {
    out[k] = A::cto(v);
    if constexpr (!std::is_same<T, double>::value) P.pool32[I.env_out + k] = make_float2(A::re(v).x, A::im(v).x);
  };
  for (int k = tm.gtid(); k < nval; k += tm.nthr()) {
    const int b = k / D2, r = k - b * D2, a = r / D, p = r - a * D;
    if (skip(b)) continue;
    typename A::S sr = A::zero(), si = A::zero();
#pragma unroll 8
    for (int q = 0; q < tm.size; ++q) {
      const E v = buf[(long long)q * nval + k];
      sr = A::add(sr, A::re(v));
      si = A::add(si, A::im(v));
    }
    emit(k, A::c(sr, si));
    if (b > 0 && b < nch && ((I.adj >> b) & 1u)) emit((b + 1) * D2 + p * D + a, A::c(sr, A::neg(si)));
  }
  tm.parity ^= 1;
  return true;
}

template <typename T>
__device__ __noinline__ void op_env(const KernelParams& P, Team& tm, const Instr& I, double2* work) {
  const NodeDesc nd = P.nodes[I.node];
  const TermList L = P.lists[I.terms];
  const long long N = nd.size;
  const long long kv = P.kvec;
  using V = typename C2<T>::t;
  const double2* Q = P.pool + nd.off;
  auto* tmp = reinterpret_cast<V*>(work + (long long)P.mmax * kv);
  V* Y = reinterpret_cast<V*>(work);  // Y_0 .. Y_nchan at Y + b*kv, compute type (fits: 1 + nchan <= mmax)
  PhaseClock pc;
  pc.start(P.profile && tm.rank == 0 && threadIdx.x == 0, tm.kind == TEAM_GRID);
  const int l = I.leg;
  const int D = I.D;
  const int nb = 1 + I.nchan;
  OpStage& os = s_os;
  stage_op<T>(P, I, L, P.chans + I.chan_first, I.nchan, os);
  V* xs = vec_smem<T>(P, os, N);
  // the operand Q in the compute type: shared memory when it fits, else (mixed precision) a
  // converted copy in the workspace, else (FP64) the tensor itself
  const V* xq;
  if (xs) {
    stage_vector<T>(xs, Q, N);
    xq = xs;
  } else if constexpr (!std::is_same<T, double>::value) {
    V* qf = reinterpret_cast<V*>(work + (long long)(P.mmax + P.n_tmp) * kv);
    for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) qf[idx] = cvt<T>(Q[idx]);
    team_sync(tm);
    xq = qf;
  } else {
    xq = reinterpret_cast<const V*>(Q);
  }
  pc.lap(P.ctl, 16);
  bool tiled = false, fibres = false;
  V* xt = nullptr;
  if (tm.kind == TEAM_GRID && xs == nullptr) xt = tiled_begin<T>(P, tm, nd, os, L, false, tiled, fibres);
  if (tiled) {
    tiled_pass<T>(P, tm, s_tp, os, L, xq, xt, fibres, 0, [&](long long g, V acc) { Y[g] = acc; });
    team_sync(tm);
    tiled_pass<T>(P, tm, s_tp, os, L, xq, xt, fibres, 1, [&](long long g, V acc) {
      V a = Y[g];
      a.x += acc.x;
      a.y += acc.y;
      Y[g] = a;
    });
  } else if (L.n2 > 0) {
    apply_stage1<T>(P, tm, nd, xq, L, tmp, kv, os);
    team_sync(tm);
  }
  for (long long idx = tm.gtid(); idx < N; idx += tm.nthr()) {
    if (!tiled) Y[idx] = apply_stage2_at<T>(P, nd, xq, L, tmp, kv, idx, os);
    for (int b = 0; b < I.nchan; ++b) Y[(long long)(1 + b) * kv + idx] = factor_dot<T>(P, nd, os.chans[b], os, xq, idx);
  }
  team_sync(tm);
  pc.lap(P.ctl, 17);
  const bool projected = xs == nullptr && project_rows<T>(P, tm, I, nd, xq, Y);  // (stages in xs's place)
  // projection: out[b][a][a'] = sum_rows conj(Q[row, a]) Y_b[row, a'].  Each CTA owns a
  // contiguous block of the output values and sums them over all rows: the rows of an output
  // are split into `parts` ranges over the CTA's threads (partial sums in the compute type in
  // runs of 64 rows, then FP64), and one thread per output adds its parts in a fixed order and
  // writes the value; no partial sums cross CTAs.
  const long long rows = N / D;
  const int nval = projected ? 0 : nb * D * D;
  const long long lst = nd.strides[l];
  const int opc = (nval + tm.size - 1) / tm.size;
  const int ob = min(nval, tm.rank * opc), oe = min(nval, ob + opc);
  const int nout = oe - ob;
  const int parts = nout > 0 ? max(1, min(16, NT / nout)) : 1;
  const long long rpp = (rows + parts - 1) / parts;
  double2* pbuf = P.cta_scratch + (long long)blockIdx.x * P.cta_scratch_stride;  // parts x nout (parts > 1)
  double2* out = P.pool + I.env_out;
  for (int it = threadIdx.x; it < nout * parts; it += NT) {
    const int o = ob + it % nout, part = it / nout;
    const int b = o / (D * D);
    const int a = (o / D) % D;
    const int a2 = o % D;
    const V* Yb = Y + (long long)b * kv;
    const long long rb0 = part * rpp, re0 = min(rows, rb0 + rpp);
    double accr = 0, acci = 0;
    for (long long r0 = rb0; r0 < re0; r0 += 64) {
      V s0, s1;
      s0.x = s0.y = s1.x = s1.y = 0;
      const long long r1 = min(re0, r0 + 64);
      long long r = r0;
      for (; r + 1 < r1; r += 2) {  // two rows at a time: independent accumulators
        const long long p0 = fdivu((int)r, (int)lst, nd.inv_strides[l]), q0 = r - p0 * lst;
        const long long p1 = fdivu((int)(r + 1), (int)lst, nd.inv_strides[l]), q1 = r + 1 - p1 * lst;
        const long long base0 = p0 * D * lst + q0, base1 = p1 * D * lst + q1;
        const V qa0 = xq[base0 + (long long)a * lst], y0 = Yb[base0 + (long long)a2 * lst];
        const V qa1 = xq[base1 + (long long)a * lst], y1 = Yb[base1 + (long long)a2 * lst];
        s0.x = fma(qa0.x, y0.x, fma(qa0.y, y0.y, s0.x));
        s0.y = fma(qa0.x, y0.y, fma(-qa0.y, y0.x, s0.y));
        s1.x = fma(qa1.x, y1.x, fma(qa1.y, y1.y, s1.x));
        s1.y = fma(qa1.x, y1.y, fma(-qa1.y, y1.x, s1.y));
      }
      if (r < r1) {
        const long long p0 = fdivu((int)r, (int)lst, nd.inv_strides[l]), q0 = r - p0 * lst;
        const long long base0 = p0 * D * lst + q0;
        const V qa0 = xq[base0 + (long long)a * lst], y0 = Yb[base0 + (long long)a2 * lst];
        s0.x = fma(qa0.x, y0.x, fma(qa0.y, y0.y, s0.x));
        s0.y = fma(qa0.x, y0.y, fma(-qa0.y, y0.x, s0.y));
      }
      accr += (double)s0.x + (double)s1.x;
      acci += (double)s0.y + (double)s1.y;
    }
    if (parts == 1) {
      out[o] = make_double2(accr, acci);
      if constexpr (!std::is_same<T, double>::value) P.pool32[I.env_out + o] = make_float2((float)accr, (float)acci);
    } else
      pbuf[(long long)part * nout + (o - ob)] = make_double2(accr, acci);  // parts * nout <= NT
  }
  __syncthreads();
  pc.lap(P.ctl, 18);
  if (parts > 1)
    for (int k = threadIdx.x; k < nout; k += NT) {
      double sr = 0.0, si = 0.0;
      for (int part = 0; part < parts; ++part) {
        const double2 v = pbuf[(long long)part * nout + k];
        sr += v.x;
        si += v.y;
      }
      out[ob + k] = make_double2(sr, si);
      if constexpr (!std::is_same<T, double>::value) P.pool32[I.env_out + ob + k] = make_float2((float)sr, (float)si);
    }
  team_sync(tm);
  pc.lap(P.ctl, 19);
  if (tm.rank == 0 && threadIdx.x == 0) {
    atomicAdd(&P.ctl->applies, 1ull);
    atomicAdd(&P.ctl->flops, I.flops);
  }
}

// ------------------------------------------------------------------ record rho_S
__device__ __noinline__ void op_record(const KernelParams& P, Team& tm, const Instr& I, int* counter) {
  const TreeDesc td = P.trees[I.tree];
  if (td.traj_off < 0) return;
  const NodeDesc nd = P.nodes[td.node0];
  const int ne = td.n_el;
  const long long rows = nd.size / ne;  // phys leg is the last leg: stride 1
  const double2* A = P.pool + nd.off;
  const int nval = ne * ne;
  double* part = team_partials(tm);
  const long long chunk = (rows + tm.size - 1) / tm.size;
  const long long r_begin = (long long)tm.rank * chunk, r_end = min(rows, r_begin + chunk);
  for (int o = threadIdx.x; o < nval; o += NT) {
    const int s1 = o / ne, s2 = o % ne;
    double accr = 0, acci = 0;
    for (long long r = r_begin; r < r_end; ++r) {
      double2 a = A[r * ne + s1], b = A[r * ne + s2];
      accr = fma(a.x, b.x, fma(a.y, b.y, accr));
      acci = fma(a.y, b.x, fma(-a.x, b.y, acci));
    }
    part[(long long)tm.rank * 2 * nval + 2 * o] = accr;
    part[(long long)tm.rank * 2 * nval + 2 * o + 1] = acci;
  }
  int slot = *counter;
  if (slot >= P.max_record) slot = P.max_record - 1;
  team_finish_multi(tm, 2 * nval, (double*)(P.pool + td.traj_off + (long long)slot * nval), 1.0);
  if (tm.rank == 0 && threadIdx.x == 0) {
    *counter = *counter + 1;
    atomicAdd(&P.ctl->steps, 1ull);
  }
}

// ------------------------------------------------------------------ interpreter
template <typename T>
__device__ void exec_op(const KernelParams& P, Team& tm, const Instr& I, double2* work);

template <typename T>
__device__ void exec(const KernelParams& P, Team& tm, const Instr& I, double2* work) {
  if (!P.profile) {
    exec_op<T>(P, tm, I, work);
    return;
  }
  const long long t0 = clock64();
  exec_op<T>(P, tm, I, work);
  if (tm.rank == 0 && threadIdx.x == 0) {
    const long long dt = clock64() - t0;
    atomicAdd(&P.ctl->prof_cycles[I.op][tm.kind], (unsigned long long)dt);
    atomicAdd(&P.ctl->prof_count[I.op][tm.kind], 1ull);
  }
}

template <typename T>
__device__ void exec_op(const KernelParams& P, Team& tm, const Instr& I, double2* work) {
  const double tau = 0.5 * P.dt;
  switch (I.op) {
    case OP_FWD:
    case OP_BOND:
      if (!op_expm_site<T>(P, tm, I, work, tau) &&
          !(tm.kind == TEAM_CLUSTER && P.cluster_resident && op_expm_cluster<T>(P, tm, I, work, tau)))
        op_expm<T>(P, tm, I, work, tau);
      break;
    case OP_QR:
      if constexpr (std::is_same<T, double>::value)
        op_qr<QrF64>(P, tm, I, work);
      else
        op_qr<QrDs>(P, tm, I, work);
      break;
    case OP_ENV:
      if (!op_env_site<T>(P, tm, I)) op_env<T>(P, tm, I, work);
      break;
    case OP_ABSORB:
      if constexpr (std::is_same<T, double>::value)
        op_absorb<QrF64>(P, tm, I);
      else
        op_absorb<QrDs>(P, tm, I);
      break;
    case OP_RECORD:
      op_record(P, tm, I, P.traj_count + I.tree);
      break;
  }
}

// The current instruction in shared memory; the next one's words are loaded into registers while
// it runs, so that no operation starts with a chain of global loads for its own record.
__shared__ Instr s_instr;
struct InstrFeed {
  static constexpr int kWords = (int)(sizeof(Instr) / 4);
  static_assert(kWords <= NT && sizeof(Instr) % 4 == 0, "one word per thread");
  const unsigned* p;
  unsigned w;
  __device__ InstrFeed(const Instr* prog) : p(reinterpret_cast<const unsigned*>(prog)), w(0) {
    if (threadIdx.x < kWords) w = p[threadIdx.x];
  }
  __device__ void next(bool more) {
    __syncthreads();  // the last instruction is done
    if (threadIdx.x < kWords) {
      reinterpret_cast<unsigned*>(&s_instr)[threadIdx.x] = w;
      p += kWords;
      if (more) w = p[threadIdx.x];
    }
    __syncthreads();
  }
};

template <typename T>
__device__ void run(const KernelParams& P, int phase) {
  const int cs = P.cluster_ctas;
  const int cluster_id = blockIdx.x / cs;
  const int n_clusters = gridDim.x / cs;
  const int crank = (int)cg::this_cluster().block_rank();
  Team ct;
  ct.kind = TEAM_CLUSTER;
  ct.rank = crank;
  ct.size = cs;
  ct.red = P.red + (long long)cluster_id * 2 * P.red_stride;
  ct.red_stride = P.red_stride;
  ct.parity = 0;
  ct.ctl = P.ctl;
  ct.spin_limit = P.spin_limit;
  ct.csize = cs;
  double2* cwork = P.work + (long long)cluster_id * P.work_stride;
  if (P.batched) {
    // A cluster takes the next tree when it is done with one, the long programs first.  Every
    // launch draws n_trees + n_clusters tickets (one too many per cluster), so the counter
    // needs no reset; batched launches have no grid barrier that would use it.
    __shared__ int s_ticket;
    for (;;) {
      __syncthreads();
      if (threadIdx.x == 0 && crank == 0)
        s_ticket = (int)(atomicAdd(&P.ctl->bar_count, 1ull) % (unsigned long long)(P.n_trees + n_clusters));
      if (cs > 1) cg::this_cluster().sync(); else __syncthreads();
      const int ticket = cs > 1 ? *cg::this_cluster().map_shared_rank(&s_ticket, 0) : s_ticket;
      if (cs > 1) cg::this_cluster().sync();  // read before rank 0 draws again or leaves
      if (ticket >= P.n_trees) break;
      const TreeDesc& td = P.trees[P.order[ticket]];
      const int first = phase == 0 ? td.init_first : (phase == 2 ? td.obs_first : (phase == 3 ? td.grow_first : td.prog_first));
      const int count = phase == 0 ? td.init_count : (phase == 2 ? td.obs_count : (phase == 3 ? td.grow_count : td.prog_count));
      const int nst = phase == 1 ? P.n_steps : 1;
      for (int s = 0; s < nst; ++s) {
        InstrFeed feed(P.prog + first);
        for (int k = 0; k < count; ++k) {
          feed.next(k + 1 < count);
          exec<T>(P, ct, s_instr, cwork);
        }
      }
    }
    return;
  }
  Team gt;
  gt.kind = TEAM_GRID;
  gt.rank = blockIdx.x;
  gt.size = gridDim.x;
  gt.red = P.red_grid;
  gt.red_stride = P.red_stride_grid;
  gt.parity = 0;
  gt.ctl = P.ctl;
  gt.spin_limit = P.spin_limit;
  gt.csize = cs;
  const TreeDesc& td = P.trees[0];
  const int first = phase == 0 ? td.init_first : (phase == 2 ? td.obs_first : (phase == 3 ? td.grow_first : td.prog_first));
  const int count = phase == 0 ? td.init_count : (phase == 2 ? td.obs_count : (phase == 3 ? td.grow_count : td.prog_count));
  const int nst = phase == 1 ? P.n_steps : 1;
  int prev = TEAM_GRID;
  for (int s = 0; s < nst; ++s) {
    InstrFeed feed(P.prog + first);
    for (int k = 0; k < count; ++k) {
      feed.next(k + 1 < count);
      const Instr& I = s_instr;
      if (I.team == TEAM_GRID) {
        if (prev == TEAM_CLUSTER) grid_sync(P.ctl, P.spin_limit);
        exec<T>(P, gt, I, P.work);
      } else if (cluster_id == 0) {
        exec<T>(P, ct, I, cwork);
        if (crank == 0 && threadIdx.x == 0) atomicAdd(&P.ctl->progress, 1u);
      }
      prev = I.team;
    }
  }
  if (prev == TEAM_CLUSTER) grid_sync(P.ctl, P.spin_limit);
}

__device__ __forceinline__ unsigned sreg_cluster_nctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned sreg_dynamic_smem_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
  return r;
}

// The two-CTA instance: what bounds batches of small trees is latency (FP64 chains, cluster
// barriers, scalar steps on one warp), and a second tree on the SM fills the waits.  It has half
// the registers and shared memory and no tensor memory (its trees are below the size at which
// the tensor-core products start).  256 chains of 10 to 40 sites on four-CTA teams (TF32X3): 327 ms
// a step with the trees in order, one per cluster at a time, 218 with the longest first on
// whichever cluster is free, 136 with two CTAs per SM (third step of a run; the first takes a fifth
// less).
__global__ void __launch_bounds__(NT, SWEEP_CTAS) k_sweep(KernelParams P, int phase) {
  // Launch self-check before any barrier or distributed-shared-memory access: the
  // interpreter addresses cluster peers by rank and stages operands up to smem_bytes, so a
  // launch with another cluster shape or less dynamic shared memory returns an error
  // status instead of running.  Every CTA takes the same decision.
  const unsigned ncta = sreg_cluster_nctarank();
  if (ncta != (unsigned)P.cluster_ctas || (long long)sreg_dynamic_smem_size() < P.smem_bytes ||
      gridDim.x % (unsigned)P.cluster_ctas != 0) {
    if (threadIdx.x == 0 && blockIdx.x == 0) set_status(P.ctl, ST_LAUNCH, 300, (int)ncta);
    return;
  }
  // tensor memory for the split-precision contractions (all 512 columns: one accumulator per K step)
  const bool tc_on = SWEEP_CTAS == 1 && (P.precision == 1 || P.precision == 2);
  if (threadIdx.x == 0) s_tc.on = 0;
  if (tc_on) {
    if ((threadIdx.x >> 5) == 0) tc::tmem_alloc(&s_tc.tmem, kTcTmemCols);
    if (threadIdx.x == 0) {
      tc::mbar_init(&s_tc.mbar, 1);
      s_tc.phase = 0;
      s_tc.on = 1;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
  }
  // the first operation writes to its peers' shared memory: every CTA of the cluster has to have
  // started (and cleared its tensor-core record) by then
  // (as one instruction pair: through the cooperative-groups call the whole kernel came out 0.7 %
  // slower)
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (P.precision == 0)
    run<double>(P, phase);
  else
    run<float>(P, phase);
  if (tc_on) {
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(s_tc.tmem, kTcTmemCols);
  }
}

#ifndef SWEEP_PAIR
// ------------------------------------------------------------------ observables
// Density of a root leg: partials of rho[b][b2] = sum_rows A[row, b] conj(A[row, b2]) along leg l,
// rows split over the blocks
__global__ void k_density_partial(const double2* A, NodeDesc nd, int l, double* partials) {
  const int D = nd.dims[l];
  const long long N = nd.size;
  const long long st = nd.strides[l];
  const long long rows = N / D;
  const long long chunk = (rows + gridDim.x - 1) / gridDim.x;
  const long long r_begin = (long long)blockIdx.x * chunk, r_end = min(rows, r_begin + chunk);
  for (int o = threadIdx.x; o < D * D; o += blockDim.x) {
    const int b = o / D, b2 = o % D;
    double accr = 0, acci = 0;
    for (long long r = r_begin; r < r_end; ++r) {
      const long long p = fdivu((int)r, (int)st, nd.inv_strides[l]), q = r - p * st;
      const long long base = p * D * st + q;
      const double2 y = A[base + (long long)b2 * st];
      const double2 xa = A[base + (long long)b * st];
      accr = fma(xa.x, y.x, fma(xa.y, y.y, accr));
      acci = fma(xa.y, y.x, fma(-xa.x, y.y, acci));
    }
    partials[(long long)blockIdx.x * 2 * D * D + 2 * o] = accr;
    partials[(long long)blockIdx.x * 2 * D * D + 2 * o + 1] = acci;
  }
}

// out[k] = sum of the blocks' partials in a fixed order, one warp per value
__global__ void k_reduce_partials(const double* partials, int nblocks, int nval, double* out) {
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int k = blockIdx.x * nw + (threadIdx.x >> 5); k < nval; k += gridDim.x * nw) {
    double s = 0;
    for (int b = lane; b < nblocks; b += 32) s += partials[(long long)b * nval + k];
    s = warp_sum(s);
    if (lane == 0) out[k] = s;
  }
}

// norm^2 and <A|H_eff|A> at the root with FP64 terms
__global__ void k_energy_partial(KernelParams P, int node, int terms, double* partials) {
  const NodeDesc nd = P.nodes[node];
  const TermList L = P.lists[terms];
  const double2* x = P.pool + nd.off;
  const long long N = nd.size;
  double e = 0, nn = 0;
  OpStage& os = s_os;
  const int nt = L.count < TTNS_MAX_TERMS ? L.count : TTNS_MAX_TERMS;
  for (int t = threadIdx.x; t < nt; t += blockDim.x) os.terms[t] = P.terms[L.first + t];
  if (threadIdx.x == 0) {
    os.a_off = os.b_off = 0;
    os.a_n = os.b_n = 0;
    os.end = 0;
  }
  __syncthreads();
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (long long)gridDim.x * blockDim.x) {
    auto a = apply_stage2_at<double>(P, nd, x, L, P.work + (long long)P.mmax * P.kvec, P.kvec, idx, os);
    double2 v = x[idx];
    e = fma(v.x, a.x, fma(v.y, a.y, e));
    nn = fma(v.x, v.x, fma(v.y, v.y, nn));
  }
  __shared__ double s1[NWARP], s2[NWARP];
  e = warp_sum(e);
  nn = warp_sum(nn);
  if ((threadIdx.x & 31) == 0) { s1[threadIdx.x >> 5] = e; s2[threadIdx.x >> 5] = nn; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int w = 0; w < NWARP; ++w) { a += s1[w]; b += s2[w]; }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = b;
  }
}

// stage 1 of a term list over a whole tensor, written to the worker-0 temporaries
__global__ void k_stage1(KernelParams P, int node, int terms) {
  const NodeDesc nd = P.nodes[node];
  const TermList L = P.lists[terms];
  const Term* tl = P.terms + L.first + (L.count - L.n2);
  const double2* x = P.pool + nd.off;
  double2* tmp = P.work + (long long)P.mmax * P.kvec;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < nd.size; idx += (long long)gridDim.x * blockDim.x) {
    for (int t = 0; t < L.n2; ++t) {
      const Factor f = tl[t].f[0];
      LegPos lp = leg_pos(nd, f.leg, idx);
      auto a = mode_dot<double>(P.pool + f.mat + (long long)lp.i * nd.dims[f.leg], nd.dims[f.leg], x, lp.base,
                                nd.strides[f.leg]);
      tmp[t * P.kvec + idx] = a;
    }
  }
}

// H x for an explicit input x with a node's term list (FP64): stage 1 of the two-stage terms
// into the worker-0 temporaries, then y = the sum of all terms
__global__ void k_stage1_x(KernelParams P, int node, int terms, const double2* x) {
  const NodeDesc nd = P.nodes[node];
  const TermList L = P.lists[terms];
  const Term* tl = P.terms + L.first + (L.count - L.n2);
  double2* tmp = P.work + (long long)P.mmax * P.kvec;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < nd.size;
       idx += (long long)gridDim.x * blockDim.x) {
    for (int t = 0; t < L.n2; ++t) {
      const Factor f = tl[t].f[0];
      LegPos lp = leg_pos(nd, f.leg, idx);
      tmp[t * P.kvec + idx] = mode_dot<double>(P.pool + f.mat + (long long)lp.i * nd.dims[f.leg], nd.dims[f.leg], x,
                                               lp.base, nd.strides[f.leg]);
    }
  }
}

// (blockIdx.y: vector of a batch, P.kvec apart; more than one only without two-stage terms)
__global__ void k_apply_x(KernelParams P, int node, int terms, const double2* x, double2* y) {
  const NodeDesc nd = P.nodes[node];
  const TermList L = P.lists[terms];
  OpStage& os = s_os;
  x += (long long)blockIdx.y * P.kvec;
  y += (long long)blockIdx.y * P.kvec;
  const int nt = L.count < TTNS_MAX_TERMS ? L.count : TTNS_MAX_TERMS;
  for (int t = threadIdx.x; t < nt; t += blockDim.x) os.terms[t] = P.terms[L.first + t];
  if (threadIdx.x == 0) {
    os.a_off = os.b_off = 0;
    os.a_n = os.b_n = 0;
    os.end = 0;
  }
  __syncthreads();
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < nd.size;
       idx += (long long)gridDim.x * blockDim.x)
    y[idx] = apply_stage2_at<double>(P, nd, x, L, P.work + (long long)P.mmax * P.kvec, P.kvec, idx, os);
}

cudaError_t launch_apply_x(const KernelParams& P, int node, int terms, int n2, const double2* x, double2* y,
                           int nblocks, int count, cudaStream_t st) {
  if (n2 > 0) k_stage1_x<<<nblocks, NT, 0, st>>>(P, node, terms, x);
  k_apply_x<<<dim3(nblocks, count), NT, 0, st>>>(P, node, terms, x, y);
  return cudaGetLastError();
}

// Self-test of the bounded wait: two CTAs; with `skip` set the second CTA never
// arrives at the barrier, so the first one must give up after spin_limit cycles.
__global__ void k_wait_selftest(Ctl* ctl, long long spin_limit, int skip) {
  if (skip && blockIdx.x == 1) return;
  grid_sync(ctl, spin_limit);
}

cudaError_t launch_wait_selftest(Ctl* ctl, long long spin_limit, int skip, cudaStream_t st) {
  void* args[] = {&ctl, &spin_limit, &skip};
  return cudaLaunchCooperativeKernel((void*)k_wait_selftest, dim3(2), dim3(NT), args, 0, st);
}

// Copy of a node tensor into a tensor of the same legs with larger (or equal) dimensions,
// zero on the new indices (row-major, legs in the node's order)
__global__ void k_pad_copy(const double2* src, NodeDesc so, double2* dst, NodeDesc dn) {
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < dn.size;
       idx += (long long)gridDim.x * blockDim.x) {
    long long rem = idx, off = 0;
    bool in = true;
    for (int l = 0; l < dn.nl; ++l) {
      const long long i = rem / dn.strides[l];
      rem -= i * dn.strides[l];
      in = in && i < so.dims[l];
      off += i * so.strides[l];
    }
    dst[idx] = in ? src[off] : make_double2(0.0, 0.0);
  }
}

cudaError_t launch_pad_copy(const double2* src_pool, const NodeDesc& so, double2* dst_pool, const NodeDesc& dn,
                            cudaStream_t st) {
  long long nb = (dn.size + 255) / 256;
  nb = nb > 4096 ? 4096 : (nb < 1 ? 1 : nb);
  k_pad_copy<<<(int)nb, 256, 0, st>>>(src_pool + so.off, so, dst_pool + dn.off, dn);
  return cudaGetLastError();
}

// FP32 mirror of the pool (after the pool was written from the host)
__global__ void k_mirror32(const double2* pool, float2* pool32, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    pool32[i] = make_float2((float)pool[i].x, (float)pool[i].y);
}

cudaError_t launch_mirror32(const double2* pool, float2* pool32, long long n, cudaStream_t st) {
  long long nb = (n + 255) / 256;
  nb = nb > 4096 ? 4096 : (nb < 1 ? 1 : nb);
  k_mirror32<<<(int)nb, 256, 0, st>>>(pool, pool32, n);
  return cudaGetLastError();
}

#endif

// ------------------------------------------------------------------ host launch helpers
static bool g_tables_set = false;

static cudaError_t upload_constants() {
  if (g_tables_set) return cudaSuccess;
  double inv[256];
  inv[0] = 0.0;
  for (int k = 1; k < 256; ++k) inv[k] = 1.0 / k;
  const cudaError_t e = cudaMemcpyToSymbol(c_inv, inv, sizeof(inv));
  if (e == cudaSuccess) g_tables_set = true;
  return e;
}

cudaError_t launch_sweep(const KernelParams& P, int phase, int grid, int cluster, int cooperative,
                         cudaStream_t stream) {
  cudaError_t e = upload_constants();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sweep, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.smem_bytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = (size_t)P.smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeCooperative;
  at[1].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = cooperative ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_sweep, P, phase);
}

cudaError_t max_grid_for(int cluster, long long smem_bytes, int* grid) {
  cudaError_t e = cudaFuncSetAttribute(k_sweep, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = (size_t)smem_bytes;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int nclusters = 0;
  e = cudaOccupancyMaxActiveClusters(&nclusters, k_sweep, &cfg);
  if (e != cudaSuccess) return e;
  *grid = nclusters * cluster;
  return cudaSuccess;
}

#ifndef SWEEP_PAIR
cudaError_t launch_density(const double2* pool, const NodeDesc& nd, int l, double* partials, int nblocks, double* out,
                           cudaStream_t st) {
  k_density_partial<<<nblocks, NT, 0, st>>>(pool + nd.off, nd, l, partials);
  const int D = nd.dims[l];
  k_reduce_partials<<<(2 * D * D + NWARP - 1) / NWARP, NT, 0, st>>>(partials, nblocks, 2 * D * D, out);
  return cudaGetLastError();
}

cudaError_t launch_energy(const KernelParams& P, int node, int terms, int n2, double* partials, int nblocks,
                          double* out, cudaStream_t st) {
  if (n2 > 0) k_stage1<<<nblocks, NT, 0, st>>>(P, node, terms);
  k_energy_partial<<<nblocks, NT, 0, st>>>(P, node, terms, partials);
  k_reduce_partials<<<1, NT, 0, st>>>(partials, nblocks, 2, out);
  return cudaGetLastError();
}

#endif
#ifdef SWEEP_PAIR
}  // namespace pair
#endif
}  // namespace ttns
