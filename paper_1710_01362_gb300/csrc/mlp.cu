// Kernels of the surrogate network (a multilayer perceptron from Hamiltonian parameters to
// population trajectories): the dense layer products on the tensor cores with fused
// epilogues, the bias gradients, the loss gradient and the Adam update.  The paper has no
// network; it names machine learning among the advances its method builds on
// (Introduction).  These kernels are the training and inference engine of this library's
// surrogate, with the plain TTNS sweep as its fallback.
//
// Layer product C = op(A) op(B) on tcgen05, one tile of 128 rows and NP = 32 or 64 columns per
// CTA, optionally with K split over the CTAs of a cluster.  Every MMA K step accumulates into
// its own TMEM columns and the steps are summed in registers in FP32 round-to-nearest (the tensor
// core's own FP32 accumulation rounds toward zero, about -0.4 ulp per instruction):
//   kind 1 (TF32X3): FP32-level products for training;
//   kind 3 (BF16X1): one BF16 product, for inference.
//
// What bounds it: latency.  The products here are small (a 256 x 256 x 256 layer is 34 MFLOP), so
// a CTA's own chain (load, split, MMA, read back, store) is the time, and the split decides how
// many SMs share it: 128 x 128 tiles ran that layer on 4 CTAs with scalar loads.  The tile is
// narrowed, then K is split, until the grid covers most of the 152 SMs; operands are loaded 16
// bytes at a time and written as whole 16-byte core-matrix rows.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "../../include/ttns.h"
#include "tc.cuh"

namespace cg = cooperative_groups;

namespace ttns {
void set_last_error(const std::string& msg);

namespace {
constexpr int kNT = 256;
constexpr int kTM = 128;             // rows per CTA (MMA M)
constexpr int kTmem = 256;           // tensor-memory columns per CTA (two CTAs fit an SM)
constexpr int kSplitMax = 8;
constexpr int kGroup = 4;            // K steps added to one partial sum before it joins the total

// status word of the layer products (TTNS_E_TIMEOUT when a completion wait gave up); a
// file-scope device variable, so that no call allocates (the calls can be captured in a graph)
__device__ int g_mlp_status;

struct GemmArgs {
  int M, N, K;
  const float* A;
  int lda, transA;  // A(m, k) = transA ? A[k * lda + m] : A[m * lda + k]
  const float* B;
  int ldb, transB;  // B(k, n) = transB ? B[n * ldb + k] : B[k * ldb + n]
  float* C;
  int ldc;
  int epi;          // 0 C = AB, 1 C = AB + bias, 2 C = tanh(AB + bias), 3 C = AB * (1 - aux^2)
  const float* aux; // bias (epi 1, 2: N values) or the layer output h (epi 3: M x N, ldc)
  long long spin_limit;
  int slots;        // partial sums that a CTA with blockIdx.z > 0 keeps apart
};

// Stages rows [r0, r0 + R) x k in [k0, k0 + kn) of an operand as K-major split planes.  Element
// (r, k) is X[r * ld + k] (kmaj) or X[k * ld + r]; outside rmax x kmax it is zero.  An item is one
// 16-byte core-matrix row of E = 16 / esize values along k (kmaj), or four rows of them.  vec: 16-
// byte loads are aligned (base, ld and k0, r0 are multiples of four floats).
template <int KIND>
__device__ __forceinline__ void stage_operand(unsigned char* dst, uint32_t plane, const float* X, int ld, bool kmaj,
                                              bool vec, int r0, int R, int rmax, int k0, int kn, int kmax) {
  using S = tc::Split<KIND>;
  constexpr int E = 16 / S::esize;
  const int nkg = kn / E;
  auto put = [&](int r, int kg, const float* v) {  // E values of row r
    unsigned char* o = dst + (uint32_t)((r >> 3) * nkg + kg) * 128u + (uint32_t)(r & 7) * 16u;
    if constexpr (KIND == tc::KIND_TF32X3) {
      float h[4], l[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        h[q] = tc::to_tf32(v[q]);
        l[q] = tc::to_tf32(v[q] - h[q]);
      }
      *reinterpret_cast<float4*>(o) = make_float4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<float4*>(o + plane) = make_float4(l[0], l[1], l[2], l[3]);
    } else {
      __nv_bfloat162 b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
      *reinterpret_cast<uint4*>(o) = *reinterpret_cast<uint4*>(b);
    }
  };
  if (kmaj) {
    // consecutive threads: 8 rows, then k groups (whole 128-byte blocks in shared memory)
    for (int it = threadIdx.x; it < R * nkg; it += kNT) {
      const int r8 = it & 7, kg = (it >> 3) % nkg, rb = (it >> 3) / nkg;
      const int r = rb * 8 + r8, row = r0 + r, k = k0 + kg * E;
      float v[E];
      const float* src = X + (long long)row * ld + k;
      if (vec && row < rmax && k + E <= kmax) {
#pragma unroll
        for (int q = 0; q < E; q += 4) {
          const float4 f = *reinterpret_cast<const float4*>(src + q);
          v[q] = f.x;
          v[q + 1] = f.y;
          v[q + 2] = f.z;
          v[q + 3] = f.w;
        }
      } else {
#pragma unroll
        for (int q = 0; q < E; ++q) v[q] = (row < rmax && k + q < kmax) ? src[q] : 0.0f;
      }
      put(r, kg, v);
    }
  } else {
    // consecutive threads: groups of four rows (contiguous in memory), then k groups
    const int nr4 = R / 4;
    for (int it = threadIdx.x; it < nr4 * nkg; it += kNT) {
      const int r = 4 * (it % nr4), kg = it / nr4;
      const int row = r0 + r, k = k0 + kg * E;
      float v[4][E];
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const float* src = X + (long long)(k + q) * ld + row;
        float f[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (k + q < kmax) {
          if (vec && row + 4 <= rmax) {
            const float4 x = *reinterpret_cast<const float4*>(src);
            f[0] = x.x;
            f[1] = x.y;
            f[2] = x.z;
            f[3] = x.w;
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (row + i < rmax) f[i] = src[i];
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i][q] = f[i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) put(r + i, kg, v[i]);
    }
  }
}

// K steps per chunk: one accumulator of NP columns each
template <int NP>
__host__ __device__ constexpr int chunk_steps() {
  return kTmem / NP;
}

template <int KIND, int NP>
__global__ void __launch_bounds__(kNT, 2) k_mlp_gemm(GemmArgs g) {
  using S = tc::Split<KIND>;
  constexpr int KS = S::kstep;
  constexpr int kSteps = chunk_steps<NP>();
  constexpr int chunk = kSteps * KS;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tbase_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = gridDim.z;  // = cluster size along z
  const unsigned row_tiles = (unsigned)((g.M - 1) / kTM) + 1u;  // (tiles on x: y ends at 65535)
  const int m0 = (int)(blockIdx.x % row_tiles) * kTM, n0 = (int)(blockIdx.x / row_tiles) * NP;
  // this CTA's part of K: whole groups of K steps
  const int steps = (g.K + KS - 1) / KS;
  const int per = ((steps + split - 1) / split + kGroup - 1) / kGroup * kGroup;
  const int kbeg = min(g.K, (int)blockIdx.z * per * KS);
  const int kend = min(g.K, kbeg + per * KS);
  constexpr uint32_t a_plane = (uint32_t)kTM * chunk * S::esize;
  constexpr uint32_t b_plane = (uint32_t)NP * chunk * S::esize;
  constexpr int ldo = NP + 1;
  // The sum runs over groups of four K steps, one group after another from k = 0 whatever the
  // split is: the CTA of the first part carries a running total, the others keep their groups'
  // sums apart (in `slots`; with more groups than slots, neighbours share one).
  float* out = reinterpret_cast<float*>(sm + S::parts * (a_plane + b_plane));
  const int groups = per / kGroup, gps = (groups + g.slots - 1) / g.slots;
  unsigned char* Ap = sm;
  unsigned char* Bp = sm + S::parts * a_plane;
  if (warp == 0) tc::tmem_alloc(&tbase_s, kTmem);
  if (tid == 0) tc::mbar_init(&mbar, 1);
  const bool va = g.lda % 4 == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0;
  const bool vb = g.ldb % 4 == 0 && (reinterpret_cast<uintptr_t>(g.B) & 15) == 0;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = tbase_s;
  const int q4 = warp & 3, half = warp >> 2, my_row = q4 * 32 + lane;
  float acc[NP / 2];  // row my_row, columns half * NP / 2 ..
#pragma unroll
  for (int c = 0; c < NP / 2; ++c) acc[c] = 0.0f;
  int grp = 0;        // groups done
  uint32_t phase = 0;
  bool ok = true;
  for (int k0 = kbeg; k0 < kend && ok; k0 += chunk) {
    const int kn = min(chunk, ((kend - k0 + KS - 1) / KS) * KS);
    stage_operand<KIND>(Ap, a_plane, g.A, g.lda, !g.transA, va, m0, kTM, g.M, k0, kn, kend);
    stage_operand<KIND>(Bp, b_plane, g.B, g.ldb, g.transB != 0, vb, n0, NP, g.N, k0, kn, kend);
    tc::fence_proxy_async();
    __syncthreads();
    const int nsteps = kn / KS;
    if (tid == 0) {
      tc::fence_after();
      for (int ks = 0; ks < nsteps; ++ks)
        tc::issue_kstep<KIND>(tbase + (uint32_t)(ks * NP), Ap, a_plane, Bp, b_plane, NP, kn, ks);
      tc::commit(&mbar);
    }
    const bool w = tc::mbar_wait(&mbar, phase, g.spin_limit);
    tc::fence_after();
    ok = __syncthreads_and(w) != 0;
    if (!ok) break;
    phase ^= 1u;
    const uint32_t lane_base = tbase + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(half * (NP / 2));
#pragma unroll
    for (int g4 = 0; g4 < kSteps; g4 += kGroup) {
      if (g4 >= nsteps) break;
#pragma unroll
      for (int c = 0; c < NP / 2; c += 8) {
        uint32_t r[kGroup][8];
#pragma unroll
        for (int ks = 0; ks < kGroup; ++ks)
          if (g4 + ks < nsteps) tc::tmem_ld8_nowait(lane_base + (uint32_t)((g4 + ks) * NP + c), r[ks]);
        tc::tmem_wait_ld();
        float t[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kGroup; ++ks)
          if (g4 + ks < nsteps) {
            tc::tmem_pin8(r[ks]);
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] += __uint_as_float(r[ks][j]);
          }
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[c + j] += t[j];
      }
      ++grp;
      if (blockIdx.z > 0 && grp % gps == 0) {
        float* o = out + (long long)(grp / gps - 1) * (kTM * ldo) + my_row * ldo + half * (NP / 2);
#pragma unroll
        for (int c = 0; c < NP / 2; ++c) {
          o[c] = acc[c];
          acc[c] = 0.0f;
        }
      }
    }
    tc::fence_before();
    __syncthreads();
  }
  if (!ok) {
    if (tid == 0) atomicCAS(&g_mlp_status, 0, (int)TTNS_E_TIMEOUT);
    tc::mbar_wait(&mbar, phase, g.spin_limit);  // the MMAs in flight finish before TMEM is released
    __syncthreads();
  }
  {  // the total (first part), or the slots not written yet (zero beyond the last group)
    int sl = blockIdx.z > 0 ? grp / gps : 0;
    const int nsl = blockIdx.z > 0 ? (groups + gps - 1) / gps : 1;
    for (; sl < nsl; ++sl) {
      float* o = out + (long long)sl * (kTM * ldo) + my_row * ldo + half * (NP / 2);
#pragma unroll
      for (int c = 0; c < NP / 2; ++c) {
        o[c] = acc[c];
        acc[c] = 0.0f;
      }
    }
  }
  // the CTAs of a split add the parts in order, each a share of the rows
  cg::cluster_group cl = cg::this_cluster();
  const int nsl = (groups + gps - 1) / gps;
  if (split > 1) cl.sync(); else __syncthreads();
  const int rps = kTM / split, rlo = blockIdx.z * rps;
  for (int idx = tid; idx < rps * NP; idx += kNT) {
    const int r = rlo + idx / NP, c = idx % NP;
    const int m = m0 + r, n = n0 + c;
    if (m >= g.M || n >= g.N) continue;
    float v;
    if (split == 1) {
      v = out[r * ldo + c];
    } else {
      v = *cl.map_shared_rank(out + r * ldo + c, 0);
      for (int z = 1; z < split; ++z) {
        const float* o = cl.map_shared_rank(out + r * ldo + c, z);
        for (int q = 0; q < nsl; ++q) v += o[q * (kTM * ldo)];
      }
    }
    if (g.epi == 1 || g.epi == 2) v += g.aux[n];
    if (g.epi == 2) v = tanhf(v);
    if (g.epi == 3) {
      const float h = g.aux[(long long)m * g.ldc + n];
      v *= 1.0f - h * h;
    }
    g.C[(long long)m * g.ldc + n] = v;
  }
  if (split > 1) cl.sync();  // the peers' tiles are read before their CTAs leave
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, kTmem);
}

// out[n] = sum_m X[m * ld + n] (bias gradients), fixed order per column
// (one thread per column, 16 loads in flight: without them each of the M additions waited for its
// own load; 32 columns per block, to use more SMs)
__global__ void __launch_bounds__(32) k_colsum(const float* X, int M, int N, int ld, float* out) {
  const int n = blockIdx.x * 32 + threadIdx.x;
  if (n >= N) return;
  float s = 0.0f;
  int m = 0;
  for (; m + 16 <= M; m += 16) {
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = X[(long long)(m + i) * ld + n];
#pragma unroll
    for (int i = 0; i < 16; ++i) s += v[i];
  }
  for (; m < M; ++m) s += X[(long long)m * ld + n];
  out[n] = s;
}

// dy = (y - t) * scale
__global__ void k_diff(const float* y, const float* t, float* dy, long long n, float scale) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dy[i] = (y[i] - t[i]) * scale;
}

__global__ void k_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

template <int KIND, int NP>
cudaError_t launch_tile(GemmArgs g, int split, cudaStream_t st) {
  using S = tc::Split<KIND>;
  constexpr size_t planes = (size_t)S::parts * (kTM + NP) * (chunk_steps<NP>() * S::kstep) * S::esize;
  constexpr size_t tile = (size_t)kTM * (NP + 1) * sizeof(float);
  // at most two CTAs per SM, so that a CTA never waits for tensor memory while its cluster's
  // other CTAs hold some
  constexpr size_t two_per_sm = 80 * 1024, most = 220 * 1024;
  static_assert(2 * kTmem <= 512, "tensor memory of two CTAs");
  const int steps = (g.K + S::kstep - 1) / S::kstep;
  const int groups = ((steps + split - 1) / split + kGroup - 1) / kGroup;
  g.slots = split > 1 ? std::min(groups, (int)((most - planes) / tile)) : 1;
  const size_t smem = std::max(planes + g.slots * tile, two_per_sm);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_gemm<KIND, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  const long long tiles = ((g.M + (long long)kTM - 1) / kTM) * ((g.N + (long long)NP - 1) / NP);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  cfg.gridDim = dim3((unsigned)tiles, 1, split);
  cfg.blockDim = dim3(kNT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = split;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mlp_gemm<KIND, NP>, g);
}

// The widest tile that still gives the chip most of its 152 SMs (each narrowing stages the rows
// of A once more), then K split in up to eight parts of at least four K steps each until there
// are CTAs for all of them (a CTA's K chunks run one after another).
template <int KIND>
cudaError_t launch_gemm(const GemmArgs& g, cudaStream_t st) {
  constexpr int kFill = 96, kFillSplit = 160;
  const long long rt = (g.M + kTM - 1) / kTM;
  auto ctas = [&](int np) { return rt * ((g.N + np - 1) / np); };
  const int np = ctas(64) >= kFill ? 64 : 32;
  const int steps = (g.K + tc::Split<KIND>::kstep - 1) / tc::Split<KIND>::kstep;
  int split = 1;
  while (split < kSplitMax && ctas(np) * split < kFillSplit && steps >= 2 * kGroup * split) split *= 2;
  if (np == 64) return launch_tile<KIND, 64>(g, split, st);
  return launch_tile<KIND, 32>(g, split, st);
}
}  // namespace
}  // namespace ttns

using ttns::set_last_error;

extern "C" ttns_status ttns_mlp_gemm(int kind, int M, int N, int K, const float* A, int lda, int transA,
                                     const float* B, int ldb, int transB, float* C, int ldc, int epilogue,
                                     const float* aux, void* cuda_stream) {
  if (!A || !B || !C || ((epilogue >= 1) && !aux)) {
    set_last_error("ttns_mlp_gemm: NULL pointer");
    return TTNS_E_INVALID;
  }
  if ((kind != 1 && kind != 3) || M < 1 || N < 1 || K < 1 || epilogue < 0 || epilogue > 3 || lda < 1 || ldb < 1 ||
      ldc < N || (!transA && lda < K) || (transA && lda < M) || (!transB && ldb < N) || (transB && ldb < K)) {
    set_last_error("ttns_mlp_gemm: bad kind, size, leading dimension or epilogue");
    return TTNS_E_INVALID;
  }
  ttns::GemmArgs g{M, N, K, A, lda, transA, B, ldb, transB, C, ldc, epilogue, aux, 20000000000LL, 1};
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaError_t e = kind == 1 ? ttns::launch_gemm<ttns::tc::KIND_TF32X3>(g, s) : ttns::launch_gemm<ttns::tc::KIND_BF16X1>(g, s);
  if (e != cudaSuccess) {
    set_last_error(std::string("ttns_mlp_gemm: ") + cudaGetErrorString(e));
    return TTNS_E_CUDA;
  }
  return TTNS_OK;
}

extern "C" ttns_status ttns_mlp_colsum(const float* X, int M, int N, int ld, float* out, void* cuda_stream) {
  if (!X || !out || M < 1 || N < 1 || ld < N) {
    set_last_error("ttns_mlp_colsum: bad arguments");
    return TTNS_E_INVALID;
  }
  ttns::k_colsum<<<(N + 31) / 32, 32, 0, (cudaStream_t)cuda_stream>>>(X, M, N, ld, out);
  return cudaGetLastError() == cudaSuccess ? TTNS_OK : TTNS_E_CUDA;
}

extern "C" ttns_status ttns_mlp_diff(const float* y, const float* t, float* dy, long long n, float scale,
                                     void* cuda_stream) {
  if (!y || !t || !dy || n < 1) {
    set_last_error("ttns_mlp_diff: bad arguments");
    return TTNS_E_INVALID;
  }
  ttns::k_diff<<<(int)std::min<long long>(1024, (n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(y, t, dy, n, scale);
  return cudaGetLastError() == cudaSuccess ? TTNS_OK : TTNS_E_CUDA;
}

extern "C" ttns_status ttns_mlp_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float beta1,
                                     float beta2, float eps, int step, void* cuda_stream) {
  if (!p || !g || !m || !v || n < 1 || step < 1 || !(lr > 0)) {
    set_last_error("ttns_mlp_adam: bad arguments");
    return TTNS_E_INVALID;
  }
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  ttns::k_adam<<<(int)std::min<long long>(1024, (n + 255) / 256), 256, 0, (cudaStream_t)cuda_stream>>>(
      p, g, m, v, n, lr, beta1, beta2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? TTNS_OK : TTNS_E_CUDA;
}

extern "C" ttns_status ttns_mlp_status(int* device_status, int clear) {
  if (!device_status) return TTNS_E_INVALID;
  if (cudaDeviceSynchronize() != cudaSuccess ||
      cudaMemcpyFromSymbol(device_status, ttns::g_mlp_status, sizeof(int)) != cudaSuccess)
    return TTNS_E_CUDA;
  if (clear) {
    const int zero = 0;
    if (cudaMemcpyToSymbol(ttns::g_mlp_status, &zero, sizeof(int)) != cudaSuccess) return TTNS_E_CUDA;
  }
  return TTNS_OK;
}
