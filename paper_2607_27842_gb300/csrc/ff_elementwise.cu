// Bandwidth-bound kernels of the FeatFix denoising step: the draft (Eq. 2),
// the fused paid check / forward (Eqs. 3-5), adaLN LayerNorm-modulation,
// conditioning tables, embedding, sampler update and the seeded latent.
// (Times in the comments: launches back to back in a CUDA graph.)
#include "ff_common.cuh"

#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace cg = cooperative_groups;

namespace ff {

static std::atomic<long long> g_launches{0};
void count_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches_total() { return g_launches.load(std::memory_order_relaxed); }

static int g_num_sms = 0;
static int num_sms() {
  if (g_num_sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 148;
  }
  return g_num_sms;
}

// ---------------------------------------------------------------------------
// Draft (Eq. 2, weight form): x <- x + sum_j w_j R_j.  One 16-byte vector per
// thread per iteration, every operand streamed once, grid-stride over a grid
// sized to a multiple of the SM count.
// ---------------------------------------------------------------------------
template <class T, int NT>
__device__ __forceinline__ void draft_vec(const T* __restrict__ xu, const Hist4& h, const float (&w)[4], long long i,
                                          float (&a)[VecN<T>::n]) {
  constexpr int V = VecN<T>::n;
  ld16(xu + i * V, a);
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    float r[V];
    ld16(reinterpret_cast<const T*>(h.p[j]) + i * V, r);
#pragma unroll
    for (int q = 0; q < V; ++q) a[q] = __fmaf_rn(w[j], r[q], a[q]);
  }
}

template <class T, int NT>
__device__ __forceinline__ float draft_scalar(const T* xu, const Hist4& h, const float (&w)[4], long long i) {
  float a = to_f(xu[i]);
#pragma unroll
  for (int j = 0; j < NT; ++j) a = __fmaf_rn(w[j], to_f(reinterpret_cast<const T*>(h.p[j])[i]), a);
  return a;
}

template <class T, int NT>
__global__ void __launch_bounds__(256) k_draft(T* __restrict__ x, Hist4 h, float w0, float w1, float w2, float w3,
                                               long long n) {
  pdl_trigger();
  pdl_wait();
  constexpr int V = VecN<T>::n;
  const float w[4] = {w0, w1, w2, w3};
  const long long nvec = n / V;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += stride) {
    float a[V];
    draft_vec<T, NT>(x, h, w, i, a);
    st16(x + i * V, a);
  }
  if (blockIdx.x == 0 && threadIdx.x < n - nvec * V) {
    const long long i = nvec * V + threadIdx.x;
    x[i] = from_f<T>(draft_scalar<T, NT>(x, h, w, i));
  }
}

static int stream_grid(long long nvec, int threads) {
  long long want = (nvec + threads - 1) / threads;
  long long cap = (long long)num_sms() * 8;
  if (want > cap) want = cap;
  if (want < 1) want = 1;
  return (int)want;
}

template <class T>
static cudaError_t draft_t(void* x, const Hist4& h, const float* w, int nt, long long n, cudaStream_t s) {
  const int grid = stream_grid(n / VecN<T>::n, 256);
  T* xp = reinterpret_cast<T*>(x);
  switch (nt) {
    case 1: launch_pdl(k_draft<T, 1>, grid, 256, 0, s, xp, h, w[0], w[1], w[2], w[3], n); break;
    case 2: launch_pdl(k_draft<T, 2>, grid, 256, 0, s, xp, h, w[0], w[1], w[2], w[3], n); break;
    case 3: launch_pdl(k_draft<T, 3>, grid, 256, 0, s, xp, h, w[0], w[1], w[2], w[3], n); break;
    case 4: launch_pdl(k_draft<T, 4>, grid, 256, 0, s, xp, h, w[0], w[1], w[2], w[3], n); break;
    default: return cudaErrorInvalidValue;
  }
  return launched();
}

cudaError_t launch_draft(DType dt, void* x, const Hist4& h, const float* w, int nt, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return dt == F32 ? draft_t<float>(x, h, w, nt, n, s) : draft_t<bf16>(x, h, w, nt, n, s);
}

// A run of nblk drafted blocks in one pass: x <- x + sum_b sum_j w_j R_{b,j}.
// Each block's draft adds its forecast increment to the incoming state, so
// the run's blocks telescope; x is read and written once instead of once
// per block, and the sum stays in fp32 until the end.
template <class T, int NT>
__global__ void __launch_bounds__(256) k_draft_seg(T* __restrict__ x, const __grid_constant__ HistSeg h, int nblk,
                                                   float w0, float w1, float w2, float w3, long long n) {
  pdl_trigger();
  pdl_wait();
  constexpr int V = VecN<T>::n;
  const float w[4] = {w0, w1, w2, w3};
  const long long nvec = n / V;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += stride) {
    float a[V];
    ld16(x + i * V, a);
    for (int b = 0; b < nblk; ++b) {
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        float r[V];
        ld16(reinterpret_cast<const T*>(h.p[b][j]) + i * V, r);
#pragma unroll
        for (int q = 0; q < V; ++q) a[q] = __fmaf_rn(w[j], r[q], a[q]);
      }
    }
    st16(x + i * V, a);
  }
  if (blockIdx.x == 0 && threadIdx.x < n - nvec * V) {
    const long long i = nvec * V + threadIdx.x;
    float a = to_f(x[i]);
    for (int b = 0; b < nblk; ++b) {
#pragma unroll
      for (int j = 0; j < NT; ++j) a = __fmaf_rn(w[j], to_f(reinterpret_cast<const T*>(h.p[b][j])[i]), a);
    }
    x[i] = from_f<T>(a);
  }
}

template <class T>
static cudaError_t draft_seg_t(void* x, const HistSeg& h, int nblk, const float* w, int nt, long long n,
                               cudaStream_t s) {
  const int grid = stream_grid(n / VecN<T>::n, 256);
  T* xp = reinterpret_cast<T*>(x);
  switch (nt) {
    case 1: launch_pdl(k_draft_seg<T, 1>, grid, 256, 0, s, xp, h, nblk, w[0], w[1], w[2], w[3], n); break;
    case 2: launch_pdl(k_draft_seg<T, 2>, grid, 256, 0, s, xp, h, nblk, w[0], w[1], w[2], w[3], n); break;
    case 3: launch_pdl(k_draft_seg<T, 3>, grid, 256, 0, s, xp, h, nblk, w[0], w[1], w[2], w[3], n); break;
    case 4: launch_pdl(k_draft_seg<T, 4>, grid, 256, 0, s, xp, h, nblk, w[0], w[1], w[2], w[3], n); break;
    default: return cudaErrorInvalidValue;
  }
  return launched();
}

cudaError_t launch_draft_seg(DType dt, void* x, const HistSeg& h, int nblk, const float* w, int nt, long long n,
                             cudaStream_t s) {
  if (n <= 0 || nblk <= 0) return cudaSuccess;
  if (nblk > SEG_MAX) return cudaErrorInvalidValue;
  return dt == F32 ? draft_seg_t<float>(x, h, nblk, w, nt, n, s) : draft_seg_t<bf16>(x, h, nblk, w, nt, n, s);
}

// out = a - b elementwise (fp32 arithmetic, rounded to the storage type).
template <class T>
__global__ void __launch_bounds__(256) k_diff(const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ out,
                                              long long n) {
  pdl_trigger();
  pdl_wait();
  constexpr int V = VecN<T>::n;
  const long long nvec = n / V;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += stride) {
    float x[V], y[V];
    ld16(a + i * V, x);
    ld16(b + i * V, y);
#pragma unroll
    for (int q = 0; q < V; ++q) x[q] -= y[q];
    st16(out + i * V, x);
  }
  if (blockIdx.x == 0 && threadIdx.x < n - nvec * V) {
    const long long i = nvec * V + threadIdx.x;
    out[i] = from_f<T>(to_f(a[i]) - to_f(b[i]));
  }
}

cudaError_t launch_diff(DType dt, const void* a, const void* b, void* out, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (dt == F32) {
    launch_pdl(k_diff<float>, stream_grid(n / 4, 256), 256, 0, s, (const float*)a, (const float*)b, (float*)out, n);
  } else {
    launch_pdl(k_diff<bf16>, stream_grid(n / 8, 256), 256, 0, s, (const bf16*)a, (const bf16*)b, (bf16*)out, n);
  }
  return launched();
}

// ---------------------------------------------------------------------------
// Paid check + forward (Eqs. 3-5), fused so h_f is read once: each thread
// rebuilds h_d from u and the history exactly as k_draft does, accumulates
// |h_d - h_f|, |h_f|, (h_d - h_f)^2, h_f^2, and (Verify arm) stores h_d over
// u.  Reduction: warp shuffles, then shared memory, then the 8 CTAs of a
// thread-block cluster combine through distributed shared memory; one
// partial per cluster goes to the workspace and a one-block kernel adds the
// partials in a fixed order (deterministic run to run).
// ---------------------------------------------------------------------------
constexpr int VERIFY_THREADS = 256;
constexpr int VERIFY_CLUSTER = 8;

// Upper bound of the grid (and so of the partials in the workspace): up to
// four CTAs per SM, whole clusters.
static int verify_grid(long long n) {
  long long nvec = n / 4 + 1;
  long long want = (nvec + VERIFY_THREADS - 1) / VERIFY_THREADS;
  long long cap = (long long)num_sms() * 4;
  if (want > cap) want = cap;
  want = (want + VERIFY_CLUSTER - 1) / VERIFY_CLUSTER * VERIFY_CLUSTER;
  if (want < VERIFY_CLUSTER) want = VERIFY_CLUSTER;
  return (int)want;
}

size_t verify_workspace_bytes(long long n) {
  return (size_t)(verify_grid(n) / VERIFY_CLUSTER) * 4 * sizeof(double);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The clusters' partials ([nparts][4] doubles) added by one warp: lane = (one of
// eight subsequences, quantity), 256 contiguous bytes a step, the eight sums
// combined in a fixed order.  (One thread per quantity walking all partials
// was a chain of dependent L2 reads: n = 1e6, two terms 9.7 -> 6.8
// us; 29.8e6 48.9 -> 45.8 us.)
__device__ __forceinline__ void finish_sums(const double* partials, int nparts, double* sums, int lane) {
  double t = 0.0;
#pragma unroll 4
  for (int k = lane; k < 4 * nparts; k += 32) t += __ldcg(partials + k);
#pragma unroll
  for (int o = 4; o <= 16; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane < 4) sums[lane] = t;
}

// Partial forwarding (token- or channel-level arm): mix != nullptr gets
// h_f where the element's row (rmask) or column (cmask) is selected and h_d
// elsewhere; mix may be the h_f buffer itself (each element is read, then
// written, by the same thread).
template <class T, int NT>
__global__ void __cluster_dims__(VERIFY_CLUSTER, 1, 1) __launch_bounds__(VERIFY_THREADS, 4)
    k_verify(T* __restrict__ u, Hist4 h, float w0, float w1, float w2, float w3, const T* hf,
             long long n, int write_draft, double* partials, T* mix,
             const unsigned char* __restrict__ rmask, const unsigned char* __restrict__ cmask, int C,
             unsigned int* done_ctr, double* __restrict__ sums) {
  pdl_trigger();
  pdl_wait();
  constexpr int V = VecN<T>::n;
  const float w[4] = {w0, w1, w2, w3};
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
  const long long nvec = n / V;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // One vector of u, the history and h_f, accumulated, stored (Verify) and
  // mixed (partial forwarding).
  auto one = [&](long long i, float (&a)[V], const float (&f)[V]) {
#pragma unroll
    for (int q = 0; q < V; ++q) {
      const float ad = round_to(a[q], (T*)nullptr);  // h_d as it would be forwarded
      const float d = ad - f[q];
      s0 += fabsf(d);
      s1 += fabsf(f[q]);
      s2 += d * d;
      s3 += f[q] * f[q];
    }
    if (write_draft) st16(u + i * V, a);
    if (mix) {  // C % V == 0: the vector lies in one row
      const long long e0 = i * V;
      const long long r = e0 / C;
      const int c0 = (int)(e0 - r * C);
      float o[V];
#pragma unroll
      for (int q = 0; q < V; ++q) o[q] = (rmask ? rmask[r] : cmask[c0 + q]) ? f[q] : a[q];
      st16(mix + i * V, o);
    }
  };
  // Two vectors per thread and iteration, all their loads issued before
  // either is used: the grid holds at most four CTAs per SM (the partials
  // stay small), so each thread keeps twice the bytes in flight instead.
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + stride < nvec; i += 2 * stride) {
    float a[V], f[V], a2[V], f2[V];
    draft_vec<T, NT>(u, h, w, i, a);
    draft_vec<T, NT>(u, h, w, i + stride, a2);
    ld16(hf + i * V, f);
    ld16(hf + (i + stride) * V, f2);
    one(i, a, f);
    one(i + stride, a2, f2);
  }
  if (i < nvec) {
    float a[V], f[V];
    draft_vec<T, NT>(u, h, w, i, a);
    ld16(hf + i * V, f);
    one(i, a, f);
  }
  if (blockIdx.x == 0 && threadIdx.x < n - nvec * V) {
    const long long i = nvec * V + threadIdx.x;
    const float a = round_to(draft_scalar<T, NT>(u, h, w, i), (T*)nullptr);
    const float f = to_f(hf[i]);
    const float d = a - f;
    s0 += fabsf(d); s1 += fabsf(f); s2 += d * d; s3 += f * f;
    if (write_draft) u[i] = from_f<T>(a);
    if (mix) mix[i] = from_f<T>((rmask ? rmask[i / C] : cmask[i % C]) ? f : a);
  }
  s0 = warp_sum(s0); s1 = warp_sum(s1); s2 = warp_sum(s2); s3 = warp_sum(s3);
  __shared__ float wsum[VERIFY_THREADS / 32][4];
  __shared__ double bsum[4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { wsum[warp][0] = s0; wsum[warp][1] = s1; wsum[warp][2] = s2; wsum[warp][3] = s3; }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int k = 0; k < VERIFY_THREADS / 32; ++k) t += (double)wsum[k][threadIdx.x];
    bsum[threadIdx.x] = t;
  }
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  if (cluster.block_rank() == 0 && threadIdx.x < 32) {
    if (threadIdx.x < 4) {
      double t = 0.0;
      for (unsigned r = 0; r < cluster.num_blocks(); ++r) {
        const double* rb = cluster.map_shared_rank(bsum, r);
        t += rb[threadIdx.x];
      }
      partials[(size_t)(blockIdx.x / VERIFY_CLUSTER) * 4 + threadIdx.x] = t;
      __threadfence();
    }
    // With a completion counter the last cluster to finish sums every
    // cluster's partials (in the same order whichever cluster is last) and
    // resets the counter for the next launch.
    if (done_ctr) {
      __syncwarp();
      const unsigned int nclusters = gridDim.x / VERIFY_CLUSTER;
      unsigned int last = 0;
      if (threadIdx.x == 0) last = atomicAdd(done_ctr, 1u) == nclusters - 1 ? 1u : 0u;
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        __threadfence();
        finish_sums(partials, (int)nclusters, sums, threadIdx.x);
        if (threadIdx.x == 0) *done_ctr = 0u;
      }
    }
  }
  cluster.sync();
}

__global__ void k_verify_finish(const double* partials, int nparts, double* sums) {
  pdl_trigger();
  pdl_wait();
  finish_sums(partials, nparts, sums, threadIdx.x);
}

// The launched grid: verify_grid's bound, cut to the clusters that are
// resident at once.  Clusters of 8 CTAs must fit in one GPC, so four CTAs
// per SM on every SM are not all co-resident; a grid sized to them left a
// second wave of a few clusters that ran alone (measured: the paid check at
// 0.6 of the copy rate, with drafts of the same size at 1.0).
template <class T, int NT>
static int verify_launch_grid(long long n) {
  static int resident = -1;  // clusters resident at once (per kernel instance)
  if (resident < 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(VERIFY_CLUSTER * 64);
    cfg.blockDim = dim3(VERIFY_THREADS);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = VERIFY_CLUSTER;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, k_verify<T, NT>, &cfg) != cudaSuccess || nc <= 0) {
      cudaGetLastError();
      nc = 0;  // unknown: keep the bound
    }
    resident = nc;
  }
  int grid = verify_grid(n);
  if (resident > 0 && grid > resident * VERIFY_CLUSTER) grid = resident * VERIFY_CLUSTER;
  return grid;
}

void verify_prepare() {
  verify_launch_grid<float, 1>(1); verify_launch_grid<float, 2>(1);
  verify_launch_grid<float, 3>(1); verify_launch_grid<float, 4>(1);
  verify_launch_grid<bf16, 1>(1); verify_launch_grid<bf16, 2>(1);
  verify_launch_grid<bf16, 3>(1); verify_launch_grid<bf16, 4>(1);
}

template <class T>
static cudaError_t verify_t(void* u, const Hist4& h, const float* w, int nt, const void* hf, long long n,
                           int write_draft, double* sums, void* ws, cudaStream_t s, const FwdMix* fm,
                           unsigned int* done_ctr) {
  const int grid = nt == 1 ? verify_launch_grid<T, 1>(n) : nt == 2 ? verify_launch_grid<T, 2>(n)
                 : nt == 3 ? verify_launch_grid<T, 3>(n) : verify_launch_grid<T, 4>(n);
  double* parts = reinterpret_cast<double*>(ws);
  T* up = reinterpret_cast<T*>(u);
  const T* fp = reinterpret_cast<const T*>(hf);
  T* mx = fm ? reinterpret_cast<T*>(fm->out) : nullptr;
  const unsigned char* rm = fm ? fm->rmask : nullptr;
  const unsigned char* cm = fm ? fm->cmask : nullptr;
  const int C = fm ? fm->C : 1;
  if (mx && (C <= 0 || C % VecN<T>::n != 0 || (!rm && !cm) || n % C != 0)) return cudaErrorInvalidValue;
  switch (nt) {
    case 1: launch_pdl(k_verify<T, 1>, grid, VERIFY_THREADS, 0, s, up, h, w[0], w[1], w[2], w[3], fp, n, write_draft, parts, mx, rm, cm, C, done_ctr, sums); break;
    case 2: launch_pdl(k_verify<T, 2>, grid, VERIFY_THREADS, 0, s, up, h, w[0], w[1], w[2], w[3], fp, n, write_draft, parts, mx, rm, cm, C, done_ctr, sums); break;
    case 3: launch_pdl(k_verify<T, 3>, grid, VERIFY_THREADS, 0, s, up, h, w[0], w[1], w[2], w[3], fp, n, write_draft, parts, mx, rm, cm, C, done_ctr, sums); break;
    case 4: launch_pdl(k_verify<T, 4>, grid, VERIFY_THREADS, 0, s, up, h, w[0], w[1], w[2], w[3], fp, n, write_draft, parts, mx, rm, cm, C, done_ctr, sums); break;
    default: return cudaErrorInvalidValue;
  }
  cudaError_t e = launched();
  if (e != cudaSuccess || done_ctr) return e;
  launch_pdl(k_verify_finish, 1, 32, 0, s, parts, grid / VERIFY_CLUSTER, sums);
  return launched();
}

cudaError_t launch_verify(DType dt, void* u, const Hist4& h, const float* w, int nt, const void* hf, long long n,
                          int write_draft, double* sums, void* ws, cudaStream_t s, const FwdMix* mix,
                          unsigned int* done_ctr) {
  if (n <= 0) return cudaErrorInvalidValue;
  return dt == F32 ? verify_t<float>(u, h, w, nt, hf, n, write_draft, sums, ws, s, mix, done_ctr)
                   : verify_t<bf16>(u, h, w, nt, hf, n, write_draft, sums, ws, s, mix, done_ctr);
}

// ---------------------------------------------------------------------------
// Operand rows of the fused-LayerNorm correction GEMMs: for job j (one
// LayerNorm of one block and stream) and modulation row r,
//   out[j][2r] = 1 + scale_r,  out[j][2r + 1] = shift_r
// (columns jobs[j].x and jobs[j].y of the row), so one GEMM with the layer's
// weight gives (1 + s) W^T and sh W^T interleaved.
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(256) k_ln_ab(const float* __restrict__ mod, long long mod_stride, int C,
                                               const int2* __restrict__ jobs, T* __restrict__ out,
                                               long long job_stride) {
  pdl_trigger();
  pdl_wait();
  const int r = blockIdx.x, j = blockIdx.y;
  const int2 jc = jobs[j];
  const float* sc = mod + (size_t)r * mod_stride + jc.x;
  const float* sh = mod + (size_t)r * mod_stride + jc.y;
  T* o = out + (size_t)j * job_stride + (size_t)2 * r * C;
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    o[c] = from_f<T>(1.0f + sc[c]);
    o[C + c] = from_f<T>(sh[c]);
  }
}

cudaError_t launch_ln_ab(DType dt, const float* mod, long long mod_stride, int rows, int C, const int2* jobs,
                         int njobs, void* out, long long job_stride, cudaStream_t s) {
  if (rows <= 0 || njobs <= 0) return cudaSuccess;
  const dim3 grid(rows, njobs);
  if (dt == F32)
    launch_pdl(k_ln_ab<float>, grid, dim3(256), 0, s, mod, mod_stride, C, jobs, (float*)out, job_stride);
  else
    launch_pdl(k_ln_ab<bf16>, grid, dim3(256), 0, s, mod, mod_stride, C, jobs, (bf16*)out, job_stride);
  return launched();
}

// ---------------------------------------------------------------------------
// adaLN branch input: LN(x) (no affine, eps 1e-6) * (1 + scale_b) + shift_b.
// One warp per row, exact two-pass mean / variance from registers, one global
// read and one write.
// ---------------------------------------------------------------------------
// One warp per row (8 rows per block, for row counts of one wave of resident
// blocks); the block first stages the shift /
// scale vectors of its first row's sample in shared memory (coalesced, read
// back by every warp of that sample instead of 4 x 16 B per lane per chunk
// from global memory).  Rows of up to six vectors per lane are held to 64
// registers, so four blocks share an SM (4096 rows of 1152: one wave).
template <class T, int NCH>
__global__ void __launch_bounds__(256, NCH <= 6 ? 4 : 1) k_ln_mod1(const T* __restrict__ x, T* __restrict__ out, long long rows, int C,
                                                const float* __restrict__ shift, const float* __restrict__ scale,
                                                int mod_stride, int seg_split, int rpb0, int rpb1) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float4 smod4[];                  // [2 * C / 4]: shift, then scale
  float* smod = reinterpret_cast<float*>(smod4);
  constexpr int V = VecN<T>::n;
  const long long r0 = (long long)blockIdx.x * 8;
  const int b0 = (int)(r0 < seg_split ? r0 / rpb0 : (r0 - seg_split) / rpb1);
  {
    const float4* sh4 = reinterpret_cast<const float4*>(shift + (size_t)b0 * mod_stride);
    const float4* sc4 = reinterpret_cast<const float4*>(scale + (size_t)b0 * mod_stride);
    for (int i = threadIdx.x; i < C / 4; i += blockDim.x) {
      smod4[i] = sh4[i];
      smod4[C / 4 + i] = sc4[i];
    }
  }
  __syncthreads();
  const long long r = r0 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const T* xr = x + r * C;
  const int nv = C / V;
  float a[NCH][V];
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const int k = lane + 32 * j;
    if (k < nv) {
      ld16(xr + k * V, a[j]);
#pragma unroll
      for (int q = 0; q < V; ++q) s += a[j][q];
    }
  }
  s = warp_sum(s);
  const float mean = s / C;
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    if (lane + 32 * j < nv) {
#pragma unroll
      for (int q = 0; q < V; ++q) { const float d = a[j][q] - mean; ss += d * d; }
    }
  }
  ss = warp_sum(ss);
  const float rstd = rsqrtf(ss / C + 1e-6f);
  const int b = (int)(r < seg_split ? r / rpb0 : (r - seg_split) / rpb1);
  // the block's sample from shared memory, a second sample (a block straddling
  // a sample boundary) from global memory
  const float* sh = b == b0 ? smod : shift + (size_t)b * mod_stride;
  const float* sc = b == b0 ? smod + C : scale + (size_t)b * mod_stride;
  T* orow = out + r * C;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const int k = lane + 32 * j;
    if (k < nv) {
      float o[V];
#pragma unroll
      for (int q = 0; q < V; q += 4) {
        const float4 s4 = *reinterpret_cast<const float4*>(sh + k * V + q);
        const float4 c4 = *reinterpret_cast<const float4*>(sc + k * V + q);
        o[q] = (a[j][q] - mean) * rstd * (1.0f + c4.x) + s4.x;
        o[q + 1] = (a[j][q + 1] - mean) * rstd * (1.0f + c4.y) + s4.y;
        o[q + 2] = (a[j][q + 2] - mean) * rstd * (1.0f + c4.z) + s4.z;
        o[q + 3] = (a[j][q + 3] - mean) * rstd * (1.0f + c4.w) + s4.w;
      }
      st16(orow + k * V, o);
    }
  }
}

// Large row counts and wide rows: each block takes a share of the rows, its warps
// every eighth of them.  Rows reach the warp through its own ring of DEPTH slots in
// shared memory by cp.async (each lane copies and reads back its own vectors,
// so a row needs no barrier), so DEPTH rows per warp are in flight while one is
// reduced; the shift / scale of the block's first sample (read back by every
// warp of that sample) are copied the same way behind the first rows, so the
// two latencies overlap.  Written in packed fp32 pairs; scalar arithmetic was as
// fast (14310 x 2048).
// The blocks' shares differ by one row at most: in blocks of equal whole rows of
// warps the last SMs run a block less or none (8000 x 2048: 334 blocks for 456
// slots).  us with rows held a register row ahead, in equal blocks, as here: 8704 x
// 3072 38.4, 25.8, 24.3; 4608 x 3072 22.2, 18.7, 15.1; 8000 x 2048 17.9, 19.1, 16.7;
// 8192 x 1152 15.2, 10.3, 9.3; 14000 x 128 9.5, 5.1, 5.1; 14310 x 2048 24.9, 24.5,
// 24.2 (4.8 TB/s).
// a 16-byte vector of four fp32 or eight bf16 values <-> pairs
__device__ __forceinline__ void unpack2x(const uint4& v, f32x2 (&p)[2]) {
  p[0] = (f32x2)v.x | ((f32x2)v.y << 32);
  p[1] = (f32x2)v.z | ((f32x2)v.w << 32);
}
__device__ __forceinline__ void unpack2x(const uint4& v, f32x2 (&p)[4]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = bf2u(w[i]);
}
__device__ __forceinline__ uint4 packv(const f32x2 (&o)[2]) {
  return make_uint4((unsigned)o[0], (unsigned)(o[0] >> 32), (unsigned)o[1], (unsigned)(o[1] >> 32));
}
__device__ __forceinline__ uint4 packv(const f32x2 (&o)[4]) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo_f(o[i]), hi_f(o[i]));
    w[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

template <class T, int NCH, int DEPTH>
__global__ void __launch_bounds__(256, NCH <= 6 ? 4 : NCH <= 8 ? 3 : 2)
    k_ln_mod(const T* __restrict__ x, T* __restrict__ out, long long rows, int C, const float* __restrict__ shift,
             const float* __restrict__ scale, int mod_stride, int seg_split, int rpb0, int rpb1, int per, int rem) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ float4 smod4[];                  // [2 * C / 4]: shift, then scale; then the rings
  float* smod = reinterpret_cast<float*>(smod4);
  constexpr int V = VecN<T>::n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the block's rows [r0, r0 + nb): per, one more in the first rem blocks
  const long long r0 = (long long)blockIdx.x * per + min((int)blockIdx.x, rem);
  const int nb = (int)min((long long)per + ((int)blockIdx.x < rem ? 1 : 0), rows - r0);
  const int b0 = (int)(r0 < seg_split ? r0 / rpb0 : (r0 - seg_split) / rpb1);
  const int nv = C / V;
  const long long rw = r0 + warp;                     // the warp's rows rw + 8 t, t < n (n may be 0)
  const int n = (nb - warp + 7) >> 3;
  uint4* const ring = reinterpret_cast<uint4*>(smod4 + C / 2) + (size_t)warp * DEPTH * nv;
  auto copy_row = [&](int t) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + (rw + 8 * t) * C);
    uint4* d = ring + (t % DEPTH) * nv;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const int k = lane + 32 * j;
      if (k < nv) cp_async16(d + k, xr + k);
    }
  };
#pragma unroll
  for (int t = 0; t < DEPTH; ++t) {
    if (t < n) copy_row(t);
    if (t == 0) {
      const float4* sh4 = reinterpret_cast<const float4*>(shift + (size_t)b0 * mod_stride);
      const float4* sc4 = reinterpret_cast<const float4*>(scale + (size_t)b0 * mod_stride);
      for (int i = threadIdx.x; i < C / 4; i += blockDim.x) {
        cp_async16(smod4 + i, sh4 + i);
        cp_async16(smod4 + C / 4 + i, sc4 + i);
      }
    }
    cp_commit();
  }
  cp_wait<DEPTH - 1>();
  for (int i = threadIdx.x; i < C / 4; i += blockDim.x) {   // 1 + scale, each thread its own copies
    float4 v = smod4[C / 4 + i];
    v.x += 1.0f; v.y += 1.0f; v.z += 1.0f; v.w += 1.0f;
    smod4[C / 4 + i] = v;
  }
  __syncthreads();
  for (int t = 0; t < n; ++t) {
    if (t > 0) cp_wait<DEPTH - 1>();
    const long long r = rw + 8 * t;
    // the row as packed fp32 pairs where they fit the registers, else as stored
    // (unpacked again in each pass)
    constexpr bool KEEP = NCH * V <= 32;
    uint4 cur[KEEP ? 1 : NCH];
    f32x2 a[KEEP ? NCH : 1][V / 2];
    const uint4* const slot = ring + (t % DEPTH) * nv;
    f32x2 s2 = 0ull;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      if (lane + 32 * j < nv) {
        const uint4 v = slot[lane + 32 * j];
        if constexpr (!KEEP) cur[j] = v;
        f32x2 (&p)[V / 2] = a[KEEP ? j : 0];
        unpack2x(v, p);
#pragma unroll
        for (int q = 0; q < V / 2; ++q) s2 = fadd2(s2, p[q]);
      }
    }
    const float mean = warp_sum(lo_f(s2) + hi_f(s2)) / C;
    if (t + DEPTH < n) copy_row(t + DEPTH);          // the slot has been read (its values are in the sum)
    cp_commit();
    const f32x2 nm = f2u(-mean, -mean);
    f32x2 ss2 = 0ull;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      if (lane + 32 * j < nv) {
        f32x2 (&p)[V / 2] = a[KEEP ? j : 0];
        if constexpr (!KEEP) unpack2x(cur[j], p);
#pragma unroll
        for (int q = 0; q < V / 2; ++q) {
          const f32x2 d = fadd2(p[q], nm);
          if constexpr (KEEP) p[q] = d;              // centred from here on
          ss2 = ffma2(d, d, ss2);
        }
      }
    }
    const float rstd = rsqrtf(warp_sum(lo_f(ss2) + hi_f(ss2)) / C + 1e-6f);
    const f32x2 rs = f2u(rstd, rstd);
    const int b = (int)(r < seg_split ? r / rpb0 : (r - seg_split) / rpb1);
    uint4* const orow = reinterpret_cast<uint4*>(out + r * C);
    // the block's sample from shared memory (scale already 1 + scale), another
    // sample (a block straddling a sample boundary) from global memory
    auto apply = [&](auto own, const float* sh, const float* sc) {
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
        const int k = lane + 32 * j;
        if (k < nv) {
          f32x2 (&p)[V / 2] = a[KEEP ? j : 0];
          if constexpr (!KEEP) unpack2x(cur[j], p);
          f32x2 o[V / 2];
#pragma unroll
          for (int q = 0; q < V / 2; q += 2) {
            const ulonglong2* const sp = reinterpret_cast<const ulonglong2*>(sh + k * V + 2 * q);
            const ulonglong2* const cp = reinterpret_cast<const ulonglong2*>(sc + k * V + 2 * q);
            ulonglong2 s4, c4;
            if constexpr (decltype(own)::value) {
              s4 = *sp;
              c4 = *cp;
            } else {
              // read-only loads: plain ones may not pass the stores of out, so each
              // vector would wait for its own (8000 x 2048 fp32, two samples 30.6 -> 26.0 us)
              s4 = __ldg(sp);
              c4 = __ldg(cp);
              const f32x2 one = f2u(1.0f, 1.0f);
              c4.x = fadd2(c4.x, one);
              c4.y = fadd2(c4.y, one);
            }
            o[q] = ffma2(fmul2(KEEP ? p[q] : fadd2(p[q], nm), rs), c4.x, s4.x);
            o[q + 1] = ffma2(fmul2(KEEP ? p[q + 1] : fadd2(p[q + 1], nm), rs), c4.y, s4.y);
          }
          orow[k] = packv(o);
        }
      }
    };
    if (b == b0) apply(std::true_type{}, smod, smod + C);
    else apply(std::false_type{}, shift + (size_t)b * mod_stride, scale + (size_t)b * mod_stride);
  }
}

template <class T, int NCH>
static cudaError_t ln_mod_launch(const T* x, T* out, long long rows, int C, const float* shift, const float* scale,
                                 int mod_stride, int seg_split, int rpb0, int rpb1, cudaStream_t s) {
  const long long sms = num_sms(), mods = 2LL * C * 4, row = (long long)C * sizeof(T);
  // A row per warp while that is one wave of k_ln_mod1's resident blocks (64
  // registers and four blocks up to six vectors a lane, then two or three fp32 and
  // two or one bf16): every row's loads in flight at once.  2432 x 2048 5.9 us
  // against 7.6 through the ring (3000 rows: 9.3 and 7.7), 900 x 4096 6.2 against
  // 8.9, 2432 x 1536 fp32 5.2 against 5.5 (3000 rows: 7.9 and 6.5).
  constexpr int FEW = NCH <= 6 ? 4 : sizeof(T) == 4 ? (NCH <= 8 ? 3 : 2) : (NCH <= 8 ? 2 : 1);
  if (rows <= 8LL * FEW * sms) {
    launch_pdl(k_ln_mod1<T, NCH>, (unsigned)((rows + 7) / 8), 256, (size_t)mods, s, x, out, rows, C, shift, scale,
               mod_stride, seg_split, rpb0, rpb1);
    return launched();
  }
  // Blocks per SM as measured: four up to six vectors a lane (8000 x 1152 9.3 us,
  // three 10.1, two 13.0), three up to eight (8000 x 2048 16.9, two 18.5, four
  // 20.2), then the two that are resident (8000 x 3072 23.4, three and four
  // in turn 32.3 and 26.8), for fp32 rows well past the L2 four in turn, in whole
  // rows of warps (20000 x 2048 52.3, shares of one row's difference 54.4, two 56.2).
  const bool past_l2 = NCH > 8 && sizeof(T) == 4 && 2 * rows * row > (180LL << 20);
  const int blocks = NCH <= 6 ? 4 : NCH <= 8 ? 3 : past_l2 ? 4 : 2;
  unsigned grid = (unsigned)std::min((rows + 7) / 8, blocks * sms);
  int per = (int)(rows / grid), rem = (int)(rows % grid);
  if (past_l2) {
    per = (per + (rem > 0) + 7) / 8 * 8;
    rem = 0;
    grid = (unsigned)((rows + per - 1) / per);
  }
  // the ring as deep as that many blocks' shared memory allows
  const long long budget = 224 * 1024 / blocks - 1024 - mods;
  const int depth = budget >= 8 * 3 * row ? 3 : budget >= 8 * 2 * row ? 2 : 1;
  const size_t smem = (size_t)(mods + 8 * depth * row);
  // The kernel attribute belongs to the process, so it is the instance's own
  // largest size, whatever this call needs: threads with rows of other widths
  // set the same value.
  auto go = [&](auto kernel, auto d) -> cudaError_t {
    constexpr int ROW_MAX = NCH * 32 * 16, MODS_MAX = NCH * 32 * VecN<T>::n * 8;
    constexpr int SMEM_MAX = MODS_MAX + 8 * decltype(d)::value * ROW_MAX;
    static_assert(SMEM_MAX <= 227 * 1024, "shared memory of a block");
    const cudaError_t a = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX);
    if (a != cudaSuccess) return a;
    launch_pdl(kernel, dim3(grid), dim3(256), smem, s, x, out, rows, C, shift, scale, mod_stride, seg_split, rpb0,
               rpb1, per, rem);
    return launched();
  };
  return depth == 3   ? go(k_ln_mod<T, NCH, 3>, std::integral_constant<int, 3>())
         : depth == 2 ? go(k_ln_mod<T, NCH, 2>, std::integral_constant<int, 2>())
                      : go(k_ln_mod<T, NCH, 1>, std::integral_constant<int, 1>());
}

template <class T>
static cudaError_t ln_mod_t(const void* x, void* out, long long rows, int C, const float* shift, const float* scale,
                            int mod_stride, int seg_split, int rpb0, int rpb1, cudaStream_t s) {
  const int nch = (C / VecN<T>::n + 31) / 32;
  if (C % 4 != 0 || 2 * C * sizeof(float) > 48 * 1024) return cudaErrorInvalidValue;
  const T* xp = (const T*)x;
  T* op = (T*)out;
#define FF_LN_CASE(n) \
  case n: return ln_mod_launch<T, n>(xp, op, rows, C, shift, scale, mod_stride, seg_split, rpb0, rpb1, s);
  const int nchr = nch <= 6 ? nch : nch <= 8 ? 8 : nch <= 12 ? 12 : nch <= 16 ? 16 : 0;
  switch (nchr) {
    FF_LN_CASE(1) FF_LN_CASE(2) FF_LN_CASE(3) FF_LN_CASE(4) FF_LN_CASE(5) FF_LN_CASE(6)
    FF_LN_CASE(8) FF_LN_CASE(12) FF_LN_CASE(16)
    default:
      return cudaErrorInvalidValue;
  }
#undef FF_LN_CASE
}

cudaError_t launch_ln_mod(DType dt, const void* x, void* out, long long rows, int C, const float* shift,
                          const float* scale, int mod_stride, int seg_split, int rpb0, int rpb1, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  if (((uintptr_t)shift & 15) || ((uintptr_t)scale & 15) || (mod_stride & 3)) return cudaErrorInvalidValue;
  if (dt == F32) return ln_mod_t<float>(x, out, rows, C, shift, scale, mod_stride, seg_split, rpb0, rpb1, s);
  return ln_mod_t<bf16>(x, out, rows, C, shift, scale, mod_stride, seg_split, rpb0, rpb1, s);
}

// Sinusoidal features of every model time: row s = [cos(t_s f_k) | sin(t_s f_k)].
template <class T>
__global__ void k_sinusoid_table(const float* __restrict__ times, int S, T* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int s = blockIdx.x;
  if (s >= S) return;
  const double t = (double)times[s];
  for (int k = threadIdx.x; k < 128; k += blockDim.x) {
    const double f = exp(-log(10000.0) * (double)k / 128.0);
    out[(size_t)s * 256 + k] = from_f<T>((float)cos(t * f));
    out[(size_t)s * 256 + 128 + k] = from_f<T>((float)sin(t * f));
  }
}

cudaError_t launch_sinusoid_table(DType dt, const float* times, int S, void* out, cudaStream_t s) {
  if (S <= 0) return cudaSuccess;
  if (dt == F32) launch_pdl(k_sinusoid_table<float>, S, 128, 0, s, times, S, (float*)out);
  else launch_pdl(k_sinusoid_table<bf16>, S, 128, 0, s, times, S, (bf16*)out);
  return launched();
}

// SiLU(c) of every (step, sample): c = temb[step] (+ y_emb[label]).
template <class T>
__global__ void k_cond_table(const float* __restrict__ temb, const T* __restrict__ y_emb, const int* __restrict__ labels,
                             int S, int B, int C, const int* __restrict__ need_row, T* __restrict__ all,
                             T* __restrict__ need) {
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x;  // s * B + b
  const int s = row / B, b = row % B;
  if (s >= S) return;
  const int nr = need_row ? need_row[s] : -1;
  for (int k = threadIdx.x; k < C; k += blockDim.x) {
    float v = temb[(size_t)s * C + k];
    if (y_emb) v += to_f(y_emb[(size_t)labels[b] * C + k]);
    const T o = from_f<T>(silu(v));
    all[(size_t)row * C + k] = o;
    if (nr >= 0) need[((size_t)nr * B + b) * C + k] = o;
  }
}

cudaError_t launch_cond_table(DType dt, const float* temb, const void* y_emb, const int* labels, int S, int B, int C,
                              const int* need_row, void* all, void* need, cudaStream_t s) {
  if (S <= 0) return cudaSuccess;
  if (dt == F32)
    launch_pdl(k_cond_table<float>, S * B, 256, 0, s, temb, (const float*)y_emb, labels, S, B, C, need_row, (float*)all,
                                              (float*)need);
  else
    launch_pdl(k_cond_table<bf16>, S * B, 256, 0, s, temb, (const bf16*)y_emb, labels, S, B, C, need_row, (bf16*)all,
                                             (bf16*)need);
  return launched();
}

// Patch features of the model batch (latent sample b % B_lat): row
// b*N_img + token, feature (channel, frame offset, row offset, col offset).
template <class T>
__global__ void k_patchify(const float* __restrict__ lat, int B_lat, int B_model, int Cin, int F, int H, int W, int p,
                           int pt, T* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int Ff = F > 0 ? F : 1, ptt = F > 0 ? pt : 1;
  const int gf = Ff / ptt, gh = H / p, gw = W / p;
  const int P = ptt * p * p, feat = Cin * P;
  const long long total = (long long)B_model * gf * gh * gw * feat;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int f = (int)(i % feat);
    const long long row = i / feat;
    const int tok = (int)(row % ((long long)gf * gh * gw));
    const int b = (int)(row / ((long long)gf * gh * gw));
    const int c = f / P, o = f % P;
    const int ot = o / (p * p), oh = (o / p) % p, ow = o % p;
    const int tw = tok % gw, th = (tok / gw) % gh, tf = tok / (gw * gh);
    const int zf = tf * ptt + ot, zh = th * p + oh, zw = tw * p + ow;
    const long long src = ((((long long)(b % B_lat) * Cin + c) * Ff + zf) * H + zh) * W + zw;
    out[i] = from_f<T>(lat[src]);
  }
}

cudaError_t launch_patchify(DType dt, const float* latent, int B_lat, int B_model, int Cin, int F, int H, int W,
                            int p, int pt, void* out, cudaStream_t s) {
  const int grid = num_sms() * 4;
  if (dt == F32) launch_pdl(k_patchify<float>, grid, 256, 0, s, latent, B_lat, B_model, Cin, F, H, W, p, pt, (float*)out);
  else launch_pdl(k_patchify<bf16>, grid, 256, 0, s, latent, B_lat, B_model, Cin, F, H, W, p, pt, (bf16*)out);
  return launched();
}

template <class T>
__global__ void k_convert(const float* __restrict__ in, T* __restrict__ out, long long n) {
  pdl_trigger();
  pdl_wait();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = from_f<T>(in[i]);
}

cudaError_t launch_convert(DType dt, const float* in, void* out, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int grid = num_sms() * 4;
  if (dt == F32) launch_pdl(k_convert<float>, grid, 256, 0, s, in, (float*)out, n);
  else launch_pdl(k_convert<bf16>, grid, 256, 0, s, in, (bf16*)out, n);
  return launched();
}

// Guidance + sampler update of the latent: g = out_u + s (out_c - out_u)
// (or out), x <- c1 x + c2 g, reading the model output through the
// unpatchify index map.  Euler: c1 = 1, c2 = sigma_{i+1} - sigma_i.  DDIM:
// c1 = sqrt(a_prev / a_t), c2 = sqrt(1 - a_prev) - sqrt(a_prev (1 - a_t) / a_t).
__global__ void k_sampler(const float* __restrict__ mo, float* __restrict__ lat, int B_lat, int cfg, float cfg_scale,
                          int Cin, int Cout, int F, int H, int W, int p, int pt, float c1, float c2) {
  pdl_trigger();
  pdl_wait();
  const int Ff = F > 0 ? F : 1, ptt = F > 0 ? pt : 1;
  const int gh = H / p, gw = W / p, gf = Ff / ptt;
  const int P = ptt * p * p;
  const long long ntok = (long long)gf * gh * gw;
  const long long total = (long long)B_lat * Cin * Ff * H * W;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int zw = (int)(i % W);
    const int zh = (int)((i / W) % H);
    const int zf = (int)((i / ((long long)W * H)) % Ff);
    const int c = (int)((i / ((long long)W * H * Ff)) % Cin);
    const int b = (int)(i / ((long long)W * H * Ff * Cin));
    const long long tok = ((long long)(zf / ptt) * gh + zh / p) * gw + zw / p;
    const int f = c * P + ((zf % ptt) * p + zh % p) * p + zw % p;
    const long long fo = (long long)Cout * P;
    float g = mo[((long long)b * ntok + tok) * fo + f];
    if (cfg) {
      const float gu = mo[((long long)(b + B_lat) * ntok + tok) * fo + f];
      g = gu + cfg_scale * (g - gu);
    }
    lat[i] = c1 * lat[i] + c2 * g;
  }
}

cudaError_t launch_sampler(const float* model_out, float* latent, int B_lat, int cfg, float cfg_scale, int Cin,
                           int Cout, int F, int H, int W, int p, int pt, float c1, float c2, cudaStream_t s) {
  launch_pdl(k_sampler, num_sms() * 2, 256, 0, s, model_out, latent, B_lat, cfg, cfg_scale, Cin, Cout, F, H, W, p, pt, c1, c2);
  return launched();
}

// Seeded N(0,1) latent: SplitMix64 word k = mix(seed + (k+1) * golden),
// u = ((w >> 11) + 0.5) 2^-53, Box-Muller on word pairs (2m, 2m+1).
__device__ __forceinline__ unsigned long long splitmix_word(unsigned long long seed, unsigned long long k) {
  unsigned long long z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_noise(unsigned long long seed, float* __restrict__ out, long long n) {
  pdl_trigger();
  pdl_wait();
  const long long pairs = (n + 1) / 2;
  for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < pairs; m += (long long)gridDim.x * blockDim.x) {
    const double u1 = ((double)(splitmix_word(seed, 2 * m) >> 11) + 0.5) * 0x1.0p-53;
    const double u2 = ((double)(splitmix_word(seed, 2 * m + 1) >> 11) + 0.5) * 0x1.0p-53;
    const double r = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincos(2.0 * 3.141592653589793 * u2, &sn, &cs);
    out[2 * m] = (float)(r * cs);
    if (2 * m + 1 < n) out[2 * m + 1] = (float)(r * sn);
  }
}

cudaError_t launch_noise(unsigned long long seed, float* out, long long n, cudaStream_t s) {
  launch_pdl(k_noise, num_sms() * 2, 256, 0, s, seed, out, n);
  return launched();
}

// Fixed 2-D sin-cos position embedding replicated over B samples:
// channels [0, C/2) encode the patch row, [C/2, C) the column, each half
// [sin(pos w_k) | cos(pos w_k)], w_k = 10000^(-k/(C/4)).
template <class T>
__global__ void k_pos2d(T* __restrict__ out, int B, int gh, int gw, int C) {
  pdl_trigger();
  pdl_wait();
  const int q = C / 4;
  const long long total = (long long)B * gh * gw * C;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const int tok = (int)((i / C) % ((long long)gh * gw));
    const int half = c / (C / 2), cc = c % (C / 2);
    const double pos = half == 0 ? (double)(tok / gw) : (double)(tok % gw);
    const int k = cc % q;
    const double a = pos * pow(10000.0, -(double)k / (double)q);
    out[i] = from_f<T>((float)(cc < q ? sin(a) : cos(a)));
  }
}

cudaError_t launch_pos2d(DType dt, void* out, int B, int gh, int gw, int C, cudaStream_t s) {
  const int grid = num_sms() * 4;
  if (dt == F32) launch_pdl(k_pos2d<float>, grid, 256, 0, s, (float*)out, B, gh, gw, C);
  else launch_pdl(k_pos2d<bf16>, grid, 256, 0, s, (bf16*)out, B, gh, gw, C);
  return launched();
}

}  // namespace ff
