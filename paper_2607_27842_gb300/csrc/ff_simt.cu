// CUDA-core (no tensor core, no TF32) dense layer and attention: the fp32
// mode of the exact block (Eq. 1) and the narrow final projection.
#include "ff_common.cuh"

#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

namespace cg = cooperative_groups;

namespace ff {

static int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 148;
  }();
  return n;
}

// ---------------------------------------------------------------------------
// out = epilogue(A[M,K] W[N,K]^T) in fp32 on CUDA cores, FFMA2.
//
// Both operands are K-contiguous, so their tiles are copied to shared memory
// as they are (cp.async, ST stages of BK columns, rows padded by 16 bytes:
// eight consecutive rows' 16-byte vectors fall into distinct banks), and a
// thread's TM x TN outputs accumulate (even k, odd k) pairs with fma.rn.f32x2:
// the 16-byte fragment loads need no transposition and no duplicated operand,
// and each output is two interleaved partial sums.  WK groups of warps share a
// tile, each taking its own 16-byte columns of every stage; the groups'
// accumulators are added through shared memory in a fixed order.  Several
// CTAs of a cluster may share a tile's K range as well (small problems, where
// the tiles alone leave the chip idle and the serial loads are the time);
// they add through distributed shared memory, rank by rank, so the result
// does not depend on timing.
//
// Bound (times: launches back to back in a CUDA graph): FFMA2 issue beside the
// fragment loads.  A register-only FFMA2 loop
// runs at 114 of the 128 FMA per SM and clock (scalar FFMA 76), with this
// kernel's 16 16-byte loads per 256 FMA 91; the 128 tile reaches 83.  What
// counted: deep stages (BK 32 -> 128 on 64 tiles: 512 x 1152 x 1152 42 -> 36
// us; every barrier leaves all warps waiting on their first loads) and copies
// whose addresses cost one addition (1024 x 4608 x 4608 985 -> 870 us, 50
// TFLOP/s).  Against 4-byte staging loads, one buffer and 64 x 128 tiles
// everywhere: 1024 x 4608 x 4608 1775 -> 870 us, 512 x 1152 x 4608 562 -> 131,
// 64 x 128 x 512 60 -> 4.3, 2 x 6912 x 1152 122 -> 15.
// ---------------------------------------------------------------------------
// BM x BN tile, warp tile 8 TM x 4 TN (lanes 8 x 4), WK groups of warps
template <int BM_, int BN_, int TM_, int TN_, int WK_, int BK_, int ST_> struct F32Cfg {
  static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_, WK = WK_, BK = BK_, ST = ST_;
  static constexpr int WM = 8 * TM, WN = 4 * TN;
  static constexpr int WARPS_M = BM / WM, WARPS_N = BN / WN;
  static constexpr int THREADS = 32 * WARPS_M * WARPS_N * WK;
  static constexpr int LD = BK + 4;                    // row stride of a staged operand (floats)
  static constexpr int STAGE = (BM + BN) * LD;         // floats of a stage
  static constexpr int LDC = BN + 4;                   // row stride of an output tile
  static constexpr int RED = WK * BM * LDC;            // the groups' output tiles, over the stages
  static constexpr size_t SMEM = sizeof(float) * (size_t)(ST * STAGE > RED ? ST * STAGE : RED);
  static_assert((BK / 4) % WK == 0, "every group takes whole 16-byte columns");
};

// TAIL: the last stage is not a whole one and only its columns of K are copied and
// multiplied (64 and 128 tiles; an instance of its own, because the loop over
// columns costs the whole stages 1%): 4096 x 1152 x 16 22 -> 14 us.
template <class C, bool VEC, bool TAIL>
__global__ void __launch_bounds__(C::THREADS) k_gemm_f32(int M, int N, int K, const float* __restrict__ A, int lda,
                                                         const float* __restrict__ W, int ldw,
                                                         const __grid_constant__ EpiArgs e) {
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wk = warp / (C::WARPS_M * C::WARPS_N), wt = warp % (C::WARPS_M * C::WARPS_N);
  const int lm = lane >> 2, ln = lane & 3;
  const int ra = (wt / C::WARPS_N) * C::WM + lm;       // the thread's A rows: ra + 8 i
  const int rb = (wt % C::WARPS_N) * C::WN + ln;       // its W rows: rb + 4 j
  // one-dimensional grid over the tiles, row blocks fastest: the CTAs running
  // together share W tiles (rows are few, W is the larger operand)
  const int num_m = (M + C::BM - 1) / C::BM;
  const int m0 = (int)(blockIdx.x % num_m) * C::BM, n0 = (int)(blockIdx.x / num_m) * C::BN;
  const int split = gridDim.y, rank = blockIdx.y;
  const int nkt = (K + C::BK - 1) / C::BK;
  const int kt0 = (int)((long long)nkt * rank / split), kt1 = (int)((long long)nkt * (rank + 1) / split);

  // Copies: the thread's column of a stage and its rows (r0 + RPP q of A, then
  // of W) are fixed, so a copy costs one address addition; rows past the end
  // and columns past K are zeros that read nothing.
  constexpr int EL = VEC ? 4 : 1, CPR = C::BK / EL, RPP = C::THREADS / CPR;
  constexpr int PA = C::BM / RPP, PW = C::BN / RPP;
  static_assert(C::BM % RPP == 0 && C::BN % RPP == 0 && PA + PW <= 64, "whole passes");
  using Mask = typename std::conditional<PA + PW <= 32, unsigned, unsigned long long>::type;
  // row offsets from the tile's first row (32 bits on the 16-byte path, whose
  // row strides the dispatch bounds)
  using Off = typename std::conditional<VEC, unsigned, size_t>::type;
  const int kc = (tid % CPR) * EL, r0 = tid / CPR;
  const Off oa = (Off)r0 * (Off)lda + kc, ow = (Off)r0 * (Off)ldw + kc;
  Mask live = 0;                                   // bit q: row r0 + RPP q of A, bit PA + q: of W
#pragma unroll
  for (int q = 0; q < PA; ++q) live |= (Mask)(m0 + r0 + RPP * q < M ? 1 : 0) << q;
#pragma unroll
  for (int q = 0; q < PW; ++q) live |= (Mask)(n0 + r0 + RPP * q < N ? 1 : 0) << (PA + q);
  const int K4 = (K + 3) & ~3;
  const float* const At = A + (size_t)m0 * lda;
  const float* const Wt = W + (size_t)n0 * ldw;
  auto load = [&](int kt, int slot) {
    float* s = sm + slot * C::STAGE + r0 * C::LD + kc;
    const int k0 = kt * C::BK;
    if (TAIL && k0 + kc >= K4) return;                 // a column that is never read
    const Mask mask = k0 + kc < K ? live : (Mask)0;
#pragma unroll
    for (int q = 0; q < PA + PW; ++q) {
      const bool in = (mask >> q) & 1;
      const float* src = q < PA ? At + k0 + (oa + (Off)(RPP * q) * (Off)lda)
                                : Wt + k0 + (ow + (Off)(RPP * (q - PA)) * (Off)ldw);
      src = in ? src : A;
      float* d = s + (q < PA ? RPP * q : C::BM + RPP * (q - PA)) * C::LD;
      if (VEC) cp_async16(d, src, in ? 16 : 0); else cp_async4(d, src, in ? 4 : 0);
    }
  };

  f32x2 acc[C::TM][C::TN];
#pragma unroll
  for (int i = 0; i < C::TM; ++i)
#pragma unroll
    for (int j = 0; j < C::TN; ++j) acc[i][j] = 0ull;

  pdl_wait();
#pragma unroll
  for (int p = 0; p < C::ST - 1; ++p) {
    if (kt0 + p < kt1) load(kt0 + p, p);
    cp_commit();
  }
  // 16-byte column kk / 4 of stage `it`
  auto column = [&](int it, int kk) {
    const float* sa = sm + (it % C::ST) * C::STAGE + ra * C::LD + kk;
    const float* sb = sm + (it % C::ST) * C::STAGE + (C::BM + rb) * C::LD + kk;
    ulonglong2 a[C::TM], b[C::TN];
#pragma unroll
    for (int i = 0; i < C::TM; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(sa + 8 * i * C::LD);
#pragma unroll
    for (int j = 0; j < C::TN; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(sb + 4 * j * C::LD);
#pragma unroll
    for (int i = 0; i < C::TM; ++i)
#pragma unroll
      for (int j = 0; j < C::TN; ++j) acc[i][j] = ffma2(a[i].x, b[j].x, acc[i][j]);
#pragma unroll
    for (int i = 0; i < C::TM; ++i)
#pragma unroll
      for (int j = 0; j < C::TN; ++j) acc[i][j] = ffma2(a[i].y, b[j].y, acc[i][j]);
  };
  const int full = TAIL ? min(kt1, K4 / C::BK) : kt1;  // whole stages [kt0, full)
  for (int kt = kt0; kt < full; ++kt) {
    cp_wait<C::ST - 2>();
    __syncthreads();
    const int it = kt - kt0;
    if (kt + C::ST - 1 < kt1) load(kt + C::ST - 1, (it + C::ST - 1) % C::ST);
    cp_commit();
#pragma unroll
    for (int c = 0; c < C::BK / 4 / C::WK; ++c) column(it, (c * C::WK + wk) * 4);
  }
  if (TAIL && full < kt1) {
    cp_wait<0>();
    __syncthreads();
#pragma unroll 1
    for (int kk = wk * 4; kk < K4 - full * C::BK; kk += C::WK * 4) column(full - kt0, kk);
  }
  cp_wait<0>();
  __syncthreads();                                     // the stages are free: output tiles over them
  {
    float* t = sm + wk * C::BM * C::LDC;
#pragma unroll
    for (int i = 0; i < C::TM; ++i)
#pragma unroll
      for (int j = 0; j < C::TN; ++j)
        t[(ra + 8 * i) * C::LDC + rb + 4 * j] = lo_f(acc[i][j]) + hi_f(acc[i][j]);
  }
  __syncthreads();
  // four consecutive columns of one row per thread: the groups' partials in
  // order, then (split) the ranks' tiles in order, then the epilogue
  constexpr int CPT = C::BN / 4;
  auto group_sum = [&](int r, int c4) {
    float4 v = *reinterpret_cast<const float4*>(sm + r * C::LDC + 4 * c4);
#pragma unroll
    for (int g = 1; g < C::WK; ++g) {
      const float4 u = *reinterpret_cast<const float4*>(sm + (g * C::BM + r) * C::LDC + 4 * c4);
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    return v;
  };
  auto finish = [&](int r, int c4, const float4& v) {
    const int m = m0 + r, n = n0 + 4 * c4;
    if (m >= M || n >= N) return;
    float x[4] = {v.x, v.y, v.z, v.w};
    epi_chunk<float, 4, 0>(e, m, n, N, x);
  };
  constexpr int PIECES = C::BM * CPT / C::THREADS;     // of a thread (0: some threads have one)
  if (split == 1 && PIECES >= 4 && ((e.resid && (PIECES > 4 || e.gate)) || e.hist_out)) {
    // Residual and history base: U pieces at a time, all their loads before their
    // stores.  (A load may not pass a store that could alias it, so piece by
    // piece each one waits for memory in turn: 1024 x 4608 x 1152 with gate,
    // residual and history 267 us, four at a time 240, eight 244.  A 64 tile's
    // four pieces with a residual only are 2% faster one by one.)
    constexpr int U = PIECES >= 4 ? 4 : 1;
    static_assert(PIECES < 4 || PIECES % U == 0, "whole batches");
#pragma unroll 1
    for (int c0 = tid; c0 < C::BM * CPT; c0 += U * C::THREADS) {
      float x[U][4];
      float4 res[U], base[U];
      bool in[U];
      int mm[U], nn[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int c = c0 + u * C::THREADS;
        mm[u] = m0 + c / CPT;
        nn[u] = n0 + 4 * (c % CPT);
        in[u] = mm[u] < M && nn[u] < N;
        const float4 v = group_sum(c / CPT, c % CPT);
        x[u][0] = v.x; x[u][1] = v.y; x[u][2] = v.z; x[u][3] = v.w;
        if (in[u] && e.resid)
          res[u] = *reinterpret_cast<const float4*>((const float*)e.resid + (size_t)mm[u] * e.ld_resid + nn[u]);
        if (in[u] && e.hist_out)
          base[u] = *reinterpret_cast<const float4*>((const float*)e.hist_base + (size_t)mm[u] * e.ldo + nn[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (in[u]) epi_math<float, 4, 0>(e, mm[u], nn[u], N, x[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (!in[u]) continue;
        float4 o = make_float4(x[u][0], x[u][1], x[u][2], x[u][3]);
        if (e.resid) { o.x += res[u].x; o.y += res[u].y; o.z += res[u].z; o.w += res[u].w; }
        const bool second = nn[u] >= e.split_col;
        float* const out = (float*)(second ? e.out2 : e.out) + (size_t)mm[u] * (second ? e.ldo2 : e.ldo) +
                           (second ? nn[u] - e.split_col : nn[u]);
        *reinterpret_cast<float4*>(out) = o;
        if (e.hist_out)
          *reinterpret_cast<float4*>((float*)e.hist_out + (size_t)mm[u] * e.ldo + nn[u]) =
              make_float4(o.x - base[u].x, o.y - base[u].y, o.z - base[u].z, o.w - base[u].w);
      }
    }
    return;
  }
  if (split == 1) {
    for (int c = tid; c < C::BM * CPT; c += C::THREADS) finish(c / CPT, c % CPT, group_sum(c / CPT, c % CPT));
    return;
  }
  for (int c = tid; C::WK > 1 && c < C::BM * CPT; c += C::THREADS)
    *reinterpret_cast<float4*>(sm + (c / CPT) * C::LDC + 4 * (c % CPT)) = group_sum(c / CPT, c % CPT);
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  const int rows = C::BM / split;                      // this rank finishes rows [rank * rows, + rows)
  for (int c = tid; c < rows * CPT; c += C::THREADS) {
    const int r = rank * rows + c / CPT, c4 = c % CPT;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = 0; q < split; ++q) {
      const float4 u = *reinterpret_cast<const float4*>(cluster.map_shared_rank(sm, q) + r * C::LDC + 4 * c4);
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    finish(r, c4, v);
  }
  cluster.sync();                                      // peers may still be reading this CTA's tile
}

template <class C, bool VEC, bool TAIL>
static cudaError_t gemm_f32_tail(int M, int N, int K, const float* A, int lda, const float* W, int ldw,
                                 const EpiArgs& e, int split, cudaStream_t s) {
  const cudaError_t attr =
      cudaFuncSetAttribute(k_gemm_f32<C, VEC, TAIL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
  if (attr != cudaSuccess) return attr;
  const long long tiles = (long long)((N + C::BN - 1) / C::BN) * ((M + C::BM - 1) / C::BM);
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tiles, split);
  cfg.blockDim = dim3(C::THREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = split;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = split > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, k_gemm_f32<C, VEC, TAIL>, M, N, K, A, lda, W, ldw, e);
  return launched();
}

template <class C, bool VEC>
static cudaError_t gemm_f32_launch(int M, int N, int K, const float* A, int lda, const float* W, int ldw,
                                   const EpiArgs& e, int split, cudaStream_t s) {
  if constexpr (C::BM >= 64)
    if (K % C::BK != 0) return gemm_f32_tail<C, VEC, true>(M, N, K, A, lda, W, ldw, e, split, s);
  return gemm_f32_tail<C, VEC, false>(M, N, K, A, lda, W, ldw, e, split, s);
}

// Tile choice by the estimated time of the launch's waves (one 128 or 64 tile
// per SM at a time; a 64 tile's FMA count at 0.9 of the 128 tile's rate, a 32
// tile's at 0.6), then a smaller tile (never a larger one: smaller tiles have
// more groups and so more partial sums, and short reductions should not lose
// accuracy) where that is faster with what a tile takes beside its columns
// of K counted in: 5.2, 2.7 and 0.53 us for the 128, 64 and 32 tiles, the time of
// 56, 90 and 58 columns (657 x 1264 x 256 19.9 us in 64 tiles, 18.3 in 32).
// Few rows or few tiles are latency- or weight-bound: 16 x 32
// tiles up to 16 rows (W read once per 16 rows: 2 x 6912 x 1152 22.7 -> 15.2
// us) and wherever 32 x 32 tiles would leave half the SMs idle (64 x 512 x 128
// 3.46 -> 2.86 us); those also split K over a cluster while every CTA keeps a
// K range of at least 128 (a split costs about 1 us: 64 x 128 x 128 in two
// halves 3.46 -> 3.98 us).
template <bool VEC>
static cudaError_t gemm_f32_t(int M, int N, int K, const float* A, int lda, const float* W, int ldw, const EpiArgs& e,
                              cudaStream_t s) {
  using C128 = F32Cfg<128, 128, 8, 8, 1, 64, 3>;
  using C64 = F32Cfg<64, 64, 8, 8, 4, 128, 2>;
  using C32 = F32Cfg<32, 32, 4, 8, 8, 64, 4>;
  using C16 = F32Cfg<16, 32, 2, 8, 8, 128, 3>;
  const long long sms = sm_count();
  const long long t128 = (long long)((M + 127) / 128) * ((N + 127) / 128);
  const long long t64 = (long long)((M + 63) / 64) * ((N + 63) / 64);
  const long long t32 = (long long)((M + 31) / 32) * ((N + 31) / 32);
  if (M > 16 && t32 * 2 > sms) {
    const double w128 = (double)((t128 + sms - 1) / sms) * 128 * 128, w64 = (double)((t64 + sms - 1) / sms) * 64 * 64;
    const double w32 = std::max(1.0, (double)t32 / sms) * 32 * 32;
    const double c128 = w128 * (K + 56), c64 = w64 * 1.165 * (K + 90), c32 = w32 * 1.7 * ((K + C32::BK - 1) / C32::BK * C32::BK + 58);
    int bm = w128 <= w64 * 1.1 && w128 <= w32 * 1.6 ? 128 : w64 * 1.1 <= w32 * 1.6 ? 64 : 32;
    if (bm == 128 && std::min(c64, c32) < c128) bm = c64 <= c32 ? 64 : 32;
    if (bm == 64 && c32 < c64) bm = 32;
    if (bm == 128) return gemm_f32_launch<C128, VEC>(M, N, K, A, lda, W, ldw, e, 1, s);
    if (bm == 64) return gemm_f32_launch<C64, VEC>(M, N, K, A, lda, W, ldw, e, 1, s);
    return gemm_f32_launch<C32, VEC>(M, N, K, A, lda, W, ldw, e, 1, s);
  }
  const long long t16 = (long long)((M + 15) / 16) * ((N + 31) / 32);
  int split = 1;
  while (split < 8 && t16 * split * 2 <= 2 * sms && K / (split * 2) >= 128) split *= 2;
  return gemm_f32_launch<C16, VEC>(M, N, K, A, lda, W, ldw, e, split, s);
}

cudaError_t gemm_f32(int M, int N, int K, const float* A, int lda, const float* W, int ldw, const EpiArgs& e,
                     cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const bool vec = K % 4 == 0 && lda % 4 == 0 && ldw % 4 == 0 && !((uintptr_t)A & 15) && !((uintptr_t)W & 15) &&
                   lda <= (1 << 24) && ldw <= (1 << 24);
  return vec ? gemm_f32_t<true>(M, N, K, A, lda, W, ldw, e, s) : gemm_f32_t<false>(M, N, K, A, lda, W, ldw, e, s);
}

// ---------------------------------------------------------------------------
// Attention on CUDA cores in fp32 (fp32 mode, and bf16 head widths without a
// tensor-core kernel): one CTA per (sample, head, 32 queries), 64 keys at a
// time through shared memory, 128 threads as 8 query groups x 16 lanes.
// Thread (tq, tk) owns queries tq + 8 i (i < 4): their scores against keys
// tk + 16 j, then, after the online softmax over the group's 16 lanes, output
// columns 2 tk + 32 g of the same queries (DG column pairs per lane).  P goes
// through shared memory but stays within its group of lanes.  The next tile's
// keys are copied while the softmax and P V run, its values while the next
// scores are computed (cp.async into the one buffer each).
//
// Bound: shared-memory fragment loads (8 per 64 FMA in q k^T, 16 per 96 in
// P V at head width 72).  Against one warp per query reading keys row by row
// from global memory (uncoalesced, no reuse): 2 x 256 tokens, 16 heads x 72
// 575 -> 42 us; 1024 tokens, 16 heads x 64 4047 -> 169 us (25 TFLOP/s); 64
// tokens, 4 heads x 32 17.4 -> 5.1 us.
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long tok_row(const AttnArgs& a, int b, int n) {
  return n < a.Nt ? (long long)b * a.Nt + n : (long long)a.B * a.Nt + (long long)b * a.Ni + (n - a.Nt);
}

constexpr int FA_BQ = 32, FA_BK = 64, FA_THREADS = 128, FA_LDP = 80;  // P rows 80 apart: two groups' rows in distinct banks
static size_t fa_smem(int hd) { return sizeof(float) * ((size_t)(FA_BQ + 2 * FA_BK) * (hd + 4) + FA_BQ * FA_LDP); }

template <class T, int DG, bool VEC>
__global__ void __launch_bounds__(FA_THREADS) k_attn_f32(AttnArgs a, float scale) {
  extern __shared__ __align__(16) float sm[];
  pdl_trigger();
  const int N = a.Nt + a.Ni, hd = a.hd, ld = hd + 4;   // (hd + 4 = 4 x odd: eight rows' vectors in distinct banks)
  float* const sQ = sm;
  float* const sK = sQ + FA_BQ * ld;
  float* const sV = sK + FA_BK * ld;
  float* const sP = sV + FA_BK * ld;
  const int h = blockIdx.y, b = blockIdx.z, q0 = blockIdx.x * FA_BQ;
  const int tid = threadIdx.x, tk = tid & 15, tq = tid >> 4;
  // rows n0 .. n0 + rows - 1 of the sample's head into s (zeros past N)
  auto load = [&](const void* base, float* s, int n0, int rows) {
    const T* g = reinterpret_cast<const T*>(base) + (size_t)h * hd;
    constexpr int E = VEC ? VecN<T>::n : 1;
    const int cpr = hd / E;
    for (int c = tid; c < rows * cpr; c += FA_THREADS) {
      const int r = c / cpr, e = (c % cpr) * E;
      const bool in = n0 + r < N;
      const T* src = in ? g + tok_row(a, b, n0 + r) * a.ld_qkv + e : g;
      float* d = s + r * ld + e;
      if constexpr (VEC && sizeof(T) == 4) {
        cp_async16(d, src, in ? 16 : 0);
      } else if constexpr (VEC) {
        float v[VecN<T>::n];
        ld16(src, v);
#pragma unroll
        for (int z = 0; z < VecN<T>::n; ++z) d[z] = in ? v[z] : 0.f;
      } else {
        *d = in ? to_f(*src) : 0.f;
      }
    }
  };
  const int nt = (N + FA_BK - 1) / FA_BK;
  pdl_wait();
  load(a.q, sQ, q0, FA_BQ);
  load(a.k, sK, 0, FA_BK);
  cp_commit();
  load(a.v, sV, 0, FA_BK);
  cp_commit();

  float m[4], l[4], o[4][2 * DG];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 2 * DG; ++c) o[i][c] = 0.f;
  }
  const float* const qp = sQ + tq * ld;
  const float* const kp = sK + tk * ld;
  float* const pp = sP + tq * FA_LDP;
  for (int t = 0; t < nt; ++t) {
    cp_wait<1>();                                      // this tile's keys (its values may be in flight)
    __syncthreads();
    f32x2 s2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[i][j] = 0ull;
#pragma unroll 2
    for (int e = 0; e < hd; e += 4) {
      ulonglong2 qv[4], kv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) qv[i] = *reinterpret_cast<const ulonglong2*>(qp + 8 * i * ld + e);
#pragma unroll
      for (int j = 0; j < 4; ++j) kv[j] = *reinterpret_cast<const ulonglong2*>(kp + 16 * j * ld + e);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s2[i][j] = ffma2(qv[i].x, kv[j].x, s2[i][j]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s2[i][j] = ffma2(qv[i].y, kv[j].y, s2[i][j]);
    }
    __syncthreads();                                   // the key buffer is free
    if (t + 1 < nt) load(a.k, sK, (t + 1) * FA_BK, FA_BK);
    cp_commit();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float s[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float dot = lo_f(s2[i][j]) + hi_f(s2[i][j]);
        s[j] = t * FA_BK + tk + 16 * j < N ? dot * scale : -INFINITY;
      }
      float cm = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) cm = fmaxf(cm, __shfl_xor_sync(0xffffffffu, cm, w));
      const float mn = fmaxf(m[i], cm);
      const float alpha = expf(m[i] - mn);
      float ps = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float p = t * FA_BK + tk + 16 * j < N ? expf(s[j] - mn) : 0.f;
        ps += p;
        pp[8 * i * FA_LDP + tk + 16 * j] = p;
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, w);
      l[i] = l[i] * alpha + ps;
      m[i] = mn;
#pragma unroll
      for (int c = 0; c < 2 * DG; ++c) o[i][c] *= alpha;
    }
    cp_wait<1>();                                      // this tile's values
    __syncthreads();
#pragma unroll 2
    for (int k = 0; k < FA_BK; k += 4) {
      float4 p4[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) p4[i] = *reinterpret_cast<const float4*>(pp + 8 * i * FA_LDP + k);
#pragma unroll
      for (int z = 0; z < 4; ++z) {
#pragma unroll
        for (int g = 0; g < DG; ++g) {
          const int c = 2 * tk + 32 * g;
          const float2 v = c < hd ? *reinterpret_cast<const float2*>(sV + (k + z) * ld + c) : make_float2(0.f, 0.f);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float p = z == 0 ? p4[i].x : z == 1 ? p4[i].y : z == 2 ? p4[i].z : p4[i].w;
            o[i][2 * g] = fmaf(p, v.x, o[i][2 * g]);
            o[i][2 * g + 1] = fmaf(p, v.y, o[i][2 * g + 1]);
          }
        }
      }
    }
    __syncthreads();                                   // the value buffer is free
    if (t + 1 < nt) load(a.v, sV, (t + 1) * FA_BK, FA_BK);
    cp_commit();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = q0 + tq + 8 * i;
    if (n >= N) continue;
    const float inv = 1.0f / l[i];
    T* out = reinterpret_cast<T*>(a.out) + tok_row(a, b, n) * a.ld_out + (size_t)h * hd;
#pragma unroll
    for (int g = 0; g < DG; ++g) {
      const int c = 2 * tk + 32 * g;
      if (c < hd) {
        out[c] = from_f<T>(o[i][2 * g] * inv);
        out[c + 1] = from_f<T>(o[i][2 * g + 1] * inv);
      }
    }
  }
}

template <class T, int DG, bool VEC>
static cudaError_t attn_f32_launch(const AttnArgs& a, cudaStream_t s) {
  const size_t smem = fa_smem(a.hd);
  const cudaError_t attr = cudaFuncSetAttribute(k_attn_f32<T, DG, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)fa_smem(32 * DG));
  if (attr != cudaSuccess) return attr;
  launch_pdl(k_attn_f32<T, DG, VEC>, dim3((a.Nt + a.Ni + FA_BQ - 1) / FA_BQ, a.H, a.B), dim3(FA_THREADS), smem, s, a,
             1.0f / sqrtf((float)a.hd));
  return launched();
}

template <class T>
static cudaError_t attn_f32_t(const AttnArgs& a, cudaStream_t s) {
  // 16-byte copies need aligned head rows; hd is a multiple of 8
  const bool vec = a.ld_qkv % VecN<T>::n == 0 && !(((uintptr_t)a.q | (uintptr_t)a.k | (uintptr_t)a.v) & 15);
#define FF_FA(dg) case dg: return vec ? attn_f32_launch<T, dg, true>(a, s) : attn_f32_launch<T, dg, false>(a, s);
  switch ((a.hd + 31) / 32) {
    FF_FA(1) FF_FA(2) FF_FA(3) FF_FA(4)
    default: return cudaErrorInvalidValue;
  }
#undef FF_FA
}

cudaError_t attention_simt(DType dt, const AttnArgs& a, cudaStream_t s) {
  return dt == F32 ? attn_f32_t<float>(a, s) : attn_f32_t<bf16>(a, s);
}

}  // namespace ff
