// bf16 dense layers of the exact block (Eq. 1) on the 5th-generation tensor
// cores: out = epilogue(A[M,K] W[N,K]^T).
//
// Persistent kernel, one CTA per SM, 10 warps:
//   warp 0      TMA producer: A and W tiles (128 and BN rows x 64 k, 128-byte
//               swizzle) into a STAGES-deep shared-memory ring;
//   warp 1      TMEM allocator and MMA issuer (the whole warp runs the loop,
//               one elected lane issues):
//               tcgen05.mma.cta_group::1.kind::f16 (M = 128, N = BN, K = 16),
//               fp32 accumulators in TMEM, tcgen05.commit frees ring slots;
//   warps 2..9  epilogue: tcgen05.ld of the accumulator (each warp one
//               32-lane quarter and one column half), the fused bias / RoPE /
//               GELU / gate / residual / history epilogue, stores through
//               swizzled shared-memory blocks and TMA (16-byte stores where
//               the output does not allow it); with one tile per CTA the
//               residual / history-base blocks arrive by TMA as well and are
//               replaced in place by the output (epi_single).
// Times in the comments are of launches back to back in a CUDA graph.
//
// Two TMEM accumulators (2 * BN columns) let the epilogue of tile i overlap
// the main loop of tile i + 1.  Every mbarrier wait is bounded: on timeout
// the CTA raises a watchdog flag, stops issuing work and releases its TMEM.
//
// With both operands in shared memory a 128 x 128 x 16 MMA is bound by the
// operand reads and takes about as long as a 128 x 256 x 16 one, so narrow
// tiles run at half rate.  With BN = 256 the columns past the last
// full 256-wide tile are covered by swapped tiles: up to 128 rows of W as
// the MMA's M side against 256 rows of A as its N side (the accumulator
// holds the transposed block: epi_single reads and writes it column by column,
// the other epilogues transpose it back through a 16 x 32 shared-memory
// buffer per warp).  DiT-XL/2's N = 1152 layers then
// run as 4 x 32 full tiles + 16 swapped tiles, one wave of 144 tiles.
#include "ff_common.cuh"
#include "ff_tc.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

namespace ff {

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int THREADS = 320;  // producer, MMA, 8 epilogue warps
using namespace tc;

__device__ unsigned int g_watchdog;

__device__ __forceinline__ bool mbar_wait_g(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait(b, parity, abort_flag, &g_watchdog);
}
// the producer's waits for a free stage poll: a suspended wait woke up
// several hundred cycles after the stage's MMAs completed, and the ring is
// only four stages deep
__device__ __forceinline__ bool mbar_wait_p(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait<true>(b, parity, abort_flag, &g_watchdog);
}
// the MMA warp's waits: every lane waits, the vote keeps the loop control
// (and the descriptors computed under it) warp-uniform, so the elected lane's
// tcgen05.mma does not block the issuing thread
__device__ __forceinline__ bool mbar_wait_u(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  const bool ok = mbar_test(b, parity) || mbar_wait_g(b, parity, abort_flag);
  return __all_sync(0xffffffffu, ok);
}

template <int BN> struct Cfg {
  static constexpr int STAGES = 4;
  static constexpr uint32_t A_BYTES = BM * BK * 2;
  static constexpr uint32_t B_BYTES = BN * BK * 2;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t TMEM_COLS = 2 * BN;
  // 4 KB per epilogue warp: two 32 x 32 bf16 output blocks for the TMA-store
  // epilogues, or the 16 x 32 fp32 transpose buffer of a swapped tile
  static constexpr uint32_t XPOSE_BYTES = 8 * 4096;
  static constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE_BYTES + XPOSE_BYTES + 256;
  // instruction descriptor, kind::f16: D fp32 (bit 4), A bf16 (bits 7-9 = 1),
  // B bf16 (bits 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                    ((uint32_t)(BM >> 4) << 24);
};

// Tile list of one launch: n_norm normal tiles (128 rows of A x BN rows of
// W, in the order of grouped_tile), then swapped tiles (128 rows of W x 256
// rows of A).
struct TileMap {
  int num_m;   // 128-row blocks of A
  int n_full;  // BN-wide column blocks of the normal tiles
  int n_norm;  // num_m * n_full
  int num_m2;  // 256-row blocks of A (swapped tiles)
  int n_tiles; // n_norm + swapped tiles
  int staged;  // normal tiles store out (and hist_out) through shared memory + TMA
  // one tile per CTA: the residual (bit 0) and the history base (bit 1) can be
  // described by a tensor map.  epi_single takes them so; the shared epilogue
  // loads them with TMA into the ring, idle after its mainloop, where the
  // LayerNorm is fused (its other instances load them per lane)
  int pre;
};

// 64-byte-swizzled [32 rows x 32 bf16] block: 16-byte chunk k of row r
__device__ __forceinline__ uint32_t blk_off(int r, int k) { return (uint32_t)(r * 64 + ((k ^ ((r >> 1) & 3)) << 4)); }
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}
__device__ __forceinline__ float2 unpack2(uint32_t u) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
}
// gelu_tanh_fast on 16 packed pairs
__device__ __forceinline__ void gelu_pairs(f32x2 (&y)[16]) {
  const unsigned long long k0 = f2u(GELU_K0, GELU_K0), k1 = f2u(GELU_K1, GELU_K1), hf = f2u(0.5f, 0.5f);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const unsigned long long in = fmul2(y[i], ffma2(fmul2(y[i], y[i]), k1, k0)), hx = fmul2(y[i], hf);
    y[i] = ffma2(hx, f2u(tanh_approx(lo_f(in)), tanh_approx(hi_f(in))), hx);
  }
}
struct TileAt {
  bool sw;
  int m0, n0;  // first output row / column
};
// Tile order: groups of GM row blocks, each swept over all column blocks with
// its rows fastest, so the tiles running together cover about a square of the
// output and a group's rows of A are read from DRAM once (with all row blocks
// fastest, 14310 x 2048 x 8192 read its 234 MB of A for each of the 8 column
// blocks: 1515 MB of DRAM traffic and 322 us, now 291 us).
template <int GM>
__device__ __forceinline__ void grouped_tile(int tile, int num_m, int num_n, int& m, int& n) {
  const int g = tile / (GM * num_n), r = tile - g * GM * num_n;
  const int gm = min(GM, num_m - g * GM);
  n = r / gm;
  m = g * GM + r - n * gm;
}
template <int BN>
__device__ __forceinline__ TileAt tile_at(const TileMap& t, int tile) {
  if (tile < t.n_norm) {
    int m, n;
    grouped_tile<16>(tile, t.num_m, t.n_full, m, n);
    return {false, m * BM, n * BN};
  }
  const int u = tile - t.n_norm;
  return {true, (u % t.num_m2) * 256, t.n_full * BN + (u / t.num_m2) * 128};
}

// Per-warp constants of the epilogue warps.
struct EpiWarp {
  uint8_t* smem;      // the 1024-aligned shared-memory base (ring first)
  uint8_t* ep;        // the warp's 4 KB output / transpose buffer
  uint64_t* rbar;     // per-warp residual / history-base barriers
  uint64_t* tfull;    // accumulator-full barriers
  volatile int* abort_flag;
  uint32_t tmem_base;
  int warp, lane, q, h, row, c_lo;
};

// The epilogue comes in three forms, a kernel instance each, so that none pays
// registers or branches for the others:
//   EPI_FULL    gate, residual, history increment (any of them);
//   EPI_PLAIN   bias, RoPE, activation only (qkv, fc1, linear1);
//   EPI_SINGLE  EPI_FULL with a residual where every CTA holds one tile, so
//               nothing hides the epilogue (epi_single below);
//   EPI_SINGLE_HIST  the same with a history increment and no residual.
enum { EPI_FULL = 0, EPI_PLAIN = 1, EPI_SINGLE = 2, EPI_SINGLE_HIST = 3 };

// The epilogue of one tile, inlined once per problem of the launch so that
// every EpiArgs / TileMap field and tensor map is read from its own kernel
// parameter (a run-time choice between two parameter structs turns every
// field access of the inner loops into a generic load).  PLAIN: normal
// tiles without residual preloads (the second problem of a grouped launch,
// the CTA pairs).  Returns false when the accumulator wait gave up.
template <int BN, bool PLAIN, int LN, int EPI>
__device__ __forceinline__ bool epi_tile(const EpiWarp& W, const EpiArgs& e, const TileMap& tm, const int M,
                                         const int N, const TileAt t, const int acc, const uint32_t aph,
                                         uint32_t& epi_cnt, const CUtensorMap* tmO, const CUtensorMap* tmH,
                                         const CUtensorMap* tmR, const CUtensorMap* tmHB) {
  const int warp = W.warp, lane = W.lane, q = W.q, h = W.h, row = W.row, c_lo = W.c_lo;
  uint8_t* const smem = W.smem;
  uint8_t* const ep = W.ep;
  float* const xp = reinterpret_cast<float*>(ep);
  uint64_t* const rbar = W.rbar;
  uint64_t* const tfull = W.tfull;
  volatile int* const abort_flag = W.abort_flag;
  const uint32_t tmem_base = W.tmem_base;
  const int pre = PLAIN || LN == 0 ? 0 : tm.pre;
  constexpr int LNM = LN == 1 ? 1 : LN == 2 ? 2 : 0;
  const bool sw = !PLAIN && t.sw;
  uint4 pr[4], ph[4];
  float pb = 0.f, pg0 = 0.f, pg1 = 0.f;
  // staged epilogue: residual / history-base rows of chunk n0 into pr /
  // ph; bias and gate of column n0 + lane into pb / pg0 / pg1 (shared
  // across the warp by shuffles: the warp's 32 rows lie in samples
  // b_lo .. b_hi, at most two of them)
  const int wr0 = t.m0 + q * 32;
  const int b_lo = e.gate ? epi_batch(e, min(wr0, M - 1)) : 0;
  const int b_hi = e.gate ? epi_batch(e, min(wr0 + 31, M - 1)) : 0;
  auto fetch = [&](int n0) {
    const int m = t.m0 + row;
    const bool cin = n0 + lane < N;
    pb = (e.bias && cin) ? __bfloat162float(reinterpret_cast<const bf16*>(e.bias)[n0 + lane]) : 0.f;
    pg0 = (e.gate && cin) ? e.gate[(size_t)b_lo * e.gate_stride + n0 + lane] : 0.f;
    pg1 = (e.gate && cin && b_hi != b_lo) ? e.gate[(size_t)b_hi * e.gate_stride + n0 + lane] : pg0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = m < M && n0 + 8 * k < N;
      if (e.resid && !(pre & 1))
        pr[k] = in ? *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(e.resid) +
                                                      (size_t)m * e.ld_resid + n0 + 8 * k)
                   : make_uint4(0, 0, 0, 0);
      if (e.hist_out && !(pre & 2))
        ph[k] = in ? *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(e.hist_base) +
                                                      (size_t)m * e.ldo + n0 + 8 * k)
                   : make_uint4(0, 0, 0, 0);
    }
  };
  // EPI_PLAIN: the chunk's bias in 16-byte loads, the same for every lane (one
  // sector each), a chunk ahead
  uint4 bv4[4];
  const bool bias_al = !((uintptr_t)e.bias & 15);
  auto fetch_bias = [&](int n0) {
    const bf16* bp = reinterpret_cast<const bf16*>(e.bias) + n0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (!e.bias || n0 + 8 * k >= N) {
        bv4[k] = make_uint4(0, 0, 0, 0);
      } else if (bias_al) {
        bv4[k] = *reinterpret_cast<const uint4*>(bp + 8 * k);
      } else {
        const unsigned short* us = reinterpret_cast<const unsigned short*>(bp + 8 * k);
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = (uint32_t)us[2 * i] | ((uint32_t)us[2 * i + 1] << 16);
        bv4[k] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  };
  if (tm.staged && !sw) {
    if constexpr (EPI == EPI_PLAIN) fetch_bias(t.n0 + c_lo); else fetch(t.n0 + c_lo);
  }
  int ok = 1;
  if (lane == 0) ok = mbar_wait_g(&tfull[acc], aph, abort_flag) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) return false;
  tc_fence_after();
  // One tile per CTA: the ring's last readers (this tile's MMAs) are
  // complete, so the warp's residual / history-base blocks (4 x 32 x 32
  // bf16 each, 64-byte swizzle: the layout of the output blocks) come by
  // TMA into its 8 KB slices of the ring; waited for at first use.
  uint8_t* rsm = smem + (warp - 2) * 8192;
  uint8_t* hsm = smem + 65536 + (warp - 2) * 8192;
  bool pre_wait = pre != 0;
  if (pre && lane == 0) {
    mbar_expect_tx(&rbar[warp - 2], ((pre & 1) ? 8192u : 0u) + ((pre & 2) ? 8192u : 0u));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int x = sw ? t.n0 + q * 32 : t.n0 + c_lo + 32 * i;
      const int y = sw ? t.m0 + h * (BN / 2) + 32 * i : t.m0 + q * 32;
      if (pre & 1) tma_load(tmR, &rbar[warp - 2], rsm + i * 2048, x, y);
      if (pre & 2) tma_load(tmHB, &rbar[warp - 2], hsm + i * 2048, x, y);
    }
  }
  auto pre_ready = [&]() -> bool {
    if (!pre_wait) return true;
    pre_wait = false;
    int w = 1;
    if (lane == 0) w = mbar_wait_g(&rbar[warp - 2], 0, abort_flag) ? 1 : 0;
    return __shfl_sync(0xffffffffu, w, 0) != 0;
  };
  const uint32_t tq = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
  if (!sw && !tm.staged) {
    const int m = t.m0 + row;
    const float2 lnr = ((LN == 1 && e.ln_in) && m < M) ? ln_row(e, m) : make_float2(1.f, 0.f);
    for (int c = h * (BN / 2); c < (h + 1) * (BN / 2); c += 32) {
      const int n0 = t.n0 + c;
      if (n0 >= N) break;
      float v[32];
      tmem_ld32(tq + (uint32_t)c, v);
      if (m < M) {
        const float2 st = epi_chunk<bf16, 32, LNM>(e, m, n0, N, v, lnr);
        if ((LN == 2 && e.ln_out)) ln_put(e, m, n0, st);
      }
    }
  } else if (EPI == EPI_PLAIN && !sw) {
    // Staged epilogue of a layer without gate, residual and history: as
    // below, in packed fp32 pairs and without shuffles (the costliest
    // instructions beside a mainloop): on single CTAs, 4096 x 4608 x 1152 with
    // GELU 39.7 -> 33.6 us, 14310 x 8192 x 2048 302 -> 273 (on pairs 30 and 254)
    const int m = t.m0 + row;
    for (int c = c_lo; c < c_lo + BN / 2; c += 32) {
      const int n0 = t.n0 + c;
      if (n0 >= N) break;
      float v[32];
      tmem_ld32(tq + (uint32_t)c, v);
      unsigned long long y[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t bb[4] = {bv4[k].x, bv4[k].y, bv4[k].z, bv4[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          y[4 * k + i] = fadd2(f2u(v[8 * k + 2 * i], v[8 * k + 2 * i + 1]), bf2u(bb[i]));
      }
      if (c + 32 < c_lo + BN / 2 && n0 + 32 < N) fetch_bias(n0 + 32);
      if (e.act == 1 && !e.rope && n0 >= e.act_col0) {
        gelu_pairs(y);
      } else if (e.rope || e.act) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          v[2 * i] = lo_f(y[i]);
          v[2 * i + 1] = hi_f(y[i]);
        }
        if (m < M) epi_rope_act<bf16, 32>(e, m, n0, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) y[i] = f2u(v[2 * i], v[2 * i + 1]);
      }
      uint8_t* b0 = ep + (epi_cnt & 1) * 2048;
      if (lane == 0) bulk_wait_read<1>();
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 4; ++k)
        *reinterpret_cast<uint4*>(b0 + blk_off(lane, k)) =
            make_uint4(pack2(lo_f(y[4 * k]), hi_f(y[4 * k])), pack2(lo_f(y[4 * k + 1]), hi_f(y[4 * k + 1])),
                       pack2(lo_f(y[4 * k + 2]), hi_f(y[4 * k + 2])), pack2(lo_f(y[4 * k + 3]), hi_f(y[4 * k + 3])));
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store(tmO, b0, n0, t.m0 + q * 32);
        bulk_commit();
      }
      ++epi_cnt;
    }
  } else if (!sw) {
    // Staged epilogue: each 32-row x 32-column chunk is written into a
    // swizzled shared-memory block and stored by one TMA copy (whole
    // lines instead of one L2 request per 16 bytes).  The residual and
    // history-base rows of a chunk are loaded ahead: the first chunk's
    // before the accumulator wait, the next one's while the current
    // chunk is finished.
    const int m = t.m0 + row;
    const int bm = m < M ? epi_batch(e, m) : 0;   // the row's sample (fused LayerNorm)
    const float2 lnr = ((LN == 1 && e.ln_in) && m < M) ? ln_row(e, m) : make_float2(1.f, 0.f);
    for (int c = c_lo; c < c_lo + BN / 2; c += 32) {
      const int n0 = t.n0 + c;
      if (n0 >= N) break;
      float v[32];
      tmem_ld32(tq + (uint32_t)c, v);
      // y = gate * act(rope(acc + bias)), the order of epi_math; rows
      // past M are not stored (the TMA store clips them)
      if ((LN == 1 && e.ln_in) && m < M) ln_correct<32>(e, bm, n0, N, lnr, v);
      if (e.bias) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += __shfl_sync(0xffffffffu, pb, j);
      }
      if (m < M) epi_rope_act<bf16, 32>(e, m, n0, v);
      if (e.gate) {
        if (b_hi == b_lo) {  // the warp's rows in one sample: one gate row (warp-uniform)
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] *= __shfl_sync(0xffffffffu, pg0, j);
        } else {
          const bool lo = m >= M || epi_batch(e, m) == b_lo;
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float g0 = __shfl_sync(0xffffffffu, pg0, j), g1 = __shfl_sync(0xffffffffu, pg1, j);
            v[j] *= lo ? g0 : g1;
          }
        }
      }
      if (pre) {
        if (!pre_ready()) { ok = 0; break; }
        const uint8_t* rb = rsm + ((c - c_lo) >> 5) * 2048;
        const uint8_t* hb2 = hsm + ((c - c_lo) >> 5) * 2048;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (pre & 1) pr[k] = *reinterpret_cast<const uint4*>(rb + blk_off(lane, k));
          if (pre & 2) ph[k] = *reinterpret_cast<const uint4*>(hb2 + blk_off(lane, k));
        }
      }
      uint32_t ob[16], hb[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t rr[4] = {pr[k].x, pr[k].y, pr[k].z, pr[k].w};
        const uint32_t hh[4] = {ph[k].x, ph[k].y, ph[k].z, ph[k].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float a = v[8 * k + 2 * i], b = v[8 * k + 2 * i + 1];
          if (e.resid) {
            const float2 r2 = unpack2(rr[i]);
            a += r2.x;
            b += r2.y;
          }
          ob[4 * k + i] = pack2(a, b);
          if (e.hist_out) {  // stored(out) - hist_base
            const float2 o2 = unpack2(ob[4 * k + i]), h2 = unpack2(hh[i]);
            hb[4 * k + i] = pack2(o2.x - h2.x, o2.y - h2.y);
          }
        }
      }
      if ((LN == 2 && e.ln_out) && m < M) {  // the next layer's scaled copy and chunk statistics
        float x[32];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float2 f = unpack2(ob[k]);
          x[2 * k] = f.x;
          x[2 * k + 1] = f.y;
        }
        ln_put(e, m, n0, ln_emit<32>(e, m, bm, n0, x));
      }
      if (c + 32 < c_lo + BN / 2 && n0 + 32 < N) fetch(n0 + 32);
      // block(s) for this chunk: out alternates between the two when
      // there is no history stream, else out -> block 0, hist -> block 1
      uint8_t* b0 = ep + (e.hist_out ? 0 : (epi_cnt & 1) * 2048);
      if (lane == 0) {
        if (e.hist_out) bulk_wait_read<0>(); else bulk_wait_read<1>();
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        *reinterpret_cast<uint4*>(b0 + blk_off(lane, k)) = make_uint4(ob[4 * k], ob[4 * k + 1], ob[4 * k + 2], ob[4 * k + 3]);
        if (e.hist_out)
          *reinterpret_cast<uint4*>(ep + 2048 + blk_off(lane, k)) =
              make_uint4(hb[4 * k], hb[4 * k + 1], hb[4 * k + 2], hb[4 * k + 3]);
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store(tmO, b0, n0, t.m0 + q * 32);
        if (e.hist_out) tma_store(tmH, ep + 2048, n0, t.m0 + q * 32);
        bulk_commit();
      }
      ++epi_cnt;
    }
  } else {
    // lane = output column n + lane; TMEM column = output row.  Blocks of
    // 16 rows x 32 columns go through the warp's buffer (XOR-swizzled,
    // conflict-free both ways); afterwards lane l holds row l / 2,
    // columns 16 (l % 2) .. + 15.
    const int n = t.n0 + q * 32;
    if (lane == 0) bulk_wait_read<0>();  // TMA stores of earlier tiles done reading the buffer
    __syncwarp();
    // preloaded form: the lane's 16 columns are the same for every block
    // of rows, so their bias stays in registers and the gate row is
    // reloaded only when the row's sample changes
    const bool pre_sw = pre && !e.out_f32 && e.split_col >= N && !e.rope;
    float bv[16], gv[16];
    int gb = -1;
    if (pre_sw) {
      const int nc0 = n + (lane & 1) * 16;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        float b8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (e.bias && nc0 + 8 * g < N) ld16(reinterpret_cast<const bf16*>(e.bias) + nc0 + 8 * g, b8);
#pragma unroll
        for (int k = 0; k < 8; ++k) bv[8 * g + k] = b8[k];
      }
    }
    for (int c = h * (BN / 2); c < (h + 1) * (BN / 2) && n < N; c += 16) {
      const int m0 = t.m0 + c;
      if (m0 >= M) break;
      {
        float u[16];
        tmem_ld16(tq + (uint32_t)c, u);  // u[j] = out[m0 + j][n + lane]
#pragma unroll
        for (int j = 0; j < 16; ++j) xp[j * 32 + (lane ^ j)] = u[j];
      }
      __syncwarp();
      const int r = lane >> 1, c0 = (lane & 1) * 16;
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = xp[r * 32 + ((c0 + j) ^ r)];  // out[m0 + r][n + c0 + j]
      __syncwarp();
      const int m = m0 + r;
      if (pre && !e.out_f32 && e.split_col >= N) {
        // residual / history base of row m from the warp's ring slices
        // (block (row in the warp's 128 rows) / 32, 16-byte chunks
        // c0 / 8 and c0 / 8 + 1 of that row)
        if (!pre_ready()) break;
        float2 lst = make_float2(0.f, 0.f);   // fused LayerNorm: this lane's 16-column statistics
        if (m < M) {
          if (pre_sw) {  // epi_math's order: act(acc + bias) * gate
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += bv[j];
            epi_rope_act<bf16, 16>(e, m, n + c0, v);
            if (e.gate) {
              const int bt = epi_batch(e, m);
              if (bt != gb) {
                gb = bt;
                const float* gp = e.gate + (size_t)bt * e.gate_stride + n + c0;
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                  const float4 g4 = n + c0 + j < N ? *reinterpret_cast<const float4*>(gp + j)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
                  gv[j] = g4.x; gv[j + 1] = g4.y; gv[j + 2] = g4.z; gv[j + 3] = g4.w;
                }
              }
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] *= gv[j];
            }
          } else {
            epi_math<bf16, 16, LNM>(e, m, n + c0, N, v);
          }
          const int rw = c - h * (BN / 2) + r;
          const uint32_t base = (uint32_t)((rw >> 5) * 2048);
          float xs[16];   // stored values of the lane's 16 columns
#pragma unroll
          for (int j = 0; j < 16; ++j) xs[j] = 0.f;
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const int nc = n + c0 + 8 * g;
            if (nc >= N) continue;
            const uint32_t off = base + blk_off(rw & 31, (c0 >> 3) + g);
            uint4 rv = make_uint4(0, 0, 0, 0), hv = make_uint4(0, 0, 0, 0);
            if (pre & 1)
              rv = *reinterpret_cast<const uint4*>(rsm + off);
            else if (e.resid)
              rv = *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(e.resid) + (size_t)m * e.ld_resid + nc);
            if (e.hist_out)
              hv = (pre & 2) ? *reinterpret_cast<const uint4*>(hsm + off)
                                : *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(e.hist_base) +
                                                                  (size_t)m * e.ldo + nc);
            const uint32_t rr4[4] = {rv.x, rv.y, rv.z, rv.w}, hh4[4] = {hv.x, hv.y, hv.z, hv.w};
            uint32_t ob[4], hb[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              float a = v[8 * g + 2 * i], b = v[8 * g + 2 * i + 1];
              if (e.resid) {
                const float2 r2 = unpack2(rr4[i]);
                a += r2.x;
                b += r2.y;
              }
              ob[i] = pack2(a, b);
              const float2 o2 = unpack2(ob[i]);
              xs[8 * g + 2 * i] = o2.x;
              xs[8 * g + 2 * i + 1] = o2.y;
              if (e.hist_out) {  // stored(out) - hist_base
                const float2 h2 = unpack2(hh4[i]);
                hb[i] = pack2(o2.x - h2.x, o2.y - h2.y);
              }
            }
            *reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(e.out) + (size_t)m * e.ldo + nc) =
                make_uint4(ob[0], ob[1], ob[2], ob[3]);
            if (e.hist_out)
              *reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(e.hist_out) + (size_t)m * e.ldo + nc) =
                  make_uint4(hb[0], hb[1], hb[2], hb[3]);
          }
          if ((LN == 2 && e.ln_out)) lst = ln_emit<16>(e, m, epi_batch(e, m), n + c0, xs);
        }
        if ((LN == 2 && e.ln_out)) {  // lanes l and l ^ 1 hold the two halves of the row's 32 columns
          lst = ln_pair(lst);
          if (!(lane & 1) && m < M) ln_put(e, m, n, lst);
        }
        continue;
      }
      float2 lst = make_float2(0.f, 0.f);
      if (m < M) lst = epi_chunk<bf16, 16, LNM>(e, m, n + c0, N, v, (LN == 1 && e.ln_in) ? ln_row(e, m) : make_float2(1.f, 0.f));
      if ((LN == 2 && e.ln_out)) {
        lst = ln_pair(lst);
        if (!(lane & 1) && m < M) ln_put(e, m, n, lst);
      }
    }
  }
  // a warp whose columns all lie past N never read its blocks: their
  // copies still land before it moves on
  if (pre_wait) pre_ready();
  return true;
}

// First row past the sample of row r.
__device__ __forceinline__ int sample_end(const EpiArgs& e, int r) {
  if (r < e.seg_split) return min((r / e.rpb0 + 1) * e.rpb0, e.seg_split);
  return e.seg_split + ((r - e.seg_split) / e.rpb1 + 1) * e.rpb1;
}

// Epilogue of the one tile of a CTA: out = resid + gate * act(acc + bias), and
// the history increment.  Nothing runs beside it, so it is all latency: the
// warp's residual blocks (32 x 32 bf16, 64-byte swizzle) are replaced by the
// output in place and stored from there, one buffer per block, so no block
// waits for another's store; two of them, the bias and the gate arrive
// during the mainloop, the other blocks in the idle ring after it.  Normal tile:
// lane = row, bias and gate broadcast from shared memory.  Swapped tile: lane =
// column, so bias and gate stay in registers and each row of a block is one
// 64-byte read and write, with no transposition buffer.
// Against the shared form with its block-by-block buffers, shuffled bias and
// gate and transposed swapped tiles: 4096 x 1152 x 1152 (gate, residual) 19.3
// -> 14.5 us, 4096 x 1152 x 4608 (and history) 46.2 -> 40.1 us.
template <int BN, bool RES>
__device__ __forceinline__ bool epi_single(const EpiWarp& W, const EpiArgs& e, const int M, const int N, const TileAt t,
                                           const CUtensorMap* tmO, const CUtensorMap* tmH, const CUtensorMap* tmR,
                                           const CUtensorMap* tmHB) {
  const int lane = W.lane, q = W.q, h = W.h;
  uint8_t* const ep = W.ep;
  uint8_t* const ring = W.smem + (W.warp - 2) * 16384;    // 12 KB of blocks, 1.5 KB of constants
  uint64_t* const rbar = &W.rbar[W.warp - 2];
  const bool hist = !RES || e.hist_out != nullptr;
  // block i: output rows y0 .. y0 + 31, columns x0 .. x0 + 31
  const int xb = t.sw ? t.n0 + q * 32 : t.n0 + W.c_lo, yb = t.sw ? t.m0 + h * (BN / 2) : t.m0 + q * 32;
  const int dx = t.sw ? 0 : 32, dy = t.sw ? 32 : 0;
  const int nb = xb < N && yb < M ? min(4, t.sw ? (M - yb + 31) >> 5 : (N - xb + 31) >> 5) : 0;
  auto rblk = [&](int i) { return i < 2 ? ep + i * 2048 : ring + (i - 2) * 2048; };
  auto hblk = [&](int i) { return ring + 4096 + i * 2048; };
  const int early = RES ? min(nb, 2) : 0;
  if (lane == 0 && early > 0) {
    mbar_expect_tx(rbar, early * 2048u);
    for (int i = 0; i < early; ++i) tma_load(tmR, rbar, rblk(i), xb + i * dx, yb + i * dy);
  }
  // bias and gate: normal tile, columns xb + 32 i + lane, samples of the warp's
  // first and last row; swapped tile, column xb + lane, samples of block i's
  // first and last row (at most two samples in 32 rows)
  float cb[4], c0[4], c1[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int col = xb + i * dx + lane;
    const int r0 = min(yb + i * dy, M - 1), r1 = min(yb + i * dy + 31, M - 1);
    const bool in = i < nb && col < N;
    cb[i] = in && e.bias ? __bfloat162float(reinterpret_cast<const bf16*>(e.bias)[col]) : 0.f;
    c0[i] = in && e.gate ? e.gate[(size_t)epi_batch(e, r0) * e.gate_stride + col] : 1.f;
    c1[i] = in && e.gate ? e.gate[(size_t)epi_batch(e, r1) * e.gate_stride + col] : 1.f;
  }
  int ok = 1;
  if (lane == 0) {
    ok = mbar_wait_p(W.tfull, 0, W.abort_flag) ? 1 : 0;
    if (early > 0) {  // the early blocks (they land before the CTA exits, also after a failed wait)
      const unsigned long long t0 = gtimer();
      while (!mbar_try(rbar, 0))
        if (gtimer() - t0 > WAIT_LIMIT_NS) { atomicOr(&g_watchdog, 2u); *W.abort_flag = 1; ok = 0; break; }
    }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) return false;
  tc_fence_after();
  const int late = (RES ? nb - early : 0) + (hist ? nb : 0);
  if (lane == 0 && late > 0) {
    mbar_expect_tx(rbar, late * 2048u);
    for (int i = 0; i < nb; ++i) {
      if (hist) tma_load(tmHB, rbar, hblk(i), xb + i * dx, yb + i * dy);
      if (RES && i >= 2) tma_load(tmR, rbar, rblk(i), xb + i * dx, yb + i * dy);
    }
  }
  bool late_wait = late > 0;
  auto late_ready = [&]() -> bool {
    if (!late_wait) return true;
    late_wait = false;
    int w = 1;
    if (lane == 0) w = mbar_wait_p(rbar, RES ? 1 : 0, W.abort_flag) ? 1 : 0;
    return __shfl_sync(0xffffffffu, w, 0) != 0;
  };
  const uint32_t tq = W.tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * (BN / 2));
  auto store = [&](int i) {
    fence_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store(tmO, rblk(i), xb + i * dx, yb + i * dy);
      if (hist) tma_store(tmH, hblk(i), xb + i * dx, yb + i * dy);
      bulk_commit();
    }
  };
  if (!t.sw) {
    float* const cst = reinterpret_cast<float*>(ring + 12288);   // bias [128], gate of the first and last row's sample
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      cst[32 * i + lane] = cb[i];
      cst[128 + 32 * i + lane] = c0[i];
      cst[256 + 32 * i + lane] = c1[i];
    }
    __syncwarp();
    const int r0 = min(yb, M - 1), m = min(yb + lane, M - 1);
    const float* const gp = cst + (e.gate && epi_batch(e, m) != epi_batch(e, r0) ? 256 : 128);
    for (int i = 0; i < nb; ++i) {
      float v[32];
      tmem_ld32(tq + (uint32_t)(32 * i), v);
      unsigned long long y[16];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const ulonglong2 b2 = *reinterpret_cast<const ulonglong2*>(cst + 32 * i + 4 * k);
        y[2 * k] = fadd2(f2u(v[4 * k], v[4 * k + 1]), b2.x);
        y[2 * k + 1] = fadd2(f2u(v[4 * k + 2], v[4 * k + 3]), b2.y);
      }
      if (e.act == 1) gelu_pairs(y);
      if (e.gate) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const ulonglong2 g2 = *reinterpret_cast<const ulonglong2*>(gp + 32 * i + 4 * k);
          y[2 * k] = fmul2(y[2 * k], g2.x);
          y[2 * k + 1] = fmul2(y[2 * k + 1], g2.y);
        }
      }
      if ((hist || i >= 2) && !late_ready()) return false;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint4* const rp = reinterpret_cast<uint4*>(rblk(i) + blk_off(lane, k));
        const uint4 r4 = RES ? *rp : make_uint4(0, 0, 0, 0);
        const uint32_t rr[4] = {r4.x, r4.y, r4.z, r4.w};
        uint32_t ob[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const unsigned long long a = RES ? fadd2(y[4 * k + z], bf2u(rr[z])) : y[4 * k + z];
          ob[z] = pack2(lo_f(a), hi_f(a));
        }
        *rp = make_uint4(ob[0], ob[1], ob[2], ob[3]);
        if (hist) {  // stored(out) - hist_base
          uint4* const hp = reinterpret_cast<uint4*>(hblk(i) + blk_off(lane, k));
          const uint4 h4 = *hp;
          const uint32_t hh[4] = {h4.x, h4.y, h4.z, h4.w};
          uint32_t hb[4];
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            const float2 o2 = unpack2(ob[z]), h2 = unpack2(hh[z]);
            hb[z] = pack2(o2.x - h2.x, o2.y - h2.y);
          }
          *hp = make_uint4(hb[0], hb[1], hb[2], hb[3]);
        }
      }
      store(i);
    }
  } else {
    uint32_t off[4];   // byte of column `lane` in a block row r with (r >> 1) & 3 = x
#pragma unroll
    for (int x = 0; x < 4; ++x) off[x] = (uint32_t)((((lane >> 3) ^ x) << 4) + (lane & 7) * 2);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i >= nb) break;
      float v[32];
      tmem_ld32(tq + (uint32_t)(32 * i), v);   // v[j] = acc[yb + 32 i + j][xb + lane]
      const int y0 = yb + 32 * i;
      const int jb = sample_end(e, y0) - y0;   // rows from jb on: the second sample's gate
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] += cb[i];
      if (e.act == 1) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = gelu_tanh_fast(v[j]);
      }
      // (the gate's product rounded before the residual is added, as in the normal
      // tiles: no contraction to an fma)
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] = __fmul_rn(v[j], j < jb ? c0[i] : c1[i]);
      if ((hist || i >= 2) && !late_ready()) return false;
      // a pass of reads, then one of writes: alternating, every read would wait
      // behind the write before it (37 x 48 x 1192, residual and history 13.6 -> 10.8 us,
      // 4096 x 1152 x 4608 with gate, residual and history 43.0 -> 40.1)
      auto at = [&](uint8_t* blk, int j) { return reinterpret_cast<bf16*>(blk + j * 64 + off[(j >> 1) & 3]); };
      if constexpr (RES) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __fadd_rn(v[j], __bfloat162float(*at(rblk(i), j)));
      }
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const bf16 o = __float2bfloat16_rn(v[j]);
        *at(rblk(i), j) = o;
        v[j] = __bfloat162float(o);
      }
      if (hist) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] -= __bfloat162float(*at(hblk(i), j));
#pragma unroll
        for (int j = 0; j < 32; ++j) *at(hblk(i), j) = __float2bfloat16_rn(v[j]);
      }
      store(i);
    }
  }
  return true;
}

// GROUPED: a second problem (group 1, tm1.n_tiles > 0) of the same N and K
// with its own A, W, rows and epilogue (the text stream of a two-stream
// block beside the image stream), its tiles first in the tile list; both
// groups then have only normal tiles and no residual preloads.  Without
// GROUPED the group-1 parameters are unused.
template <int BN, bool GROUPED, int LN, int EPI>
__global__ void __launch_bounds__(THREADS, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              const __grid_constant__ CUtensorMap tmW128, const __grid_constant__ CUtensorMap tmA256,
              const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmH,
              const __grid_constant__ CUtensorMap tmR, const __grid_constant__ CUtensorMap tmHB, int M0, int N, int K,
              const __grid_constant__ TileMap tm0, const __grid_constant__ EpiArgs e0,
              const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
              const __grid_constant__ CUtensorMap tmO1, const __grid_constant__ CUtensorMap tmH1, int M1,
              const __grid_constant__ TileMap tm1, const __grid_constant__ EpiArgs e1) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  float* xpose = reinterpret_cast<float*>(sB + C::STAGES * C::B_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + C::STAGES * C::B_BYTES + C::XPOSE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* rbar = tempty + 2;  // per epilogue warp: its residual / history-base blocks landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rbar + 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n1 = GROUPED ? tm1.n_tiles : 0;
  const int num_tiles = tm0.n_tiles + n1;
  const int num_kb = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 256);
    }
    for (int w = 0; w < 8; ++w) mbar_init(&rbar[w], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB) : "memory");
    if (tm0.pre & 1) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmR) : "memory");
    if (tm0.pre & 2) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmHB) : "memory");
    if (GROUPED && n1) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA1) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB1) : "memory");
    }
    if (tm0.n_tiles > tm0.n_norm) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmW128) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA256) : "memory");
    }
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                 "r"(C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // dependents may launch once every CTA holds its TMEM; the previous
  // kernel's outputs are complete after the wait
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        const bool g1 = GROUPED && tile < n1;
        const TileAt t = g1 ? tile_at<BN>(tm1, tile) : tile_at<BN>(tm0, tile - n1);
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it % C::STAGES;
          const uint32_t ph = (it / C::STAGES) & 1;
          if (!mbar_wait_p(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          mbar_expect_tx(&full[s], C::STAGE_BYTES);
          // normal: A rows -> M side, W rows -> N side; swapped: the reverse.
          // (Each call names its kernel parameter: a tensor map must stay in
          // parameter space, never be copied to local memory.)
          if (g1) {
            tma_load(&tmA1, &full[s], sA + s * C::A_BYTES, kb * BK, t.m0);
            tma_load(&tmB1, &full[s], sB + s * C::B_BYTES, kb * BK, t.n0);
          } else if (!t.sw) {
            tma_load(&tmA, &full[s], sA + s * C::A_BYTES, kb * BK, t.m0);
            tma_load(&tmB, &full[s], sB + s * C::B_BYTES, kb * BK, t.n0);
          } else {
            tma_load(&tmW128, &full[s], sA + s * C::A_BYTES, kb * BK, t.n0);
            tma_load(&tmA256, &full[s], sB + s * C::B_BYTES, kb * BK, t.m0);
          }
        }
      }
      // Copies still in flight complete on their full barriers; wait for
      // the last ring's worth so none lands after the CTA exits.
      for (uint32_t k = 0; k < (uint32_t)C::STAGES && k < it; ++k) {
        const uint32_t j = it - 1 - k;
        const unsigned long long t0 = gtimer();
        while (!mbar_try(&full[j % C::STAGES], (j / C::STAGES) & 1)) {
          if (gtimer() - t0 > WAIT_LIMIT_NS) { atomicOr(&g_watchdog, 2u); break; }
        }
      }
    }
  } else if (warp == 1) {
    // the whole warp runs the loop, one elected block issues a step's MMAs and
    // its commit (with polled waits in epi_single: DiT-XL/2 sampling 47.7 -> 47.4 ms)
    uint32_t it = 0;
    int tc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x, ++tc) {
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1;
      if (!mbar_wait_u(&tempty[acc], aph ^ 1, abort_flag)) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
      for (int kb = 0; kb < num_kb; ++kb, ++it) {
        const int s = it % C::STAGES;
        const uint32_t ph = (it / C::STAGES) & 1;
        if (!mbar_wait_u(&full[s], ph, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint64_t ad = sw128_desc(saddr(sA + s * C::A_BYTES));
        const uint64_t bd = sw128_desc(saddr(sB + s * C::B_BYTES));
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)  // +32 bytes (16 bf16) along K inside the swizzle atom
            umma(d_tmem, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), C::IDESC, (kb | k) != 0);
          umma_commit(&empty[s]);
        }
      }
      if (!ok) break;
      if (elect_one()) umma_commit(&tfull[acc]);
    }
  } else {
    // 8 epilogue warps: TMEM lane quarter q = warp % 4 (the quarter a warp
    // may access), column half h of the tile
    const int q = warp & 3;
    const int h = (warp - 2) >> 2;
    const EpiWarp W = {smem, reinterpret_cast<uint8_t*>(xpose) + (warp - 2) * 4096, rbar, tfull, abort_flag,
                       tmem_base, warp, lane, q, h, q * 32 + lane, h * (BN / 2)};
    int tc = 0;
    uint32_t epi_cnt = 0;
    for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x, ++tc) {
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1;
      bool ok;
      if constexpr (EPI == EPI_SINGLE || EPI == EPI_SINGLE_HIST) {
        ok = epi_single<BN, EPI == EPI_SINGLE>(W, e0, M0, N, tile_at<BN>(tm0, tile), &tmO, &tmH, &tmR, &tmHB);
      } else if constexpr (GROUPED) {
        ok = tile < n1 ? epi_tile<BN, true, LN, EPI>(W, e1, tm1, M1, N, tile_at<BN>(tm1, tile), acc, aph, epi_cnt, &tmO1,
                                            &tmH1, &tmR, &tmHB)
                       : epi_tile<BN, true, LN, EPI>(W, e0, tm0, M0, N, tile_at<BN>(tm0, tile - n1), acc, aph, epi_cnt, &tmO,
                                            &tmH, &tmR, &tmHB);
      } else {
        ok = epi_tile<BN, false, LN, EPI>(W, e0, tm0, M0, N, tile_at<BN>(tm0, tile), acc, aph, epi_cnt, &tmO, &tmH, &tmR,
                                 &tmHB);
      }
      if (!ok) break;
      tc_fence_before();
      mbar_arrive(&tempty[acc]);
    }
    if (lane == 0) bulk_wait_all();  // TMA stores complete before exit
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// CTA-pair variant: a cluster of 2 CTAs computes a 256 x BN tile with
// tcgen05.mma.cta_group::2 (M = 256).  Each CTA stages its own 128 rows of A
// and half (BN/2 rows) of W, so per CTA the shared-memory traffic per FLOP
// is that of a 128 x 2BN tile.  The even CTA issues the MMAs; its full
// barriers collect both CTAs' TMA bytes; commits are multicast to both CTAs'
// empty / accumulator-full barriers; both CTAs' epilogues arrive on the even
// CTA's accumulator-empty barrier.
// ---------------------------------------------------------------------------
template <int BN> struct Cfg2 {
  static constexpr int HB = BN / 2;
  static constexpr int STAGES = BN >= 256 ? 6 : 8;
  static constexpr uint32_t A_BYTES = BM * BK * 2;
  static constexpr uint32_t B_BYTES = HB * BK * 2;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr uint32_t TMEM_COLS = 2 * BN;
  static constexpr uint32_t XPOSE_BYTES = 8 * 4096;  // the staged epilogue's output blocks
  static constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE_BYTES + XPOSE_BYTES + 256;
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                    ((uint32_t)(256 >> 4) << 24);
};

// The epilogue is epi_tile's (staged TMA-store blocks where tm.staged), each
// CTA on its own 128 rows of the pair's 256-row tile.
// GROUPED: a second problem of the same N and K (its own A, W, rows,
// epilogue and store maps: the text stream of a two-stream block beside the
// image stream), its tiles first in the tile list, so its few tiles fill the
// first problem's last wave instead of running alone on a handful of SMs.
template <int BN, int LN, bool GROUPED, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k_gemm_tc2(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmH, int M, int N, int K,
               const __grid_constant__ TileMap tm, const __grid_constant__ EpiArgs e,
               const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
               const __grid_constant__ CUtensorMap tmO1, const __grid_constant__ CUtensorMap tmH1, int M1,
               const __grid_constant__ TileMap tm1, const __grid_constant__ EpiArgs e1) {
  using C = Cfg2<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  uint8_t* xpose = sB + C::STAGES * C::B_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(xpose + C::XPOSE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int num_m = (M + 2 * BM - 1) / (2 * BM), num_n = (N + BN - 1) / BN;
  const int num_m1 = GROUPED ? (M1 + 2 * BM - 1) / (2 * BM) : 0;
  const int n1 = num_m1 * num_n;              // group 1's tiles come first
  const int num_tiles = n1 + num_m * num_n;
  // (group, row block, column block) of tile `tile`
  auto tile_of = [&](int tile, bool& g1, int& mb, int& nb) {
    g1 = GROUPED && tile < n1;
    const int u = g1 ? tile : tile - n1;
    grouped_tile<8>(u, g1 ? num_m1 : num_m, num_n, mb, nb);
  };
  const int num_kb = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 2 * 256);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB) : "memory");
    if (GROUPED && n1) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA1) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB1) : "memory");
    }
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(tmem_slot)),
                 "r"(C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // both CTAs' barriers initialised before any cross-CTA use
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // dependents may launch once every CTA holds its TMEM; the previous
  // kernel's outputs are complete after the wait
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs) {
        bool g1;
        int mb, nb;
        tile_of(tile, g1, mb, nb);
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it % C::STAGES;
          const uint32_t ph = (it / C::STAGES) & 1;
          if (!mbar_wait_p(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          if (leader) mbar_expect_tx(&full[s], 2 * C::STAGE_BYTES);
          const uint32_t fb = map_to(&full[s], 0);
          // (each call names its kernel parameter: a tensor map stays in
          // parameter space)
          if (g1) {
            tma_load_pair(&tmA1, fb, sA + s * C::A_BYTES, kb * BK, mb * 2 * BM + (int)rank * BM);
            tma_load_pair(&tmB1, fb, sB + s * C::B_BYTES, kb * BK, nb * BN + (int)rank * C::HB);
          } else {
            tma_load_pair(&tmA, fb, sA + s * C::A_BYTES, kb * BK, mb * 2 * BM + (int)rank * BM);
            tma_load_pair(&tmB, fb, sB + s * C::B_BYTES, kb * BK, nb * BN + (int)rank * C::HB);
          }
        }
      }
      if (leader) {  // the even CTA's full barriers track both CTAs' copies
        for (uint32_t k = 0; k < (uint32_t)C::STAGES && k < it; ++k) {
          const uint32_t j = it - 1 - k;
          const unsigned long long t0 = gtimer();
          while (!mbar_try(&full[j % C::STAGES], (j / C::STAGES) & 1)) {
            if (gtimer() - t0 > WAIT_LIMIT_NS) { atomicOr(&g_watchdog, 2u); break; }
          }
        }
      }
    }
  } else if (warp == 1) {
    if (leader) {  // the whole warp runs the loop, one elected lane issues
      uint32_t it = 0;
      int tc = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += npairs, ++tc) {
        const int acc = tc & 1;
        const uint32_t aph = (tc >> 1) & 1;
        if (!mbar_wait_u(&tempty[acc], aph ^ 1, abort_flag)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        for (int kb = 0; kb < num_kb; ++kb, ++it) {
          const int s = it % C::STAGES;
          const uint32_t ph = (it / C::STAGES) & 1;
          if (!mbar_wait_u(&full[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint64_t ad = sw128_desc(saddr(sA + s * C::A_BYTES));
          const uint64_t bd = sw128_desc(saddr(sB + s * C::B_BYTES));
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_pair(d_tmem, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), C::IDESC, (kb | k) != 0);
            umma_commit_pair(&empty[s]);
          }
        }
        if (!ok) break;
        if (elect_one()) umma_commit_pair(&tfull[acc]);
      }
    }
  } else {
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    const int h = (warp - 2) >> 2;  // column half of the tile
    const EpiWarp W = {smem, xpose + (warp - 2) * 4096, tfull, tfull, abort_flag, tmem_base, warp, lane, q, h,
                       q * 32 + lane, h * (BN / 2)};
    int tc = 0;
    uint32_t epi_cnt = 0;
    for (int tile = pair; tile < num_tiles; tile += npairs, ++tc) {
      bool g1;
      int mb, nb;
      tile_of(tile, g1, mb, nb);
      const int acc = tc & 1;
      const uint32_t aph = (tc >> 1) & 1;
      const TileAt t = {false, mb * 2 * BM + (int)rank * BM, nb * BN};
      bool ok;
      if (g1)
        ok = epi_tile<BN, true, LN, EPI>(W, e1, tm1, M1, N, t, acc, aph, epi_cnt, &tmO1, &tmH1, &tmO1,
                                                     &tmO1);
      else
        ok = epi_tile<BN, true, LN, EPI>(W, e, tm, M, N, t, acc, aph, epi_cnt, &tmO, &tmH, &tmO, &tmO);
      if (!ok) break;
      tc_fence_before();
      mbar_arrive_cluster(map_to(&tempty[acc], 0));
    }
    if (lane == 0) bulk_wait_all();  // TMA stores complete before exit
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();  // no CTA leaves while its peer may still address its TMEM or barriers
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Kernel instance for a fused-LayerNorm side (0 none, 1 consumer, 2 producer)
// and an epilogue form (the fused sides have the full one only).
template <int BN, bool G>
auto gemm_fn(int ln, int epi) -> decltype(&k_gemm_tc<BN, G, 0, EPI_FULL>) {
  if (ln == 1) return k_gemm_tc<BN, G, 1, EPI_FULL>;
  if (ln == 2) return k_gemm_tc<BN, G, 2, EPI_FULL>;
  if (epi == EPI_PLAIN) return k_gemm_tc<BN, G, 0, EPI_PLAIN>;
  if constexpr (!G) {
    if (epi == EPI_SINGLE) return k_gemm_tc<BN, G, 0, EPI_SINGLE>;
    if (epi == EPI_SINGLE_HIST) return k_gemm_tc<BN, G, 0, EPI_SINGLE_HIST>;
  }
  return k_gemm_tc<BN, G, 0, EPI_FULL>;
}
template <int BN, bool G = false>
auto gemm2_fn(int ln, int epi) -> decltype(&k_gemm_tc2<BN, 0, G, EPI_FULL>) {
  if (ln == 1) return k_gemm_tc2<BN, 1, G, EPI_FULL>;
  if (ln == 2) return k_gemm_tc2<BN, 2, G, EPI_FULL>;
  return epi == EPI_PLAIN ? k_gemm_tc2<BN, 0, G, EPI_PLAIN> : k_gemm_tc2<BN, 0, G, EPI_FULL>;
}
int epi_form(const EpiArgs& e) { return e.gate || e.resid || e.hist_out ? EPI_FULL : EPI_PLAIN; }
int ln_side(const EpiArgs& e) { return e.ln_in ? 1 : e.ln_out ? 2 : 0; }
// a fused LayerNorm side: one side per launch, bf16 output of whole
// 32-column chunks for the producer, 16-byte aligned rows everywhere
bool ln_ok(const EpiArgs& e, int N) {
  if (e.ln_in && e.ln_out) return false;
  if (e.ln_out && (e.out_f32 || N % 32 != 0 || e.split_col < N || e.ldo % 8 != 0 || !e.ln_scale || !e.ln_stats ||
                   e.ln_stride % 4 != 0 || ((uintptr_t)e.ln_scale & 15) || ((uintptr_t)e.ln_out & 15) ||
                   e.ln_slots * 32 < N))
    return false;
  if (e.ln_in && (!e.ln_c || !e.ln_d || e.ln_cols <= 0 || e.ln_slots * 32 != e.ln_cols || (e.ln_slots & 1) ||
                  e.ln_cd_stride % 4 != 0 ||
                  ((uintptr_t)e.ln_c & 15) || ((uintptr_t)e.ln_d & 15) || ((uintptr_t)e.ln_in & 15)))
    return false;
  return true;
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_once;
int g_sms = 0;

bool init_driver() {
  std::call_once(g_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_sms <= 0) g_sms = 148;
    auto smem = [](const void* fn, size_t bytes) {
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    for (int ln = 0; ln < 3; ++ln)
      for (int epi : {EPI_FULL, EPI_PLAIN, EPI_SINGLE, EPI_SINGLE_HIST}) {
        smem((const void*)gemm_fn<256, false>(ln, epi), Cfg<256>::SMEM);
        smem((const void*)gemm_fn<256, true>(ln, epi), Cfg<256>::SMEM);
        smem((const void*)gemm2_fn<128>(ln, epi), Cfg2<128>::SMEM);
        smem((const void*)gemm2_fn<256>(ln, epi), Cfg2<256>::SMEM);
        smem((const void*)gemm2_fn<128, true>(ln, epi), Cfg2<128>::SMEM);
        smem((const void*)gemm2_fn<256, true>(ln, epi), Cfg2<256>::SMEM);
      }
  });
  return g_encode != nullptr;
}

// 2-D bf16 tensor map over a row-major [rows, cols] matrix with row stride
// ld elements, box [box_rows, 64], 128-byte swizzle, zero fill out of bounds.
bool make_map(CUtensorMap* m, const void* base, int rows, int cols, int ld, int box_rows) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Store map of the staged epilogue: [rows, cols] bf16 with row stride ld
// elements, box 32 x 32, 64-byte swizzle (one block row = 64 bytes).
bool make_store_map(CUtensorMap* m, void* base, int rows, int cols, int ld) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {32, 32};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// The staged (TMA-store) epilogue: one bf16 output of 16-byte aligned rows,
// plus the history stream when present, and a warp's 32 rows spanning at
// most two gate rows.  Encodes the store maps; false where the per-lane
// store path has to be used.
bool staged_maps(const EpiArgs& e, int M, int N, CUtensorMap* mo, CUtensorMap* mh) {
  const bool aligned = !((uintptr_t)e.out & 15) && e.ldo % 8 == 0 &&
                       (!e.hist_out || (!((uintptr_t)e.hist_out & 15) && !((uintptr_t)e.hist_base & 15)));
  const bool gate_ok = !e.gate || ((e.seg_split <= 0 || e.rpb0 >= 32) && e.rpb1 >= 32);
  return !e.out_f32 && e.split_col >= N && aligned && gate_ok && make_store_map(mo, e.out, M, N, e.ldo) &&
         (!e.hist_out || make_store_map(mh, e.hist_out, M, N, e.ldo));
}

// Tile width of the CTA-pair kernel, 0 where single CTAs are the better
// choice.  m256, t128x256: 256-row blocks of A over the launch's problems, and
// the single-CTA kernel's 128 x 256 tiles (its swapped remainder tiles
// counted).  A pair's 256 x 256 tile and a CTA's 128 x 256 tile take each SM
// about as long, the pair 5-20% less (an SM takes in about 64 bytes of tiles a
// clock: 48 KB per 64-deep step alone, 32 KB in a pair, against 512 clocks of
// MMA; 14310 x 6144 x 2048 219 -> 199 us, 4608 x 3072 x 2048 51 -> 43, 4096 x
// 4608 x 1152 with GELU 33.8 -> 29.5), so pairs run wherever they need no more
// waves; within one wave short reductions stay with single CTAs, whose
// epilogue blocks come by TMA (1024 x 4608 x 256 9.2 against 9.5 us), up to a K
// of 1024 and with a history increment, whose epilogue is the longest, of 4096
// (singles against pairs, gate, residual and history: 1103 x 3624 x 2296 29.7
// and 38.1 us, 1485 x 1816 x 3864 7% apart; without history, 718 x 5768 x 4744,
// pairs take 14% less).
// 128-wide pair tiles take 0.85 of a 256-wide tile's time, so they pay only
// where the 256-wide tiles leave half the pairs idle; counted at half the time
// they took 8192 x 8192 x 8192, 945 us against 590.
int pair_bn(long long m256, long long t128x256, int N, int K, bool hist, int sms) {
  const int pairs = sms / 2;
  const long long w_single = (t128x256 + sms - 1) / sms;
  const long long w256 = (m256 * ((N + 255) / 256) + pairs - 1) / pairs;
  const long long w128 = (m256 * ((N + 127) / 128) + pairs - 1) / pairs;
  if (w256 > w_single) return 0;
  if (w128 <= w256) return 128;
  return w256 > 1 || K >= (hist ? 4096 : 1024) ? 256 : 0;
}

// The single-CTA kernel's 128 x 256 tiles, remainder columns in swapped tiles.
long long wide_tiles(int M, int N) {
  const int rem = N % 256;
  return (long long)((M + BM - 1) / BM) * (N / 256) + (rem ? (long long)((rem + 127) / 128) * ((M + 255) / 256) : 0);
}

}  // namespace

cudaError_t gemm_tc(int M, int N, int K, const void* A, int lda, const void* W, int ldw, const EpiArgs& e,
                    cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (!init_driver()) return cudaErrorNotSupported;
  if (K % 8 != 0 || lda % 8 != 0 || ldw % 8 != 0 || N % 8 != 0) return cudaErrorInvalidValue;
  if (!ln_ok(e, N)) return cudaErrorInvalidValue;
  if (((uintptr_t)A & 15) || ((uintptr_t)W & 15)) return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  const int bn = M >= 2 * BM ? pair_bn((M + 2 * BM - 1) / (2 * BM), wide_tiles(M, N), N, K, e.hist_out != nullptr, g_sms) : 0;
  if (bn) {
    const int pairs = g_sms / 2;
    if (!make_map(&ma, A, M, K, lda, BM) || !make_map(&mb, W, N, K, ldw, bn / 2)) return cudaErrorInvalidValue;
    const long long tiles = (long long)((M + 2 * BM - 1) / (2 * BM)) * ((N + bn - 1) / bn);
    const int grid = 2 * (int)(tiles < pairs ? tiles : pairs);
    TileMap tm2 = {};
    CUtensorMap mo = ma, mh = ma;
    tm2.staged = staged_maps(e, M, N, &mo, &mh) ? 1 : 0;
    const TileMap none = {};
    if (bn == 256)
      launch_pdl(gemm2_fn<256>(ln_side(e), epi_form(e)), grid, THREADS, Cfg2<256>::SMEM, s, ma, mb, mo, mh, M, N, K, tm2, e, ma, mb,
                 mo, mh, 0, none, e);
    else
      launch_pdl(gemm2_fn<128>(ln_side(e), epi_form(e)), grid, THREADS, Cfg2<128>::SMEM, s, ma, mb, mo, mh, M, N, K, tm2, e, ma, mb,
                 mo, mh, 0, none, e);
    return launched();
  }
  // 128 x 256 tiles, remainder columns in swapped tiles (128-wide tiles would run
  // at half rate and be as many at least)
  TileMap tm;
  const int rem = N % 256;
  const long long tiles = wide_tiles(M, N);
  tm.num_m = (M + BM - 1) / BM;
  tm.num_m2 = (M + 255) / 256;
  tm.n_full = N / 256;
  tm.n_norm = tm.num_m * tm.n_full;
  tm.n_tiles = (int)tiles;
  tm.pre = 0;
  CUtensorMap mw128 = {}, ma256 = {}, mo = {}, mh = {}, mr = {}, mhb = {};
  if (!make_map(&ma, A, M, K, lda, BM) || !make_map(&mb, W, N, K, ldw, 256)) return cudaErrorInvalidValue;
  if (rem && (!make_map(&mw128, W, N, K, ldw, BM) || !make_map(&ma256, A, M, K, lda, 256)))
    return cudaErrorInvalidValue;
  tm.staged = staged_maps(e, M, N, &mo, &mh) ? 1 : 0;
  // one tile per CTA: residual / history-base blocks by TMA (16-byte aligned
  // rows; otherwise the per-lane loads stay)
  int epi = epi_form(e);
  if (tm.staged && tiles <= g_sms) {
    if (e.resid && make_store_map(&mr, const_cast<void*>(e.resid), M, N, e.ld_resid)) tm.pre |= 1;
    if (e.hist_out && make_store_map(&mhb, const_cast<void*>(e.hist_base), M, N, e.ldo)) tm.pre |= 2;
    const bool blocks = (!e.resid || (tm.pre & 1)) && (!e.hist_out || (tm.pre & 2)) && tm.pre;
    if (blocks && !e.rope && e.act != 2 && e.act_col0 == 0) epi = e.resid ? EPI_SINGLE : EPI_SINGLE_HIST;
  }
  const int grid = (int)(tiles < g_sms ? tiles : g_sms);
  const TileMap none = {};
  launch_pdl(gemm_fn<256, false>(ln_side(e), epi), grid, THREADS, Cfg<256>::SMEM, s, ma, mb, mw128, ma256, mo, mh, mr, mhb, M, N, K, tm,
             e, ma, mb, mo, mh, 0, none, e);
  return launched();
}

namespace {
// Normal 128 x 256 tiles of one problem (N a multiple of 256) with the
// staged TMA-store epilogue where the output allows it.
bool group_maps(int M, int N, int K, const void* A, int lda, const void* W, int ldw, const EpiArgs& e, TileMap* tm,
                CUtensorMap* ma, CUtensorMap* mb, CUtensorMap* mo, CUtensorMap* mh) {
  *tm = {};
  tm->num_m = (M + BM - 1) / BM;
  tm->num_m2 = (M + 255) / 256;
  tm->n_full = N / 256;
  tm->n_norm = tm->num_m * tm->n_full;
  tm->n_tiles = tm->n_norm;
  if (!make_map(ma, A, M, K, lda, BM) || !make_map(mb, W, N, K, ldw, 256)) return false;
  *mo = *ma;
  *mh = *ma;
  tm->staged = staged_maps(e, M, N, mo, mh) ? 1 : 0;
  return true;
}
}  // namespace

cudaError_t gemm_tc_grouped(int M0, const void* A0, const void* W0, const EpiArgs& e0, int M1, const void* A1,
                            const void* W1, const EpiArgs& e1, int N, int K, int lda, int ldw, cudaStream_t s) {
  if (M1 <= 0) return gemm_tc(M0, N, K, A0, lda, W0, ldw, e0, s);
  if (M0 <= 0) return gemm_tc(M1, N, K, A1, lda, W1, ldw, e1, s);
  if (!init_driver()) return cudaErrorNotSupported;
  if (!ln_ok(e0, N) || !ln_ok(e1, N) || (ln_side(e0) && ln_side(e1) && ln_side(e0) != ln_side(e1)))
    return cudaErrorInvalidValue;
  // both problems in one CTA-pair launch (256-row tiles of the text rows,
  // then of the image rows)
  const long long rows_t = ((M0 + 2 * BM - 1) / (2 * BM)) + ((M1 + 2 * BM - 1) / (2 * BM));
  const int bn = M0 >= 2 * BM ? pair_bn(rows_t, wide_tiles(M0, N) + wide_tiles(M1, N), N, K, false, g_sms) : 0;
  if (bn) {
    if (K % 8 != 0 || lda % 8 != 0 || ldw % 8 != 0 || N % 8 != 0) return cudaErrorInvalidValue;
    if (((uintptr_t)A0 & 15) || ((uintptr_t)W0 & 15) || ((uintptr_t)A1 & 15) || ((uintptr_t)W1 & 15))
      return cudaErrorInvalidValue;
    const int pairs = g_sms / 2;
    CUtensorMap a0, b0, a1, b1;
    if (!make_map(&a0, A0, M0, K, lda, BM) || !make_map(&b0, W0, N, K, ldw, bn / 2) ||
        !make_map(&a1, A1, M1, K, lda, BM) || !make_map(&b1, W1, N, K, ldw, bn / 2))
      return cudaErrorInvalidValue;
    TileMap t0 = {}, t1 = {};
    CUtensorMap o0 = a0, h0 = a0, o1 = a1, h1 = a1;
    t0.staged = staged_maps(e0, M0, N, &o0, &h0) ? 1 : 0;
    t1.staged = staged_maps(e1, M1, N, &o1, &h1) ? 1 : 0;
    const long long tiles = rows_t * ((N + bn - 1) / bn);
    const int grid = 2 * (int)(tiles < pairs ? tiles : pairs);
    const int ln = std::max(ln_side(e0), ln_side(e1));
    const int epi = epi_form(e0) == EPI_PLAIN && epi_form(e1) == EPI_PLAIN ? EPI_PLAIN : EPI_FULL;
    if (bn == 256)
      launch_pdl(gemm2_fn<256, true>(ln, epi), grid, THREADS, Cfg2<256>::SMEM, s, a0, b0, o0, h0, M0, N, K, t0, e0, a1, b1, o1,
                 h1, M1, t1, e1);
    else
      launch_pdl(gemm2_fn<128, true>(ln, epi), grid, THREADS, Cfg2<128>::SMEM, s, a0, b0, o0, h0, M0, N, K, t0, e0, a1, b1, o1,
                 h1, M1, t1, e1);
    return launched();
  }
  // column counts that need swapped tiles run as two launches
  if (N % 256 != 0) {
    const cudaError_t r = gemm_tc(M1, N, K, A1, lda, W1, ldw, e1, s);
    return r != cudaSuccess ? r : gemm_tc(M0, N, K, A0, lda, W0, ldw, e0, s);
  }
  if (K % 8 != 0 || lda % 8 != 0 || ldw % 8 != 0) return cudaErrorInvalidValue;
  if (((uintptr_t)A0 & 15) || ((uintptr_t)W0 & 15) || ((uintptr_t)A1 & 15) || ((uintptr_t)W1 & 15))
    return cudaErrorInvalidValue;
  TileMap t0, t1;
  CUtensorMap a0, b0, o0, h0, a1, b1, o1, h1;
  if (!group_maps(M0, N, K, A0, lda, W0, ldw, e0, &t0, &a0, &b0, &o0, &h0) ||
      !group_maps(M1, N, K, A1, lda, W1, ldw, e1, &t1, &a1, &b1, &o1, &h1))
    return cudaErrorInvalidValue;
  const long long tiles = (long long)t0.n_tiles + t1.n_tiles;
  const int grid = (int)(tiles < g_sms ? tiles : g_sms);
  const int ln = std::max(ln_side(e0), ln_side(e1));
  const int epi = epi_form(e0) == EPI_PLAIN && epi_form(e1) == EPI_PLAIN ? EPI_PLAIN : EPI_FULL;
  launch_pdl(gemm_fn<256, true>(ln, epi), grid, THREADS, Cfg<256>::SMEM, s, a0, b0, a0, a0, o0, h0, a0, a0, M0, N, K, t0, e0, a1,
             b1, o1, h1, M1, t1, e1);
  return launched();
}

// ---------------------------------------------------------------------------
// Watchdog probe (failure-detection test hook): one CTA takes TMEM like the
// GEMM does, then waits with the GEMM's bounded wait on an mbarrier that
// nothing arrives on.  The wait gives up after limit_ns, raises the same
// watchdog flag a stuck GEMM raises, and the CTA frees its TMEM and returns.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(64, 1) k_watchdog_probe(unsigned long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);   // one arrival expected; none comes
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_slot)), "r"(32)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (lane == 0) mbar_wait<true>(&bar, 0, &abort_flag, &g_watchdog, limit_ns);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(32) : "memory");
  }
}

cudaError_t watchdog_probe(unsigned long long limit_ns, cudaStream_t s) {
  k_watchdog_probe<<<1, 64, 0, s>>>(limit_ns);
  count_launches(1);
  return cudaGetLastError();
}

unsigned int gemm_tc_watchdog_take() {
  unsigned int v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_watchdog, sizeof(v)) != cudaSuccess) return 0;
  if (v) cudaMemcpyToSymbol(g_watchdog, &z, sizeof(z));
  return v;
}

}  // namespace ff
