// Dense prompt prefill kernels (sm_103a): the tcgen05 GEMM with its fused epilogues, causal
// attention of the prompt's tokens over the user's KV cache, row RMSNorm, the prompt's input rows
// and the greedy argmax over the column tiles.
//
// The prefill computes what one decode step per prompt token computes (section III: a stage
// applies its block range to every token; the head's sampler is greedy), with the tokens of a
// pass as the rows of dense matrix products instead of one weight pass per token.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "../../include/kafila_gemm.h"
#include "prefill_tc.cuh"

namespace kfl {

namespace {

// ---------------------------------------------------------------------------- GEMM epilogues
// Thread = one token t of the tile (its tensor-memory lane); v[j] = Y[t][n + j], j < 32.

template <int MODE>
struct EpiState {
  float best = -INFINITY;
  int bidx = 0x7FFFFFFF;
};

template <int MODE>
__device__ __forceinline__ void epilogue32(const PrefillEpiParams &ep, int t, int n, const uint32_t (&r)[32],
                                           EpiState<MODE> &st) {
  float v[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
  if constexpr (MODE == PE_STORE || MODE == PE_RESID) {
    float *row = ep.out + (size_t)t * ep.ldo + n;
    if (n + 32 <= ep.N) {
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        float4 y = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        if constexpr (MODE == PE_RESID) {
          const float4 h = *reinterpret_cast<const float4 *>(row + j);
          y.x += h.x;
          y.y += h.y;
          y.z += h.z;
          y.w += h.w;
        }
        *reinterpret_cast<float4 *>(row + j) = y;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (n + j < ep.N) row[j] = (MODE == PE_RESID ? row[j] : 0.f) + v[j];
    }
  } else if constexpr (MODE == PE_SWIGLU) {
    // 16 outputs j0 .. j0 + 15, as hi and lo terms
    const int j0 = n >> 1;
    uint32_t w[8], wl[8];
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      const float g0 = v[2 * i], u0 = v[2 * i + 1], g1 = v[2 * i + 2], u1 = v[2 * i + 3];
      split_pack(g0 / (1.0f + expf(-g0)) * u0, g1 / (1.0f + expf(-g1)) * u1, w[i / 2], wl[i / 2], ep.f16, ep.err);
    }
    uint16_t *row = ep.out16 + (size_t)t * ep.ldo16 + j0;
    uint16_t *rlo = ep.out16lo + (size_t)t * ep.ldo16 + j0;
    if (n + 32 <= ep.N) {
      reinterpret_cast<uint4 *>(row)[0] = make_uint4(w[0], w[1], w[2], w[3]);
      reinterpret_cast<uint4 *>(row)[1] = make_uint4(w[4], w[5], w[6], w[7]);
      reinterpret_cast<uint4 *>(rlo)[0] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
      reinterpret_cast<uint4 *>(rlo)[1] = make_uint4(wl[4], wl[5], wl[6], wl[7]);
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (n + 2 * i + 1 < ep.N) {
          row[i] = (uint16_t)(w[i / 2] >> (16 * (i & 1)));
          rlo[i] = (uint16_t)(wl[i / 2] >> (16 * (i & 1)));
        }
    }
  } else if constexpr (MODE == PE_QKV) {
    const int pos = ep.positions[t];
    if (pos < 0) return;
    const int half = ep.hd / 2;
    if (n < ep.qdim + ep.kvdim) {
      // 16 RoPE pairs (i, i + hd/2) of one head
      const bool is_q = n < ep.qdim;
      const int r0 = is_q ? n : n - ep.qdim;
      const int head = r0 / ep.hd, i0 = (r0 % ep.hd) / 2;
      // the 16 factors of each kind are 64 contiguous, 64-byte aligned bytes
      const float4 *cs = reinterpret_cast<const float4 *>(ep.rope_cos + (size_t)pos * half + i0);
      const float4 *sn = reinterpret_cast<const float4 *>(ep.rope_sin + (size_t)pos * half + i0);
      float c[16], sv[16];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 a = cs[j], b = sn[j];
        c[4 * j] = a.x, c[4 * j + 1] = a.y, c[4 * j + 2] = a.z, c[4 * j + 3] = a.w;
        sv[4 * j] = b.x, sv[4 * j + 1] = b.y, sv[4 * j + 2] = b.z, sv[4 * j + 3] = b.w;
      }
      uint16_t *dst;
      if (is_q) {
        dst = ep.out16 + (size_t)t * ep.ldo16 + (size_t)head * ep.hd;
      } else {
        dst = ep.kcache + (((size_t)ep.slot * ep.hkv + head) * ep.max_ctx + pos) * ep.hd;
      }
      if (is_q && ep.out) {  // q in fp32
        float *q1 = ep.out + (size_t)t * ep.ldo + (size_t)head * ep.hd + i0, *q2 = q1 + half;
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          float y1[4], y2[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float a1 = v[2 * (i + j)], a2 = v[2 * (i + j) + 1];
            y1[j] = a1 * c[i + j] - a2 * sv[i + j];
            y2[j] = a2 * c[i + j] + a1 * sv[i + j];
          }
          *reinterpret_cast<float4 *>(q1 + i) = make_float4(y1[0], y1[1], y1[2], y1[3]);
          *reinterpret_cast<float4 *>(q2 + i) = make_float4(y2[0], y2[1], y2[2], y2[3]);
        }
        return;
      }
      // rotated first halves -> dst[i0 ..], second halves -> dst[i0 + hd/2 ..]: 32 bytes each
      uint32_t w1[8], w2[8];
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        const float a1 = v[2 * i], a2 = v[2 * i + 1], b1 = v[2 * i + 2], b2 = v[2 * i + 3];
        w1[i / 2] = pack_bf16(a1 * c[i] - a2 * sv[i], b1 * c[i + 1] - b2 * sv[i + 1]);
        w2[i / 2] = pack_bf16(a2 * c[i] + a1 * sv[i], b2 * c[i + 1] + b1 * sv[i + 1]);
      }
      uint4 *d1 = reinterpret_cast<uint4 *>(dst + i0), *d2 = reinterpret_cast<uint4 *>(dst + i0 + half);
      d1[0] = make_uint4(w1[0], w1[1], w1[2], w1[3]);
      d1[1] = make_uint4(w1[4], w1[5], w1[6], w1[7]);
      d2[0] = make_uint4(w2[0], w2[1], w2[2], w2[3]);
      d2[1] = make_uint4(w2[4], w2[5], w2[6], w2[7]);
    } else {
      const int r0 = n - ep.qdim - ep.kvdim;
      const int head = r0 / ep.hd, j0 = r0 % ep.hd;
      uint16_t *dst = ep.vcache + (((size_t)ep.slot * ep.hkv + head) * ep.max_ctx + pos) * ep.hd + j0;
      uint32_t w[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
#pragma unroll
      for (int i = 0; i < 16; i += 4) reinterpret_cast<uint4 *>(dst)[i / 4] = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
  } else if constexpr (MODE == PE_ARGMAX) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (n + j < ep.N && v[j] > st.best) {
        st.best = v[j];
        st.bidx = n + j;
      }
  }
}

// The MMAs of one K block of 64 (a 128-byte swizzled row): 16 K values at a time, both terms of X
// against the same W slice.  A slice starts 32 bytes (2 in the descriptor's units) after the one before.
__device__ __forceinline__ void mma_kblock(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, bool accumulate) {
#pragma unroll
  for (int k = 0; k < PG_K / 16; ++k) {
    mma_bf16_ss(d, da + 2 * k, db + 2 * k, idesc, accumulate || k > 0);
    mma_bf16_ss(d, da + (PG_A_BYTES >> 4) + 2 * k, db + 2 * k, idesc, 1);
  }
}

// ---------------------------------------------------------------------------- GEMM kernel
// One CTA per SM walks its share of the tiles (TileShare).  The TMA ring runs on across tile
// boundaries, and two accumulators (all 512 TMEM columns) let the MMAs proceed while
// the epilogue warps read the previous one.  Warp 0 issues TMA, warp 1 MMAs, warps 2-5 (2-9) run the
// epilogue (warp w reads TMEM lanes 32 (w % 4) ..).  Every wait is bounded; a CTA that gives up sets
// ERR_TIMEOUT, lets its copies and MMAs in flight complete (bounded), frees its TMEM and returns.
//
// Bound by the tensor pipe (two terms against every weight).  Splitting K over clusters of 2 to 8 CTAs,
// as this did where the tiles fill the last round badly, cost 7 to 39 us a round of CTAs in cluster
// launch and distributed shared memory: the down projection of 500 tokens (56 tiles) took 173 us, now
// 85 with the kernel that sums its parts.  Two 7B-shaped blocks: 931 -> 815 us at 500 tokens, 2620 -> 1951 at
// 1500, 2608 at 2048 as before (its tiles fill their rounds).
//
// DRAIN (the plain product): each accumulator takes only PP_CHUNK K blocks, and eight epilogue warps add
// the chunks up in registers: tensor-core accumulation truncates (prefill_narrow_kernel says how
// much), and an unsplit K of 18944 leaves the product of 2048 tokens 3.8e-5 off, drained 3.3e-6.  A
// stage's products, of K = d_model mostly, go without: the sums' registers cost the fused epilogues
// spills.
//
// Residual products and Q/K/V take a long K in equal chunks, whose sums meet in the workspace while the
// next chunk multiplies (coalesced, loaded a step ahead: adding each to the rows of the residual stream
// took 2 to 13 % of a pass, as it stalled the MMAs).  O and down: at most PR_CHUNK K blocks (K = 4096:
// truncation takes 8e-6), where a whole tile of K = 18944 or 29568 lost 3.8e-5 or 5.9e-5.  Q/K/V of more
// than 2 PQ_CHUNK: at most PQ_CHUNK (K = 2048), because a softmax of large scores feels every relative
// error of q and k: two 72B-shaped int4 blocks of 900 tokens are 6.23e-3 from 64 bits unchunked, 6.17e-3 in
// chunks of 4096 and 6.14e-3 so.  Those two take 4985 us for 4890 unchunked, four 7B-shaped blocks of 2048
// tokens 5165 for 5098.
constexpr int PP_CHUNK = 16, PR_CHUNK = 64, PQ_CHUNK = 32;
// K blocks of one accumulation of a segment of n.
template <int MODE>
__device__ __forceinline__ int pp_chunk(int n) {
  if (MODE == PE_STORE) return PP_CHUNK;
  if ((MODE != PE_RESID && MODE != PE_QKV) || (MODE == PE_QKV && n <= 2 * PQ_CHUNK)) return n;
  constexpr int MOST = MODE == PE_RESID ? PR_CHUNK : PQ_CHUNK;
  const int parts = (n + MOST - 1) / MOST;
  return (n + parts - 1) / parts;
}
__host__ __device__ constexpr int pp_epi_warps(bool drain) { return drain ? 8 : 4; }
__host__ __device__ constexpr int pp_threads(bool drain) { return (2 + pp_epi_warps(drain)) * 32; }
constexpr int PP_TMEM_COLS = 2 * PG_N;

// Where (in float4, plus the token row) a partial holds columns 4 j .. of the tile.
__device__ __forceinline__ size_t wide_partial(int part, int j) { return ((size_t)part * (PG_N / 4) + j) * PG_M; }

template <int MODE, bool DRAIN>
__global__ void __launch_bounds__(pp_threads(DRAIN), 1)
    prefill_gemm_persistent(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_a2,
                            const __grid_constant__ CUtensorMap tm_b, int w_rows, TileShare share, float *ws,
                            PrefillEpiParams ep) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_full[PG_STAGES], s_empty[PG_STAGES], s_acc_full[2], s_acc_empty[2], s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const int t_tiles = (ep.T + PG_M - 1) / PG_M;
  const uint32_t raw = smem_addr(smem_raw);
  const uint32_t sa = (raw + 1023u) & ~1023u;  // [stage][hi, lo] activation tiles
  const uint32_t sb = sa + PG_STAGES * 2 * PG_A_BYTES;
  if (threadIdx.x == 0) {
    for (int s = 0; s < PG_STAGES; ++s) {
      mbar_init(smem_addr(&s_full[s]), 1);
      mbar_init(smem_addr(&s_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_addr(&s_acc_full[b]), 1);
      mbar_init(smem_addr(&s_acc_empty[b]), pp_epi_warps(DRAIN));  // one arrival per epilogue warp
    }
    mbar_init(smem_addr(&s_drain), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_addr(&s_tmem), PP_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int *abort_flag = &s_abort;
  pdl_launch_dependents();
  pdl_wait();

  if (warp == 0) {
    // ---- TMA producer (the whole warp, one elected lane issuing)
    asm volatile("fence.proxy.async;" ::: "memory");  // the previous kernel's stores, before TMA reads them
    int s = 0, use = 0;
    bool ok = true;
    for (TileWalk w(share); ok && w.next();) {
      const int t0 = (w.tile % t_tiles) * PG_M, n0 = (w.tile / t_tiles) * PG_N;
      for (int kb = w.kb0; kb < w.kb1; ++kb) {
        ok = __all_sync(0xffffffffu,
                        !*abort_flag && (use == 0 || mbar_wait(smem_addr(&s_empty[s]), (uint32_t)(use - 1) & 1)));
        if (!ok) break;
        const uint32_t full = smem_addr(&s_full[s]);
        if (elect_one()) {
          mbar_arrive_expect_tx(full, 2 * PG_A_BYTES + PG_B_BYTES);
          tma_load_2d(sa + s * 2 * PG_A_BYTES, &tm_a, kb * PG_K, t0, full);
          tma_load_2d(sa + s * 2 * PG_A_BYTES + PG_A_BYTES, &tm_a2, kb * PG_K, t0, full);
          // weight tiles: (column within the K tile, row within the row block, K tile, row block)
          if (w_rows)
            tma_load_2d(sb + s * PG_B_BYTES, &tm_b, kb * PG_K, n0, full);
          else
            tma_load_4d(sb + s * PG_B_BYTES, &tm_b, (kb & 1) * PG_K, 0, kb >> 1, n0 / RB, full);
        }
        __syncwarp();
        if (++s == PG_STAGES) s = 0, ++use;
      }
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicOr(ep.err, ERR_TIMEOUT);
      }
      // let the copies in flight land before the CTA's shared memory is released
      for (int i = 0; i < PG_STAGES; ++i) {
        const int last = use - (i >= s ? 1 : 0);
        if (last >= 0) mbar_wait(smem_addr(&s_full[i]), (uint32_t)last & 1);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (the whole warp, one elected lane issuing): chunk i of this CTA's segments
    // accumulates into TMEM columns (i % 2) * PG_N
    const uint32_t idesc = ep.f16 ? idesc_kind_f16(PG_M, PG_N, false) : idesc_kind_f16(PG_M, PG_N, true);
    TileWalk w(share);
    int s = 0, left = 0, chunk = 0;
    uint32_t use = 0;
    bool ok = true;
    for (int i = 0; ok; ++i) {
      if (left == 0) {
        if (!w.next()) break;
        left = w.kb1 - w.kb0;
        chunk = pp_chunk<MODE>(left);
      }
      const int n = min(left, chunk), buf = i & 1;
      left -= n;
      if (i >= 2) ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&s_acc_empty[buf]), ((i >> 1) - 1) & 1));
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)(buf * PG_N);
      for (int kb = 0; kb < n; ++kb) {
        ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_full[s]), use & 1));
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = sdesc_k_sw128(sa + s * 2 * PG_A_BYTES), db = sdesc_k_sw128(sb + s * PG_B_BYTES);
        if (elect_one()) {
          mma_kblock(d, da, db, idesc, kb != 0);
          mma_commit(smem_addr(&s_empty[s]));
        }
        __syncwarp();
        if (++s == PG_STAGES) s = 0, ++use;
      }
      if (ok && elect_one()) mma_commit(smem_addr(&s_acc_full[buf]));
      __syncwarp();
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(ep.err, ERR_TIMEOUT);
    }
    // every MMA issued has completed before TMEM can be freed
    if (elect_one()) mma_commit(smem_addr(&s_drain));
    __syncwarp();
    mbar_wait(smem_addr(&s_drain), 0);
  } else {
    // ---- epilogue warps: TMEM lanes 32 q .. 32 q + 31 (q = warp % 4) are tokens t0 + 32 q + lane
    const int q = warp & 3, row = 32 * q + lane;
    const uint32_t lanes = tmem + ((uint32_t)(32 * q) << 16);
    int i = 0;
    // accumulator i is complete; false: given up
    auto wait_acc = [&]() {
      const bool ready = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_acc_full[i & 1]), (i >> 1) & 1));
      if (!ready && lane == 0) {
        *abort_flag = 1;
        atomicOr(ep.err, ERR_TIMEOUT);
      }
      tc_fence_after();
      return ready;
    };
    auto release_acc = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&s_acc_empty[i & 1]));
      ++i;
    };
    bool ok = true;
    for (TileWalk w(share); ok && w.next();) {
      const int n_tile = w.tile / t_tiles, t = (w.tile % t_tiles) * PG_M + row, n0 = n_tile * PG_N;
      const bool whole = w.whole();
      EpiState<MODE> st;
      // where this row's partial sums are; a whole tile's chunks meet where this CTA's first part goes later
      float4 *part = reinterpret_cast<float4 *>(ws) + wide_partial(whole ? blockIdx.x : w.part, 0) + row;
      // 32 columns' sums, `last` if no chunk of them follows
      auto finish = [&](int c, const uint32_t(&r)[32], bool last) {
        if (whole && last) {
          if (t < ep.T) epilogue32<MODE>(ep, t, n0 + 32 * c, r, st);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            part[(8 * c + j) * PG_M] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                                   __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
        }
      };
      if constexpr (DRAIN) {
        // warps 2-5 take columns 0-127, warps 6-9 columns 128-255
        const int c0 = (warp - 2) >> 2 << 2;
        uint32_t sum[4][32];
        for (int left = w.kb1 - w.kb0; left > 0; left -= PP_CHUNK) {
          if (!(ok = wait_acc())) break;
          const bool first = left == w.kb1 - w.kb0;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            uint32_t r[16];
            tmem_ld16(lanes + (uint32_t)((i & 1) * PG_N + 32 * c0 + 16 * c), r);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              uint32_t &y = sum[c / 2][(c & 1) * 16 + j];
              y = first ? r[j] : __float_as_uint(__uint_as_float(y) + __uint_as_float(r[j]));
            }
          }
          release_acc();
        }
        if (!ok) break;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (n0 + 32 * (c0 + c) < ep.N) finish(c0 + c, sum[c], true);  // uniform across the warp
      } else {
        constexpr bool CHUNKS = MODE == PE_RESID || MODE == PE_QKV;
        const int chunk = pp_chunk<MODE>(w.kb1 - w.kb0);
        for (int left = w.kb1 - w.kb0, done = 0; left > 0; left -= chunk, ++done) {
          // the earlier chunks' sums of 32 columns, loaded one step ahead
          float4 x[2][8];
          auto fetch = [&](int c, float4(&y)[8]) {
            if (CHUNKS && done > 0 && n0 + 32 * c < ep.N)
#pragma unroll
              for (int j = 0; j < 8; ++j) y[j] = part[(8 * c + j) * PG_M];
          };
          fetch(0, x[0]);
          if (!(ok = wait_acc())) break;
          auto step = [&](int c, const float4(&y)[8]) {
            if (n0 + 32 * c >= ep.N) return;  // uniform across the warp
            uint32_t r[32];
            tmem_ld32(lanes + (uint32_t)((i & 1) * PG_N + 32 * c), r);
            if (CHUNKS && done > 0) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                r[4 * j] = __float_as_uint(y[j].x + __uint_as_float(r[4 * j]));
                r[4 * j + 1] = __float_as_uint(y[j].y + __uint_as_float(r[4 * j + 1]));
                r[4 * j + 2] = __float_as_uint(y[j].z + __uint_as_float(r[4 * j + 2]));
                r[4 * j + 3] = __float_as_uint(y[j].w + __uint_as_float(r[4 * j + 3]));
              }
            }
            finish(c, r, left <= chunk);
          };
          for (int c = 0; c < PG_N / 32; c += 2) {
            fetch(c + 1, x[1]);
            step(c, x[0]);
            if (c + 2 < PG_N / 32) fetch(c + 2, x[0]);
            step(c + 1, x[1]);
          }
          release_acc();
        }
        if (!ok) break;
        if constexpr (MODE == PE_ARGMAX) {
          if (whole && t < ep.T) {
            ep.amax[(size_t)t * ep.n_tiles + n_tile] = st.best;
            ep.aidx[(size_t)t * ep.n_tiles + n_tile] = st.bidx;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, PP_TMEM_COLS);
  }
}

// The tiles that several CTAs share: their partial sums, added in K order, and the epilogue.  One
// block (thread = token) per tile and 32 columns (PE_ARGMAX: per tile, whose maximum it keeps).
template <int MODE>
__global__ void __launch_bounds__(PG_M) wide_reduce_kernel(TileShare share, int gemm_ctas, const float *ws,
                                                            PrefillEpiParams ep) {
  pdl_launch_dependents();
  constexpr int CHUNKS = PG_N / 32, PER = MODE == PE_ARGMAX ? CHUNKS : 1;
  const int sk = blockIdx.x / (CHUNKS / PER), c0 = blockIdx.x % (CHUNKS / PER) * PER;
  const int t_tiles = (ep.T + PG_M - 1) / PG_M, tile = share.waves * gemm_ctas + sk;
  const TileParts parts(share, sk, gemm_ctas);
  const int n_tile = tile / t_tiles, t = (tile % t_tiles) * PG_M + threadIdx.x;
  pdl_wait();
  if (parts.n == 1 || t >= ep.T) return;
  EpiState<MODE> st;
  for (int c = c0; c < c0 + PER && n_tile * PG_N + 32 * c < ep.N; ++c) {
    float v[32] = {};
    for (int k = 0; k < parts.n; k += 2) {
      float4 x[2][8];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 *at =
            reinterpret_cast<const float4 *>(ws) + wide_partial(parts.part(k + i), 8 * c) + threadIdx.x;
#pragma unroll
        for (int j = 0; j < 8; ++j) x[i][j] = k + i < parts.n ? __ldcg(at + j * PG_M) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          v[4 * j] += x[i][j].x;
          v[4 * j + 1] += x[i][j].y;
          v[4 * j + 2] += x[i][j].z;
          v[4 * j + 3] += x[i][j].w;
        }
    }
    uint32_t r[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(v[j]);
    epilogue32<MODE>(ep, t, n_tile * PG_N + 32 * c, r, st);
  }
  if constexpr (MODE == PE_ARGMAX) {
    ep.amax[(size_t)t * ep.n_tiles + n_tile] = st.best;
    ep.aidx[(size_t)t * ep.n_tiles + n_tile] = st.bidx;
  }
}

// ---------------------------------------------------------------------------- attention
// Causal attention of a block of 64 prompt tokens (4 warps x 16) for one query head over the
// user's cache rows [0, position]: S = Q K^T and O = P V on bf16 m16n8k16 MMAs, softmax online
// over key blocks of 64 rows double-buffered in shared memory (rows padded by 16 bytes so the
// matrix loads are free of bank conflicts).
//
// A short prompt has few such blocks (28 at 43 tokens and 28 heads) while its keys may be many: the
// key blocks are then split over a cluster of up to 8 CTAs, whose (m, l, O) meet in distributed
// shared memory in rank order (43 tokens at 700: a serial chain of 12 key blocks, 31 us, on 28 of
// 152 SMs before).
//
// PRECISE: q is fp32 and enters, like the softmax weights, as a bf16 pair (rounded + rest, about 2^-17),
// as in the decode step's attention; the output has p.terms terms.  Twice the MMAs: taken for passes of up
// to 512 tokens and wherever the GEMMs run on few-token tiles (7B-shaped, 43 tokens at 700: the block's
// error against 64 bits 5.2e-4 -> 1.8e-5, the four-block pass 615 -> 564 us with the split; 500
// tokens 1.2e-3 -> 1.7e-4 for 1% of the pass).

constexpr int PA_ROWS = 64;
constexpr int PA_THREADS = 128;
constexpr int PA_MAX_SPLIT = 8;  // CTAs of a key-split cluster

__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int HD>
struct PaLayout {
  static constexpr int ROW = (HD + 8) * 2;  // bytes per padded row
  static constexpr int TILE = PA_ROWS * ROW;
  static constexpr int Q_OFF = 0;
  static constexpr int K_OFF = TILE;          // 2 buffers
  static constexpr int V_OFF = 3 * TILE;      // 2 buffers
  static constexpr int POS_OFF = 5 * TILE;    // int [64]
  static constexpr int ML_OFF = POS_OFF + PA_ROWS * 4;  // float (m, l) [64]
  static constexpr int BYTES = ML_OFF + PA_ROWS * 8;
  // after the key loop, where K and V were: this CTA's O [64][O_LD] for its cluster
  static constexpr int O_LD = HD + 4;
  static_assert(PA_ROWS * O_LD * 4 <= 4 * TILE, "O fits where K and V were");
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_cluster_f2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}

// Two values as packed pairs of bf16 (rounded) and of what rounding left (bf16 again).
__device__ __forceinline__ void pair_bf16(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  hi = pack_bf16(x0, x1);
  lo = pack_bf16(x0 - bf16_lo(hi), x1 - bf16_hi(hi));
}

// Rows [r0, r0 + 64) of a [rows][HD] bf16 matrix (row stride ld elements) into a padded tile;
// rows at or above `limit` are zero.
template <int HD>
__device__ __forceinline__ void pa_load_tile(uint8_t *tile, const uint16_t *src, size_t ld, int r0, int limit) {
  constexpr int CH = HD / 8;
  for (int e = threadIdx.x; e < PA_ROWS * CH; e += PA_THREADS) {
    const int r = e / CH, ch = e % CH;
    uint8_t *dst = tile + r * PaLayout<HD>::ROW + ch * 16;
    if (r0 + r < limit)
      cp_async16(smem_addr(dst), src + (size_t)(r0 + r) * ld + ch * 8);
    else
      *reinterpret_cast<uint4 *>(dst) = make_uint4(0, 0, 0, 0);
  }
}

// Two consecutive output elements as the O projection's input terms.
__device__ __forceinline__ void store_terms(const PrefillAttnParams &p, size_t at, float x0, float x1) {
  uint32_t hi, lo;
  split_pack(x0, x1, hi, lo, p.f16, p.err);
  *reinterpret_cast<uint32_t *>(p.o + at) = hi;
  *reinterpret_cast<uint32_t *>(p.o + p.term_stride + at) = lo;
  if (p.terms == 3) {  // bf16 terms: what the first two leave
    const float r0 = x0 - bf16_lo(hi) - bf16_lo(lo), r1 = x1 - bf16_hi(hi) - bf16_hi(lo);
    *reinterpret_cast<uint32_t *>(p.o + 2 * p.term_stride + at) = pack_bf16(r0, r1);
  }
}

template <int HD, bool PRECISE>
__global__ void __launch_bounds__(PA_THREADS) prefill_attn_kernel(PrefillAttnParams p) {
  using L = PaLayout<HD>;
  extern __shared__ __align__(16) uint8_t sm[];
  pdl_launch_dependents();
  pdl_wait();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int g = lane / 4, c = lane % 4;
  // the longest blocks (latest tokens) first
  const int qb = gridDim.x - 1 - blockIdx.x;
  const int h = blockIdx.y, kvh = h / (p.n_heads / p.n_kv_heads);
  const int rank = blockIdx.z, n_split = gridDim.z;
  const int t0 = qb * PA_ROWS;
  int *s_pos = reinterpret_cast<int *>(sm + L::POS_OFF);
  if (threadIdx.x < PA_ROWS) s_pos[threadIdx.x] = t0 + threadIdx.x < p.T ? p.positions[t0 + threadIdx.x] : -1;
  if constexpr (!PRECISE) pa_load_tile<HD>(sm + L::Q_OFF, p.q + h * HD, p.ldq, t0, p.T);
  cp_async_commit();
  __syncthreads();
  int max_pos = -1;
  for (int i = 0; i < PA_ROWS; ++i) max_pos = max(max_pos, s_pos[i]);
  const int n_all = (max_pos + PA_ROWS) / PA_ROWS;  // key blocks covering [0, max_pos]
  const int kb0 = rank * n_all / n_split, n_kb = (rank + 1) * n_all / n_split;  // this CTA's: [kb0, n_kb)
  const int kv_limit = min(max_pos + 1, p.max_ctx);
  const size_t head_base = ((size_t)p.slot * p.n_kv_heads + kvh) * p.max_ctx * HD;
  const uint16_t *kg = p.kcache + head_base, *vg = p.vcache + head_base;
  if (kb0 < n_kb) {
    pa_load_tile<HD>(sm + L::K_OFF, kg, HD, kb0 * PA_ROWS, kv_limit);
    pa_load_tile<HD>(sm + L::V_OFF, vg, HD, kb0 * PA_ROWS, kv_limit);
  }
  cp_async_commit();
  const int qp0 = s_pos[16 * warp + g], qp1 = s_pos[16 * warp + g + 8];
  // Q fragments of this warp's 16 rows
  uint32_t qf[HD / 16][4], ql[PRECISE ? HD / 16 : 1][4];
  if constexpr (PRECISE) {
    const int ra = t0 + 16 * warp + g, rb = ra + 8;
    const float *qa = p.q32 + (size_t)min(ra, p.T - 1) * p.ldq + h * HD, *qr = p.q32 + (size_t)min(rb, p.T - 1) * p.ldq + h * HD;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk)
#pragma unroll
      for (int j = 0; j < 4; ++j) {  // rows g, g + 8; columns 2c, 2c + 1 then + 8
        const float2 v = *reinterpret_cast<const float2 *>((j & 1 ? qr : qa) + kk * 16 + 2 * c + (j & 2 ? 8 : 0));
        pair_bf16(v.x, v.y, qf[kk][j], ql[kk][j]);
      }
  }
  cp_async_wait_all();
  __syncthreads();
  if constexpr (!PRECISE) {
    const uint32_t qbase = smem_addr(sm + L::Q_OFF) + (16 * warp + (lane % 16)) * L::ROW + (lane / 16) * 16;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) ldsm_x4(qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3], qbase + kk * 32);
  }
  float oacc[HD / 8][4] = {};
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  for (int kb = kb0; kb < n_kb; ++kb) {
    const int buf = (kb - kb0) & 1;
    if (kb + 1 < n_kb) {  // the next block loads while this one is used
      pa_load_tile<HD>(sm + L::K_OFF + (buf ^ 1) * L::TILE, kg, HD, (kb + 1) * PA_ROWS, kv_limit);
      pa_load_tile<HD>(sm + L::V_OFF + (buf ^ 1) * L::TILE, vg, HD, (kb + 1) * PA_ROWS, kv_limit);
    }
    cp_async_commit();
    const uint32_t kbase = smem_addr(sm + L::K_OFF + buf * L::TILE);
    const uint32_t vbase = smem_addr(sm + L::V_OFF + buf * L::TILE);
    // S = Q K^T: 8 key tiles of 8.  Four tiles' fragments are loaded before their MMAs: a warp issues in
    // order, and a load behind each pair of MMAs stood for its latency (2048 tokens, 28 heads: 196 ->
    // 180 us with P V's the same way; the pairs' registers leave no room for it)
    float s[8][4] = {};
    if constexpr (PRECISE) {
#pragma unroll
      for (int nt = 0; nt < 8; ++nt)
#pragma unroll
        for (int kk = 0; kk < HD / 16; kk += 2) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4(b0, b1, b2, b3, kbase + (nt * 8 + (lane % 8)) * L::ROW + kk * 32 + (lane / 8) * 16);
          mma16816(s[nt], qf[kk][0], qf[kk][1], qf[kk][2], qf[kk][3], b0, b1);
          mma16816(s[nt], qf[kk + 1][0], qf[kk + 1][1], qf[kk + 1][2], qf[kk + 1][3], b2, b3);
          mma16816(s[nt], ql[kk][0], ql[kk][1], ql[kk][2], ql[kk][3], b0, b1);
          mma16816(s[nt], ql[kk + 1][0], ql[kk + 1][1], ql[kk + 1][2], ql[kk + 1][3], b2, b3);
        }
    } else {
#pragma unroll
      for (int kk = 0; kk < HD / 16; kk += 2)
#pragma unroll
        for (int n0 = 0; n0 < 8; n0 += 4) {
          uint32_t b[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            ldsm_x4(b[i][0], b[i][1], b[i][2], b[i][3],
                    kbase + ((n0 + i) * 8 + (lane % 8)) * L::ROW + kk * 32 + (lane / 8) * 16);
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              mma16816(s[n0 + i], qf[kk + h2][0], qf[kk + h2][1], qf[kk + h2][2], qf[kk + h2][3], b[i][2 * h2],
                       b[i][2 * h2 + 1]);
        }
    }
    // scale, causal mask, online softmax (rows g and g + 8 of the warp)
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int kp = kb * PA_ROWS + nt * 8 + 2 * c;
      s[nt][0] = kp <= qp0 ? s[nt][0] * p.scale_log2 : -INFINITY;
      s[nt][1] = kp + 1 <= qp0 ? s[nt][1] * p.scale_log2 : -INFINITY;
      s[nt][2] = kp <= qp1 ? s[nt][2] * p.scale_log2 : -INFINITY;
      s[nt][3] = kp + 1 <= qp1 ? s[nt][3] * p.scale_log2 : -INFINITY;
      mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][1]));
      mx1 = fmaxf(mx1, fmaxf(s[nt][2], s[nt][3]));
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
    // rows with no visible key yet keep m = -inf; their factors stay 0 / 1
    const float base0 = mn0 == -INFINITY ? 0.f : mn0, base1 = mn1 == -INFINITY ? 0.f : mn1;
    const float corr0 = exp2f(m0 - base0), corr1 = exp2f(m1 - base1);
    m0 = mn0;
    m1 = mn1;
    float rs0 = 0.f, rs1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      s[nt][0] = exp2f(s[nt][0] - base0);
      s[nt][1] = exp2f(s[nt][1] - base0);
      s[nt][2] = exp2f(s[nt][2] - base1);
      s[nt][3] = exp2f(s[nt][3] - base1);
      rs0 += s[nt][0] + s[nt][1];
      rs1 += s[nt][2] + s[nt][3];
    }
    l0 = l0 * corr0 + rs0;
    l1 = l1 * corr1 + rs1;
    // O = O corr + P V: 4 key steps of 16; V fragments by transposed matrix loads
    const uint32_t vlane = vbase + ((lane % 8) + ((lane / 8) & 1) * 8) * L::ROW + (lane / 16) * 16;
    if constexpr (PRECISE) {
      // a block's products from zero, added to O in fp32: tensor-core accumulation truncates, and over
      // thousands of keys that would show (see prefill_narrow_kernel)
      uint32_t a[4][4], e[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) pair_bf16(s[2 * j + i / 2][2 * (i & 1)], s[2 * j + i / 2][2 * (i & 1) + 1], a[j][i], e[j][i]);
#pragma unroll
      for (int dt = 0; dt < HD / 8; dt += 2) {
        float y[2][4] = {};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4_t(b0, b1, b2, b3, vlane + j * 16 * L::ROW + dt * 16);
          mma16816(y[0], e[j][0], e[j][1], e[j][2], e[j][3], b0, b1);
          mma16816(y[1], e[j][0], e[j][1], e[j][2], e[j][3], b2, b3);
          mma16816(y[0], a[j][0], a[j][1], a[j][2], a[j][3], b0, b1);
          mma16816(y[1], a[j][0], a[j][1], a[j][2], a[j][3], b2, b3);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          oacc[dt + i][0] = oacc[dt + i][0] * corr0 + y[i][0];
          oacc[dt + i][1] = oacc[dt + i][1] * corr0 + y[i][1];
          oacc[dt + i][2] = oacc[dt + i][2] * corr1 + y[i][2];
          oacc[dt + i][3] = oacc[dt + i][3] * corr1 + y[i][3];
        }
      }
    } else {
#pragma unroll
      for (int dt = 0; dt < HD / 8; ++dt) {
        oacc[dt][0] *= corr0;
        oacc[dt][1] *= corr0;
        oacc[dt][2] *= corr1;
        oacc[dt][3] *= corr1;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t a0 = pack_bf16(s[2 * j][0], s[2 * j][1]), a1 = pack_bf16(s[2 * j][2], s[2 * j][3]);
        const uint32_t a2 = pack_bf16(s[2 * j + 1][0], s[2 * j + 1][1]), a3 = pack_bf16(s[2 * j + 1][2], s[2 * j + 1][3]);
#pragma unroll
        for (int d0 = 0; d0 < HD / 8; d0 += 8) {
          uint32_t b[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            ldsm_x4_t(b[i][0], b[i][1], b[i][2], b[i][3], vlane + j * 16 * L::ROW + (d0 + 2 * i) * 16);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            mma16816(oacc[d0 + 2 * i], a0, a1, a2, a3, b[i][0], b[i][1]);
            mma16816(oacc[d0 + 2 * i + 1], a0, a1, a2, a3, b[i][2], b[i][3]);
          }
        }
      }
    }
    cp_async_wait_all();
    __syncthreads();
  }
  // row sums over the quad
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
  l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  if (n_split > 1) {
    // this CTA's state for the cluster; every warp is past its last key block (the loop ends in a barrier)
    float *so = reinterpret_cast<float *>(sm + L::K_OFF);
    float2 *sml = reinterpret_cast<float2 *>(sm + L::ML_OFF);
    const int r = 16 * warp + g;
#pragma unroll
    for (int dt = 0; dt < HD / 8; ++dt) {
      *reinterpret_cast<float2 *>(so + r * L::O_LD + dt * 8 + 2 * c) = make_float2(oacc[dt][0], oacc[dt][1]);
      *reinterpret_cast<float2 *>(so + (r + 8) * L::O_LD + dt * 8 + 2 * c) = make_float2(oacc[dt][2], oacc[dt][3]);
    }
    if (c == 0) {
      sml[r] = make_float2(m0, l0);
      sml[r + 8] = make_float2(m1, l1);
    }
    cluster_sync_all();
    // rank k merges rows [k 64 / n, (k + 1) 64 / n), four columns per thread and step
    const int rows = PA_ROWS / n_split;
    for (int e = threadIdx.x; e < rows * (HD / 4); e += PA_THREADS) {
      const int row = rank * rows + e / (HD / 4), col = e % (HD / 4) * 4, t = t0 + row;
      float2 ml[PA_MAX_SPLIT];
      float4 o[PA_MAX_SPLIT];
#pragma unroll
      for (int k = 0; k < PA_MAX_SPLIT; ++k)
        if (k < n_split) {
          ml[k] = ld_cluster_f2(map_to_rank(smem_addr(sml + row), k));
          o[k] = ld_cluster_f4(map_to_rank(smem_addr(so + row * L::O_LD + col), k));
        }
      float m = -INFINITY;
#pragma unroll
      for (int k = 0; k < PA_MAX_SPLIT; ++k)
        if (k < n_split) m = fmaxf(m, ml[k].x);
      float l = 0.f, y[4] = {};
#pragma unroll
      for (int k = 0; k < PA_MAX_SPLIT; ++k)
        if (k < n_split && ml[k].y != 0.f) {  // (a CTA that saw a key: m stays -inf, l is NaN where all were NaN)
          const float w = exp2f(ml[k].x - m);
          l += ml[k].y * w;
          y[0] += o[k].x * w;
          y[1] += o[k].y * w;
          y[2] += o[k].z * w;
          y[3] += o[k].w * w;
        }
      const float inv = l > 0.f ? 1.f / l : 0.f;
      if (t < p.T) {
        store_terms(p, (size_t)t * p.ldo + h * HD + col, y[0] * inv, y[1] * inv);
        store_terms(p, (size_t)t * p.ldo + h * HD + col + 2, y[2] * inv, y[3] * inv);
      }
    }
    cluster_sync_all();  // no CTA leaves while others read its shared memory
    return;
  }
  const float inv0 = l0 > 0.f ? 1.f / l0 : 0.f, inv1 = l1 > 0.f ? 1.f / l1 : 0.f;
  const int ta = t0 + 16 * warp + g, tb = ta + 8;
#pragma unroll
  for (int dt = 0; dt < HD / 8; ++dt) {
    const int col = h * HD + dt * 8 + 2 * c;
    if (ta < p.T) store_terms(p, (size_t)ta * p.ldo + col, oacc[dt][0] * inv0, oacc[dt][1] * inv0);
    if (tb < p.T) store_terms(p, (size_t)tb * p.ldo + col, oacc[dt][2] * inv1, oacc[dt][3] * inv1);
  }
}

// ---------------------------------------------------------------------------- small kernels
// One block per prompt token: its input row (embedding row or given hidden state) and its
// position, refused (-1, ERR_POSITION) outside [0, max_ctx) or when an earlier token of the pass
// holds the same position.
__global__ void prefill_input_kernel(const int *ids, const float *hidden_in, const int *positions_in, int T,
                                     const uint16_t *embed, int vocab, int d, int ldh, float *h, int *positions,
                                     int max_ctx, int user, int *slots, unsigned *err) {
  const int t = blockIdx.x;
  pdl_launch_dependents();
  if (slots && threadIdx.x == 0) slots[t] = user;
  int id = embed ? ids[t] : 0;
  if (embed && (id < 0 || id >= vocab)) {
    if (threadIdx.x == 0) atomicOr(err, ERR_TOKEN);
    id = 0;
  }
  // eight elements and eight earlier positions in flight per thread: one at a time, the kernel was its
  // loads' latency (100 tokens x 8192, cold: 18.1 -> 5.6 us; 2048 x 3584: 18.9 -> 10.9)
  float *row = h + (size_t)t * ldh;
  for (int i0 = threadIdx.x; i0 < d; i0 += 8 * blockDim.x) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + j * blockDim.x;
      if (i < d) v[j] = embed ? bf16_to_f32(embed[(size_t)id * d + i]) : hidden_in[(size_t)t * d + i];
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (i0 + j * (int)blockDim.x < d) row[i0 + j * blockDim.x] = v[j];
  }
  const int pos = positions_in[t];
  int bad = 0;
#pragma unroll 8
  for (int j = threadIdx.x; j < t; j += blockDim.x) bad |= positions_in[j] == pos;
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    const bool ok = pos >= 0 && pos < max_ctx && !bad;
    if (!ok) atomicOr(err, ERR_POSITION);
    positions[t] = ok ? pos : -1;
  }
}

// x[t] = h[t] / rms(h[t]) * g as two or three 16-bit terms (term_stride elements apart), one block per
// token, four elements per thread step (d a multiple of 8; h, g and x rows 16-byte aligned).  Bound
// by latency: a thread's first RN_V groups of h and g are loaded at once and kept (2048 x 3584:
// 13.9 us, 4.2 TB/s; 17.8 one group at a time, read twice).  A block has no more threads than those
// groups need, but 64: at d 320, 256 threads with their registers for all four made 2048 tokens' two norms
// of a block 13 us longer.
constexpr int RN_V = 4;
__global__ void prefill_rmsnorm_kernel(const float *h, int ldh, int d, const float *g, float eps, uint16_t *x,
                                       size_t term_stride, int terms, int ldx, int f16, unsigned *err) {
  const int t = blockIdx.x, d4 = d / 4;
  pdl_launch_dependents();
  const float4 *g4 = reinterpret_cast<const float4 *>(g);
  float4 v[RN_V], gg[RN_V];
#pragma unroll
  for (int j = 0; j < RN_V; ++j) {
    const int i = threadIdx.x + j * blockDim.x;
    if (i < d4) gg[j] = g4[i];
  }
  pdl_wait();
  const float4 *row = reinterpret_cast<const float4 *>(h + (size_t)t * ldh);
#pragma unroll
  for (int j = 0; j < RN_V; ++j) {
    const int i = threadIdx.x + j * blockDim.x;
    v[j] = i < d4 ? row[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < RN_V; ++j) ss += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
  for (int i = threadIdx.x + RN_V * blockDim.x; i < d4; i += blockDim.x) {
    const float4 a = row[i];
    ss += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
  }
  __shared__ float red[32];
  const float inv = 1.0f / sqrtf(block_sum(ss, red) / d + eps);
  uint16_t *xt = x + (size_t)t * ldx;
#pragma unroll
  for (int j = 0; j < RN_V; ++j) {
    const int i = threadIdx.x + j * blockDim.x;
    if (i < d4) store_normed(v[j], inv, gg[j], xt + 4 * i, term_stride, terms, f16, err);
  }
  for (int i = threadIdx.x + RN_V * blockDim.x; i < d4; i += blockDim.x)
    store_normed(row[i], inv, g4[i], xt + 4 * i, term_stride, terms, f16, err);
}

// Half an int4 tile (64 rows x 128 columns) to its fp16 tile, code x scale rounded once (decode_word,
// scale_pair): warp r16 decodes 16 rows, in the fragment order of the codes, into shared memory by
// matrix stores, and the block writes the 16 KiB tile out in 16-byte pieces.  Bound by HBM: 0.53 bytes
// read and 2 written per weight.  (One thread per 8 outputs, gathering the codes word by word and
// rounding each product on its own, ran at 2.9 TB/s: a 72B-shaped block of 900 tokens 2940 -> 2389 us.)
constexpr int DQ_ROW = KT * 2 + 16;  // bytes per staged row: eight rows' pieces fall on distinct banks
__global__ void __launch_bounds__(128) dequant_int4_f16_kernel(const uint8_t *tiles4, int n_tiles, uint16_t *dst) {
  __shared__ __align__(16) uint8_t stage[RB * DQ_ROW];
  const int r16 = threadIdx.x / 32, lane = threadIdx.x % 32, gid = lane >> 2;
  // matrices 0..3 of a 16-column step: rows 0-7 and 8-15 of its first 8 columns, then of its last 8
  const uint32_t st = smem_addr(stage) + (r16 * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * DQ_ROW + (lane >> 4) * 16;
  for (int h = blockIdx.x; h < 2 * n_tiles; h += gridDim.x) {
    const uint8_t *tile = tiles4 + (size_t)(h >> 1) * TILE4_BYTES;
    uint4 w[2];
    uint32_t sc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      w[q] = __ldcs(reinterpret_cast<const uint4 *>(tile + (h & 1) * 4096 + r16 * 1024 + q * 512) + lane);
      sc[q] = *reinterpret_cast<const uint32_t *>(tile + TILE4_CODE_BYTES +
                                                  2 * tile4_scale_index(r16 * 16 + gid, 2 * (h & 1) + q));
    }
    __syncthreads();  // the stage is free
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const ScalePair sp(sc[q]);
      const bool exact = __all_sync(0xffffffffu, sp.exact());
      const uint32_t words[4] = {w[q].x, w[q].y, w[q].z, w[q].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t c0, c1, c2, c3;
        decode_word(words[j], c0, c1, c2, c3);
        sp.apply(exact, c0, c1, c2, c3);
        stsm_x4(st + q * 128 + j * 32, c0, c1, c2, c3);
      }
    }
    __syncthreads();
    uint4 *out = reinterpret_cast<uint4 *>(dst + (size_t)h * RB * KT);  // fp16 tile (rb, 2 kt + half)
#pragma unroll
    for (int e = threadIdx.x; e < RB * KT / 8; e += 128)
      __stcs(out + e, *reinterpret_cast<const uint4 *>(stage + (e / (KT / 8)) * DQ_ROW + (e % (KT / 8)) * 16));
  }
}

// fp32 rows [T][K] (stride ldx) -> hi and lo bf16 terms (stride ld), 1024 columns to a block; *err = 0.
__global__ void __launch_bounds__(256) split_rows_kernel(const float *x, int K, int ldx, uint16_t *hi, uint16_t *lo,
                                                         int ld, unsigned *err) {
  pdl_launch_dependents();
  const int t = blockIdx.y, i0 = blockIdx.x * 1024 + threadIdx.x;
  if (t == 0 && i0 == 0) *err = 0;
  float v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = i0 + 256 * j < K ? x[(size_t)t * ldx + i0 + 256 * j] : 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (i0 + 256 * j < K) split_bf16(v[j], hi[(size_t)t * ld + i0 + 256 * j], lo[(size_t)t * ld + i0 + 256 * j]);
}

// A row-major matrix [N][K] whose rows TMA cannot address as weight tiles [n_rb][n_kt][RB][KT]
// (zero-padded), one block per tile: each thread has 32 two-byte loads in flight.  (The loaders' repack
// kernel, a thread per 16 bytes over a fixed grid with 64-bit index arithmetic, took 110 us for 233 MB.)
__global__ void __launch_bounds__(256) tile_rows_kernel(const uint16_t *w, int N, int K, int n_kt, uint8_t *dst) {
  const int rb = blockIdx.x / n_kt, kt = blockIdx.x - rb * n_kt;
  const int ch = threadIdx.x % (KT / 8), r0 = threadIdx.x / (KT / 8), k0 = kt * KT + ch * 8;
  uint16_t v[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = rb * RB + r0 + 16 * i;
#pragma unroll
    for (int j = 0; j < 8; ++j) v[i][j] = r < N && k0 + j < K ? w[(size_t)r * K + k0 + j] : uint16_t(0);
  }
  uint4 *tile = reinterpret_cast<uint4 *>(dst + (size_t)blockIdx.x * TILE_BYTES);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    tile[(r0 + 16 * i) * (KT / 8) + ch] =
        make_uint4(v[i][0] | (uint32_t)v[i][1] << 16, v[i][2] | (uint32_t)v[i][3] << 16, v[i][4] | (uint32_t)v[i][5] << 16,
                   v[i][6] | (uint32_t)v[i][7] << 16);
}

// next_ids[t]: the lowest index among the largest logits, over the column tiles' partial maxima;
// one warp per token (each lane scans every 32nd tile, then the warp keeps the largest value and,
// among equal values, the lowest index).
__global__ void prefill_argmax_kernel(const float *amax, const int *aidx, int n_tiles, int T, int *next_ids) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (t >= T) return;  // uniform per warp
  float best = -INFINITY;
  int bi = 0x7FFFFFFF;
  for (int j = lane; j < n_tiles; j += 32) {
    const float v = amax[(size_t)t * n_tiles + j];
    const int i = aidx[(size_t)t * n_tiles + j];
    if (v > best || (v == best && i < bi)) {
      best = v;
      bi = i;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) {
      best = ov;
      bi = oi;
    }
  }
  if (lane == 0) next_ids[t] = bi == 0x7FFFFFFF ? 0 : bi;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> found{nullptr};
  PFN_cuTensorMapEncodeTiled_v12000 fn = found.load();
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      found = fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    else
      cudaGetLastError();
  }
  return fn;
}

}  // namespace

// ---------------------------------------------------------------------------- host side
// Activation rows [rows][K] bf16 at row stride ld (a multiple of 8): boxes of 64 columns x PG_M
// rows; columns >= K and rows >= rows read as zero.
int encode_act_map(CUtensorMap *map, const uint16_t *base, int K, int rows, int ld) {
  auto fn = encode_fn();
  if (!fn || ld % 8 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return -1;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {PG_K, PG_M};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -1;
}

int encode_terms_map(CUtensorMap *map, const uint16_t *base, int K, int rows, int ld, int terms, size_t term_stride,
                     int box_rows) {
  auto fn = encode_fn();
  if (!fn || ld % 8 != 0 || term_stride % 8 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return -1;
  const cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)terms};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)term_stride * 2};
  const cuuint32_t box[3] = {PG_K, (cuuint32_t)box_rows, (cuuint32_t)terms};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -1;
}

int encode_rows_map(CUtensorMap *map, const uint16_t *w, int K, int N, int box_rows) {
  auto fn = encode_fn();
  if (!fn || K % 8 != 0 || (reinterpret_cast<uintptr_t>(w) & 15) != 0) return -1;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)N};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {PG_K, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(w), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -1;
}

// Weight tiles [n_rb][n_kt][RB][KT] bf16 as a 4-D tensor (column, row, K tile, row block):
// boxes of 64 columns x RB rows x 1 K tile x box_rb row blocks; row blocks >= n_rb read as zero.
int encode_tiles_map(CUtensorMap *map, const uint8_t *tiles, int n_kt, int n_rb, int box_rb) {
  auto fn = encode_fn();
  if (!fn) return -1;
  const cuuint64_t dims[4] = {(cuuint64_t)KT, (cuuint64_t)RB, (cuuint64_t)n_kt, (cuuint64_t)n_rb};
  const cuuint64_t strides[3] = {(cuuint64_t)KT * 2, (cuuint64_t)TILE_BYTES, (cuuint64_t)TILE_BYTES * n_kt};
  const cuuint32_t box[4] = {PG_K, RB, 1, (cuuint32_t)box_rb};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint8_t *>(tiles), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? 0
             : -1;
}

// Launches a kernel that waits for the kernel before it only where it needs its results.
template <typename... P, typename... A>
static cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int MODE>
static cudaError_t launch_mode(const CUtensorMap &a, const CUtensorMap &a2, const CUtensorMap &b, bool w_rows, int n_kb,
                               const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s) {
  constexpr bool DRAIN = MODE == PE_STORE;
  static SmemOptIn opt_in;
  cudaError_t e = opt_in(reinterpret_cast<const void *>(prefill_gemm_persistent<MODE, DRAIN>), (int)PG_SMEM);
  if (e != cudaSuccess) return e;
  // one persistent CTA per SM (fewer if there are not four K blocks for each)
  const int tiles = (ep.T + PG_M - 1) / PG_M * ((ep.N + PG_N - 1) / PG_N);
  const int grid = (int)std::min<long long>(ws.n_sm, std::max<long long>(std::min(tiles, ws.n_sm), (long long)tiles * n_kb / 4));
  const TileShare share = share_tiles(tiles, n_kb, grid, false, NW_PARTS);
  e = launch_pdl(prefill_gemm_persistent<MODE, DRAIN>, dim3(grid), pp_threads(DRAIN), PG_SMEM, s, a, a2, b, (int)w_rows,
                 share, ws.partial, ep);
  if (e == cudaSuccess && share.cut())
    e = launch_pdl(wide_reduce_kernel<MODE>, dim3(share.tail * (MODE == PE_ARGMAX ? 1 : PG_N / 32)), PG_M, 0, s, share,
                   grid, ws.partial, ep);
  return e;
}

cudaError_t launch_prefill_gemm(int mode, const CUtensorMap &a, const CUtensorMap &a2, const CUtensorMap &b,
                                bool w_rows, int K, const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s) {
  if (ep.T <= 0 || ep.N <= 0) return cudaSuccess;
  const int n_kb = (K + PG_K - 1) / PG_K;
  switch (mode) {
    case PE_STORE: return launch_mode<PE_STORE>(a, a2, b, w_rows, n_kb, ws, ep, s);
    case PE_RESID: return launch_mode<PE_RESID>(a, a2, b, w_rows, n_kb, ws, ep, s);
    case PE_SWIGLU: return launch_mode<PE_SWIGLU>(a, a2, b, w_rows, n_kb, ws, ep, s);
    case PE_QKV: return launch_mode<PE_QKV>(a, a2, b, w_rows, n_kb, ws, ep, s);
    case PE_ARGMAX: return launch_mode<PE_ARGMAX>(a, a2, b, w_rows, n_kb, ws, ep, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int HD, bool PRECISE>
static cudaError_t launch_attn_hd(const PrefillAttnParams &p, int n_sm, cudaStream_t s) {
  static SmemOptIn opt_in;
  const int bytes = PaLayout<HD>::BYTES;
  const cudaError_t e = opt_in(reinterpret_cast<const void *>(prefill_attn_kernel<HD, PRECISE>), bytes);
  if (e != cudaSuccess) return e;
  // split the keys until about two CTAs per SM (as many as fit) have work
  const int blocks = (p.T + PA_ROWS - 1) / PA_ROWS * p.n_heads;
  int split = 1;
  while (split < PA_MAX_SPLIT && blocks * split * 2 <= 2 * n_sm) split *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((p.T + PA_ROWS - 1) / PA_ROWS, p.n_heads, split);
  cfg.blockDim = dim3(PA_THREADS);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  pdl_attribute(at[0]);
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = split;
  cfg.attrs = at;
  cfg.numAttrs = split > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, prefill_attn_kernel<HD, PRECISE>, p);
}

cudaError_t launch_prefill_attention(const PrefillAttnParams &p, int hd, int n_sm, cudaStream_t s) {
  if (p.T <= 0) return cudaSuccess;
  if (p.q32) return hd == 128 ? launch_attn_hd<128, true>(p, n_sm, s) : launch_attn_hd<64, true>(p, n_sm, s);
  return hd == 128 ? launch_attn_hd<128, false>(p, n_sm, s) : launch_attn_hd<64, false>(p, n_sm, s);
}

cudaError_t launch_prefill_input(const int *ids, const float *hidden_in, const int *positions_in, int T,
                                 const uint16_t *embed, int vocab, int d, int ldh, float *h, int *positions,
                                 int max_ctx, int user, int *slots, unsigned *err, cudaStream_t s) {
  prefill_input_kernel<<<T, 256, 0, s>>>(ids, hidden_in, positions_in, T, embed, vocab, d, ldh, h, positions,
                                         max_ctx, user, slots, err);
  return cudaGetLastError();
}

cudaError_t launch_prefill_rmsnorm(const float *h, int ldh, int T, int d, const float *g, float eps, uint16_t *x,
                                   size_t term_stride, int terms, int ldx, int f16, unsigned *err, cudaStream_t s) {
  int threads = 64;
  while (threads < 1024 && threads * 4 * RN_V < d) threads *= 2;
  return launch_pdl(prefill_rmsnorm_kernel, dim3(T), threads, 0, s, h, ldh, d, g, eps, x, term_stride, terms, ldx, f16, err);
}

cudaError_t launch_dequant_int4_f16(const uint8_t *tiles4, int n_rb, int n_kt, uint16_t *dst, int n_sm,
                                    cudaStream_t s) {
  dequant_int4_f16_kernel<<<8 * n_sm, 128, 0, s>>>(tiles4, n_rb * n_kt, dst);
  return cudaGetLastError();
}

cudaError_t launch_split_bf16(const float *x, int T, int K, int ldx, uint16_t *hi, uint16_t *lo, int ld, unsigned *err,
                              cudaStream_t s) {
  for (int t0 = 0; t0 < T; t0 += 65535) {  // the grid's y limit
    const int n = std::min(65535, T - t0);
    split_rows_kernel<<<dim3((K + 1023) / 1024, n), 256, 0, s>>>(x + (size_t)t0 * ldx, K, ldx, hi + (size_t)t0 * ld,
                                                               lo + (size_t)t0 * ld, ld, err);
  }
  return cudaGetLastError();
}

cudaError_t launch_prefill_argmax(const float *amax, const int *aidx, int n_tiles, int T, int *next_ids,
                                  cudaStream_t s) {
  return launch_pdl(prefill_argmax_kernel, dim3((T + 3) / 4), 128, 0, s, amax, aidx, n_tiles, T, next_ids);
}

}  // namespace kfl

// ---------------------------------------------------------------------------- C ABI
namespace {

// The device's memory pool for kfl_matmul_bf16w's temporary buffers, made at its first call there.  Of
// what the calls free, the pool keeps up to MATMUL_KEEP_BYTES for the next and returns the rest at
// their synchronisation.  A cudaMalloc and cudaFree per call cost 80 to 250 us, and what the pool has to
// return at once costs more (613 MB: 1.2 ms of a 1.8 ms call), so that buffers beyond its bound, which only
// more than some 4000 tokens of a K of 18944 need, are allocated by themselves.
// Calls on several threads and streams each take buffers of their own from it.
constexpr uint64_t MATMUL_KEEP_BYTES = 512ull << 20;
constexpr uint64_t MATMUL_SLAB_BYTES = 128ull << 20;  // a copy of weight tiles may always have this much
constexpr int MATMUL_MAX_DEVICES = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[MATMUL_MAX_DEVICES] = {};

cudaMemPool_t matmul_pool(int dev) {
  if (dev < 0 || dev >= MATMUL_MAX_DEVICES) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = MATMUL_KEEP_BYTES;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaGetLastError();
      if (pool) cudaMemPoolDestroy(pool);
      return nullptr;
    }
    g_pool[dev] = pool;
  }
  return g_pool[dev];
}

}  // namespace

namespace kfl {
// Returns what the current device's pool keeps.
static bool release_matmul_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MATMUL_MAX_DEVICES) return false;
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  return g_pool[dev] && cudaMemPoolTrimTo(g_pool[dev], 0) == cudaSuccess;
}

bool device_alloc(void **p, size_t bytes) {
  if (cudaMalloc(p, bytes) == cudaSuccess) return true;
  cudaGetLastError();
  if (release_matmul_pool() && cudaMalloc(p, bytes) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}
}  // namespace kfl

extern "C" int kfl_matmul_bf16w(const float *x, int T, int K, int ldx, const uint16_t *w, int N, float *y, int ldy,
                                void *cuda_stream) {
  using namespace kfl;
  if (!x || !w || !y || T < 1 || K < 1 || N < 1 || ldx < K || ldy < N || ldy % 4 != 0 ||
      (reinterpret_cast<uintptr_t>(y) & 15) != 0)
    return KFL_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int n_kt = (K + KT - 1) / KT, ld = (K + 63) / 64 * 64;
  int dev = 0, n_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return KFL_ERR_CUDA;
  }
  // few tokens: the few-token kernel.  A matrix whose rows TMA can address is read where it is; others
  // (K not a multiple of 8, or an unaligned start) are copied into weight tiles first
  const bool narrow = T <= NW_MAX_TP, w_rows = K % 8 == 0 && (reinterpret_cast<uintptr_t>(w) & 15) == 0;
  const int rows = (T + 7) / 8 * 8;
  const size_t x_bytes = (size_t)rows * ld * 2, ws_bytes = narrow_ws_bytes(n_sm, T), fixed = 2 * x_bytes + ws_bytes + 16;
  // a copied matrix goes a slab of rows at a time through what the pool may keep
  int slab = N;
  if (!w_rows) {
    const size_t room = fixed + MATMUL_SLAB_BYTES <= MATMUL_KEEP_BYTES ? MATMUL_KEEP_BYTES - fixed : MATMUL_SLAB_BYTES;
    const size_t most = std::max<size_t>(room / ((size_t)n_kt * KT * 2) / PG_N, 1) * PG_N;
    slab = (int)std::min<size_t>(N, most);
  }
  const size_t tile_bytes = w_rows ? 0 : (size_t)((slab + RB - 1) / RB) * n_kt * TILE_BYTES, bytes = tile_bytes + fixed;
  const bool pooled = bytes <= MATMUL_KEEP_BYTES;
  void *mem = nullptr;
  if (pooled) {
    cudaMemPool_t pool = matmul_pool(dev);
    if (!pool || cudaMallocFromPoolAsync(&mem, bytes, pool, s) != cudaSuccess) {
      cudaGetLastError();
      return KFL_ERR_OOM;
    }
  } else if (!device_alloc(&mem, bytes)) {
    return KFL_ERR_OOM;
  }
  uint8_t *tiles = static_cast<uint8_t *>(mem);
  uint16_t *xhi = reinterpret_cast<uint16_t *>(tiles + tile_bytes);
  uint16_t *xlo = xhi + (size_t)rows * ld;
  float *partial = reinterpret_cast<float *>(xlo + (size_t)rows * ld);
  unsigned *err = reinterpret_cast<unsigned *>(reinterpret_cast<uint8_t *>(partial) + ws_bytes);
  int rc = KFL_OK;
  unsigned h_err = 0;
  CUtensorMap mh, ml, mb;
  if (narrow ? encode_terms_map(&mh, xhi, K, T, ld, 2, (size_t)rows * ld, narrow_tp(T, 2))
             : encode_act_map(&mh, xhi, K, T, ld) || encode_act_map(&ml, xlo, K, T, ld))
    rc = KFL_ERR_CUDA;
  for (int n0 = 0; n0 < N && rc == KFL_OK; n0 += slab) {
    PrefillEpiParams e = {};
    e.T = T;
    e.N = std::min(slab, N - n0);
    e.out = y + n0;
    e.ldo = ldy;
    e.err = err;
    const int n_rb = (e.N + RB - 1) / RB;
    // (these two are launched when all before them is done, and so is what follows a slab's copy: the
    // few-token kernel reads weights before it waits for the kernel before it)
    if (!w_rows) tile_rows_kernel<<<(unsigned)n_rb * n_kt, 256, 0, s>>>(w + (size_t)n0 * K, e.N, K, n_kt, tiles);
    if (cudaPeekAtLastError() != cudaSuccess ||
        (n0 == 0 && launch_split_bf16(x, T, K, ldx, xhi, xlo, ld, err, s) != cudaSuccess) ||
        (w_rows ? encode_rows_map(&mb, w, K, N, narrow ? 128 : PG_N)
                : encode_tiles_map(&mb, tiles, n_kt, n_rb, (narrow ? 128 : PG_N) / RB))) {
      rc = KFL_ERR_CUDA;
      break;
    }
    const NarrowWorkspace ws = {partial, n_sm};
    if ((narrow ? launch_prefill_narrow(PE_STORE, mb, w_rows, mh, K, 2, ws, e, s, nullptr, n0 == 0)
                : launch_prefill_gemm(PE_STORE, mh, ml, mb, w_rows, K, ws, e, s)) != cudaSuccess)
      rc = KFL_ERR_CUDA;
  }
  if (rc == KFL_OK && cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess) rc = KFL_ERR_CUDA;
  // freed before the synchronisation: there the pool returns what it holds beyond its threshold
  if (pooled) cudaFreeAsync(mem, s);
  if (cudaStreamSynchronize(s) != cudaSuccess && rc == KFL_OK) rc = KFL_ERR_CUDA;
  if (!pooled) cudaFree(mem);
  if (rc == KFL_OK && (h_err & ERR_TIMEOUT)) rc = KFL_ERR_TIMEOUT;
  cudaGetLastError();
  return rc;
}
