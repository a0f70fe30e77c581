// The prefill GEMM of few tokens (sm_103a): Y^T[N][T] = W[N][K] X[T][K]^T with the weight rows as the
// M = 128 rows of the tcgen05 products and the tokens' terms side by side as their N columns, split
// stream-K over one CTA per SM.
//
// Up to 128 tokens the product is bound by the weights' stream from HBM (2 T flops per weight
// byte and term: at T = 128 the MMAs of a 16 KiB weight slice take about 512 cycles, its share of
// the HBM bandwidth about 750).  So every SM streams an equal share of the matrix, whatever its
// shape (TileShare), and a row tile that several CTAs share is summed from their partial sums in CTA
// order by a small kernel behind it (narrow_reduce_kernel; a residual's by the next norm,
// narrow_norm_kernel).
// The tokens' terms share each MMA: 128 weight rows x (terms x tokens) columns, so a token count
// of 16 costs an eighth of the 128-token tile of prefill_gemm_persistent, and the epilogue's lanes
// hold consecutive output columns of one token.
//
// Measured (7B-shaped blocks, 43 tokens): the gate/up loop streams its 272 MB in 36 us (7.0 TB/s
// after the first ring fill).  Clusters of up to 8 CTAs per 128-token tile, reducing through
// distributed shared memory, took 51 us for Q/K/V, 39 for O and down on average and 58 for gate/up
// (four blocks with everything between: 954 us, now 522).
#include <algorithm>
#include <type_traits>

#include "prefill_tc.cuh"

namespace kfl {

namespace {

constexpr int NW_WARPS = 10;             // TMA, MMA, 8 epilogue warps
constexpr int NW_THREADS = NW_WARPS * 32;
constexpr int NW_EPI_THREADS = 256;
constexpr int NW_DRAIN_TP = 80;          // tokens of a tile of three terms
constexpr int NW_DRAIN_KB = 2;           // K blocks per drained accumulator of three-term passes
constexpr int NW_PRODUCT_KB = 16;        // and of the plain product's two terms
// the most tokens of a drained tile
__host__ __device__ constexpr int narrow_drain_tp(int mode) { return mode == PE_STORE ? NW_MAX_TP : NW_DRAIN_TP; }
constexpr int NW_EPI_WARP = 2;            // the first epilogue warp
constexpr int NW_MAX_STAGES = 12;
constexpr int NW_RING = 226 * 1024;      // shared memory of the rings: a block's 227 KiB less the barriers' KiB

struct NarrowParams {
  TileShare share;  // of row tiles (of 128 mb rows) x token tiles, in K blocks of 64 (int4: units of 128)
  int t_tiles;
  int w_rows;       // the weight map is over a row-major matrix (encode_rows_map), not over weight tiles
  int tp, terms;    // tokens of a tile (a multiple of 16), terms per token: tp * terms columns
  int stages, stage_bytes;
  int acc_cols;     // TMEM columns of one 128-row accumulator (tp * terms rounded up to 32)
  int bufs;         // accumulators: 1 or 2
  int chunk;        // K blocks that one accumulator takes before the epilogue warps add it up (DRAIN; else all)
  int tmem_cols;
  float *ws;        // partial sums (narrow_partial)
};

// Where (in floats) a partial holds the sums of 128-row block m and token group gr: [part][m][gr][16
// tokens][128 rows].
__device__ __forceinline__ size_t narrow_partial(int part, int m, int gr, int mb, int tp) {
  return ((size_t)part * mb * (tp / 16) + (size_t)m * (tp / 16) + gr) * (16 * 128);
}

// The epilogue of 16 tokens t0 .. t0 + 15 of output row n (this lane's; the warp's lanes hold 32
// consecutive rows starting at a multiple of 32): load() fetches what it needs besides the sums, all
// of it in flight together and before the sums are there; store() finishes.
template <int MODE>
struct NarrowEpilogue {
  int pos[MODE == PE_QKV ? 16 : 1];
  float a[MODE == PE_QKV || MODE == PE_RESID ? 16 : 1];  // h; cos
  float b[MODE == PE_QKV ? 16 : 1];                       // sin

  __device__ __forceinline__ void load(const PrefillEpiParams &ep, int n, int t0, int lane) {
    const int nt = min(16, ep.T - t0);  // tokens that exist (uniform)
    if constexpr (MODE == PE_RESID) {
      const float *p = ep.out + (size_t)t0 * ep.ldo + n;
#pragma unroll
      for (int j = 0; j < 16; ++j) a[j] = n < ep.N && j < nt ? p[(size_t)j * ep.ldo] : 0.f;
    } else if constexpr (MODE == PE_QKV) {
#pragma unroll
      for (int j = 0; j < 16; ++j) pos[j] = j < nt ? ep.positions[t0 + j] : -1;
      if (n - lane < ep.qdim + ep.kvdim) {
        const int half = ep.hd / 2, i = (n < ep.qdim ? n : n - ep.qdim) % ep.hd / 2;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const size_t f = (size_t)max(pos[j], 0) * half + i;
          a[j] = ep.rope_cos[f];
          b[j] = ep.rope_sin[f];
        }
      }
    }
  }

  // slot: the argmax partial of these 32 rows
  __device__ __forceinline__ void store(const PrefillEpiParams &ep, int n, int t0, const float (&v)[16], int lane,
                                        int slot) const {
    const bool row_ok = n < ep.N;
    const int nt = min(16, ep.T - t0);
    if constexpr (MODE == PE_STORE || MODE == PE_RESID) {
      float *p = ep.out + (size_t)t0 * ep.ldo + n;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (row_ok && j < nt) p[(size_t)j * ep.ldo] = MODE == PE_RESID ? a[j] + v[j] : v[j];
    } else if constexpr (MODE == PE_SWIGLU) {
      // even rows hold gates, odd rows the matching ups: the even lane takes tokens t0 .. t0 + 7,
      // the odd lane t0 + 8 .. t0 + 15
      const bool odd = lane & 1;
      uint16_t *o = ep.out16 + (size_t)(t0 + (odd ? 8 : 0)) * ep.ldo16 + (n >> 1);
#pragma unroll
      for (int i = 0; i < 8; ++i, o += ep.ldo16) {
        const float other = __shfl_xor_sync(0xffffffffu, odd ? v[i] : v[8 + i], 1);
        const float g = odd ? other : v[i], u = odd ? v[8 + i] : other;
        if (row_ok && (odd ? 8 + i : i) < nt) {
          const float y = g / (1.0f + expf(-g)) * u;
          if (ep.f16 && !(fabsf(y) < 65520.f)) atomicOr(ep.err, ERR_F16_RANGE);
          uint16_t term[3];
          split_terms(y, term, ep.terms, ep.f16);
          o[0] = term[0];
          o[ep.term_stride] = term[1];
          if (ep.terms == 3) o[2 * ep.term_stride] = term[2];
        }
      }
    } else if constexpr (MODE == PE_QKV) {
      if (n - lane < ep.qdim + ep.kvdim) {
        // rows (2 i, 2 i + 1) of a head are its RoPE pair (i, i + hd / 2)
        const bool odd = lane & 1, is_q = n - lane < ep.qdim;
        const int r0 = is_q ? n : n - ep.qdim, head = r0 / ep.hd, i = (r0 % ep.hd) / 2, at = odd ? i + ep.hd / 2 : i;
        float *q32 = is_q && ep.out ? ep.out + (size_t)t0 * ep.ldo + (size_t)head * ep.hd + at : nullptr;
        uint16_t *base = is_q ? ep.out16 + (size_t)t0 * ep.ldo16 + (size_t)head * ep.hd + at
                              : ep.kcache + ((size_t)ep.slot * ep.hkv + head) * ep.max_ctx * ep.hd + at;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float other = __shfl_xor_sync(0xffffffffu, v[j], 1);
          const float y = odd ? v[j] * a[j] + other * b[j] : v[j] * a[j] - other * b[j];
          if (q32) {
            if (pos[j] >= 0 && row_ok) q32[(size_t)j * ep.ldo] = y;
          } else if (pos[j] >= 0 && row_ok) {
            base[is_q ? (size_t)j * ep.ldo16 : (size_t)pos[j] * ep.hd] = f32_to_bf16_rne(y);
          }
        }
      } else {
        const int r0 = n - ep.qdim - ep.kvdim;
        uint16_t *base = ep.vcache + ((size_t)ep.slot * ep.hkv + r0 / ep.hd) * ep.max_ctx * ep.hd + r0 % ep.hd;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (pos[j] >= 0 && row_ok) base[(size_t)pos[j] * ep.hd] = f32_to_bf16_rne(v[j]);
      }
    } else if constexpr (MODE == PE_ARGMAX) {
      float best = -INFINITY;
      int bidx = 0x7FFFFFFF;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        // order-preserving integer of the value; rows past the end and NaN never win
        const float x = row_ok && v[j] > -INFINITY ? v[j] : -INFINITY;
        const int k = __float_as_int(x), key = k ^ ((k >> 31) & 0x7FFFFFFF);
        const int m = __reduce_max_sync(0xffffffffu, key);
        const int first = __ffs(__ballot_sync(0xffffffffu, key == m)) - 1;
        const float mv = __int_as_float(m ^ ((m >> 31) & 0x7FFFFFFF));
        if (lane == j && mv > -INFINITY) {
          best = mv;
          bidx = n - lane + first;
        }
      }
      if (lane < nt && slot < ep.n_tiles) {
        ep.amax[(size_t)(t0 + lane) * ep.n_tiles + slot] = best;
        ep.aidx[(size_t)(t0 + lane) * ep.n_tiles + slot] = bidx;
      }
    }
  }
};

// The epilogue warps' part of a CTA: every segment's sums, from its
// accumulator to the outputs or, where CTAs share the tile, to the partial sums (narrow_reduce_kernel).
template <int MODE, int MB, bool DRAIN>
__device__ __forceinline__ void narrow_epilogue_warps(const NarrowParams &p, const PrefillEpiParams &ep, uint32_t tmem,
                                                      uint64_t *s_acc_full, uint64_t *s_acc_empty,
                                                      volatile int *abort_flag) {
  static_assert(!DRAIN || MB == 1, "a drained tile's sums fit the registers");
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  // ---- epilogue warps: TMEM lanes 32 q .. (q = warp % 4) are 32 consecutive rows of the tile;
  // the two warps of a quadrant take alternate groups of 16 tokens
  pdl_wait();  // h, the partial sums and the outputs may still be in use by the previous kernel
  const int q = warp & 3, grp = (warp - NW_EPI_WARP) >> 2, row = 32 * q + lane;
  const int groups = p.tp / 16;
  int seg = 0;
  // accumulator number `seg` (a segment, or a chunk of one) is complete; false: given up
  auto wait_acc = [&]() {
    const uint32_t bar = smem_addr(&s_acc_full[p.bufs == 2 ? seg & 1 : 0]);
    const bool ready =
        __all_sync(0xffffffffu, !*abort_flag && mbar_wait(bar, (uint32_t)(p.bufs == 2 ? seg >> 1 : seg) & 1));
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
    if (lane == 0) mbar_arrive(smem_addr(&s_acc_empty[p.bufs == 2 ? seg & 1 : 0]));
    ++seg;
  };
  // 16 tokens' sums of the accumulator, the smaller terms first
  auto read_acc = [&](int m, int gr, float(&v)[16]) {
    const int buf = p.bufs == 2 ? seg & 1 : 0;
    const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((buf * MB + m) * p.acc_cols + gr * 16);
    uint32_t r0[16], r1[16], r2[16];
    tmem_ld16(ta, r0);
    tmem_ld16(ta + p.tp, r1);
    if (p.terms == 3) tmem_ld16(ta + 2 * p.tp, r2);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float lo = p.terms == 3 ? __uint_as_float(r1[j]) + __uint_as_float(r2[j]) : __uint_as_float(r1[j]);
      v[j] = __uint_as_float(r0[j]) + lo;
    }
  };
  for (TileWalk w(p.share); w.next();) {
    const bool whole = w.whole();
    const int r_tile = w.tile / p.t_tiles, tt0 = (w.tile % p.t_tiles) * p.tp;
    auto finish = [&](int m, int gr, const float(&v)[16], const NarrowEpilogue<MODE> &e) {
      const int n = (r_tile * MB + m) * 128 + row;
      if (whole) {
        e.store(ep, n, tt0 + gr * 16, v, lane, (r_tile * MB + m) * 4 + q);
      } else {
        float *at = p.ws + narrow_partial(w.part, m, gr, MB, p.tp) + row;
#pragma unroll
        for (int j = 0; j < 16; ++j) at[j * 128] = v[j];
      }
    };
    if constexpr (DRAIN) {
      constexpr int OWN = (narrow_drain_tp(MODE) / 16 + 1) / 2;  // groups of this warp
      float sum[OWN][16] = {};
      for (int left = w.kb1 - w.kb0; left > 0; left -= p.chunk) {
        if (!wait_acc()) return;
#pragma unroll
        for (int k = 0; k < OWN; ++k) {
          const int gr = grp + 2 * k;
          if (gr < groups) {
            float v[16];
            read_acc(0, gr, v);
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[k][j] += v[j];
          }
        }
        release_acc();
      }
#pragma unroll
      for (int k = 0; k < OWN; ++k) {
        const int gr = grp + 2 * k, t0 = tt0 + gr * 16;
        if (gr < groups && t0 < ep.T) {
          NarrowEpilogue<MODE> e;
          if (whole) e.load(ep, r_tile * 128 + row, t0, lane);
          finish(0, gr, sum[k], e);
        }
      }
    } else {
      if (!wait_acc()) return;
      for (int m = 0; m < MB; ++m)
        for (int gr = grp; gr < groups; gr += 2) {
          const int t0 = tt0 + gr * 16;
          if (t0 >= ep.T) break;
          NarrowEpilogue<MODE> e;
          if (whole) e.load(ep, (r_tile * MB + m) * 128 + row, t0, lane);
          float v[16];
          read_acc(m, gr, v);
          finish(m, gr, v, e);
        }
      release_acc();
    }
  }
}

// The tiles that several CTAs share: their partial sums, added in K order, and the epilogue.  One
// block per 128 rows x 16 tokens, so that the sums (up to 70 KB a CTA of the GEMM) are read by the
// whole GPU at once: summed by the last CTA to arrive at a tile, inside the GEMM, they cost 4 to 8 us
// at 43 tokens and 20 to 50 us at 100, of a tail in which most SMs were idle.
template <int MODE>
__global__ void __launch_bounds__(128) narrow_reduce_kernel(NarrowParams p, int mb, int gemm_ctas, PrefillEpiParams ep) {
  pdl_launch_dependents();
  const int groups = p.tp / 16, gr = blockIdx.x % groups, m = blockIdx.x / groups % mb, sk = blockIdx.x / groups / mb;
  const int q = threadIdx.x / 32, lane = threadIdx.x % 32, row = threadIdx.x;
  const int tile = p.share.waves * gemm_ctas + sk;
  const int r_tile = tile / p.t_tiles, t0 = (tile % p.t_tiles) * p.tp + gr * 16;
  const TileParts parts(p.share, sk, gemm_ctas);
  pdl_wait();
  if (parts.n == 1 || t0 >= ep.T) return;
  const int n = (r_tile * mb + m) * 128 + row;
  const float *ws = p.ws + row;
  NarrowEpilogue<MODE> e;
  e.load(ep, n, t0, lane);
  float v[16] = {};
  for (int k = 0; k < parts.n; k += 4) {
    float x[4][16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float *w = ws + narrow_partial(parts.part(k + i), m, gr, mb, p.tp);
#pragma unroll
      for (int j = 0; j < 16; ++j) x[i][j] = k + i < parts.n ? __ldcg(w + j * 128) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] += x[i][j];
  }
  e.store(ep, n, t0, v, lane, (r_tile * mb + m) * 4 + q);
}

// One token's residual stream after a residual GEMM: the partial sums of the cut tiles added to h (in K
// order, then h: as narrow_reduce_kernel), and its RMSNorm, in place of two kernels of which
// each was latency.  A thread has NW_NORM_V groups of four elements in flight (43 tokens x 3584: 7.0 us for
// 8.6 + 6.3, cold; 100 x 8192: 10.2 for 8.5 + 9.0).
constexpr int NW_NORM_THREADS = 1024, NW_NORM_V = 2;
__global__ void __launch_bounds__(NW_NORM_THREADS) narrow_norm_kernel(NarrowPending p, float *h, int ldh, int d,
                                                                       const float *g, float eps, uint16_t *x,
                                                                       size_t term_stride, int terms, int ldx, int f16,
                                                                       unsigned *err) {
  __shared__ TileParts s_parts[NW_NORM_MAX_D / 128];
  __shared__ float red[NW_NORM_THREADS / 32];
  pdl_launch_dependents();
  const int t = blockIdx.x, rows = 128 * p.mb, tt = t / p.tp, tl = t - tt * p.tp;
  const int dp = p.share.waves * p.grid;  // tiles below it are whole, and in h already
  for (int r = threadIdx.x; r * rows < d; r += blockDim.x) {
    const int tile = r * p.t_tiles + tt;
    s_parts[r] = TileParts(p.share, max(tile - dp, 0), p.grid);
    if (tile < dp) s_parts[r].n = 1;
  }
  __syncthreads();
  pdl_wait();
  float *row = h + (size_t)t * ldh;
  const float *ws = p.ws + (size_t)(tl & 15) * 128;
  auto residual = [&](int n0) {
    const TileParts parts = s_parts[n0 / rows];
    float4 v = *reinterpret_cast<const float4 *>(row + n0), y = make_float4(0.f, 0.f, 0.f, 0.f);
    if (parts.n > 1) {
      const float *at = ws + n0 % 128;
      for (int k = 0; k < parts.n; k += 4) {
        float4 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          a[i] = k + i < parts.n ? __ldcg(reinterpret_cast<const float4 *>(
                                       at + narrow_partial(parts.part(k + i), n0 / 128 % p.mb, tl / 16, p.mb, p.tp)))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) y.x += a[i].x, y.y += a[i].y, y.z += a[i].z, y.w += a[i].w;
      }
      v = make_float4(v.x + y.x, v.y + y.y, v.z + y.z, v.w + y.w);
      *reinterpret_cast<float4 *>(row + n0) = v;
    }
    return v;
  };
  float ss = 0.f;
  float4 v[NW_NORM_V];
#pragma unroll
  for (int i = 0; i < NW_NORM_V; ++i) {  // d is a multiple of 8
    const int n0 = 4 * (threadIdx.x + i * blockDim.x);
    v[i] = n0 < d ? residual(n0) : make_float4(0.f, 0.f, 0.f, 0.f);
    ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  }
  for (int n0 = 4 * (threadIdx.x + NW_NORM_V * blockDim.x); n0 < d; n0 += 4 * blockDim.x) {
    const float4 a = residual(n0);
    ss += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
  }
  const float inv = 1.0f / sqrtf(block_sum(ss, red) / d + eps);
  auto put = [&](int n0, float4 a) {
    store_normed(a, inv, *reinterpret_cast<const float4 *>(g + n0), x + (size_t)t * ldx + n0, term_stride, terms, f16,
                 err);
  };
#pragma unroll
  for (int i = 0; i < NW_NORM_V; ++i) {
    const int n0 = 4 * (threadIdx.x + i * blockDim.x);
    if (n0 < d) put(n0, v[i]);
  }
  for (int n0 = 4 * (threadIdx.x + NW_NORM_V * blockDim.x); n0 < d; n0 += 4 * blockDim.x)
    put(n0, *reinterpret_cast<const float4 *>(row + n0));  // this thread's own h
}

// A producer's place in its CTA's segments: the K block it loads next, of row tile r_tile and the tokens
// from t0 (worked out once a segment).
struct NarrowAt {
  TileWalk w;
  int kb, r_tile, t0;
  bool more;
  __device__ __forceinline__ explicit NarrowAt(const NarrowParams &p) : w(p.share) { seek(p); }
  __device__ __forceinline__ void seek(const NarrowParams &p) {
    more = w.next();
    kb = more ? w.kb0 : 0;
    r_tile = more ? w.tile / p.t_tiles : 0;
    t0 = more ? (w.tile - r_tile * p.t_tiles) * p.tp : 0;
  }
  __device__ __forceinline__ void next(const NarrowParams &p) {
    if (++kb == w.kb1) seek(p);
  }
};

// MB: 128-row blocks per tile, 1 or 2.  DRAIN (three terms, and the plain product; MB 1, two accumulators):
// each accumulator takes only p.chunk K blocks, and the epilogue warps add the chunks up in registers.  A tensor-core accumulation
// truncates: about 3e-8 of the sum per 16 K values, always towards zero, so 224 of them (K = 3584) put
// the products of three-term activations at 5e-6, an order above the fp32 FMAs of a decode step;
// chunks of 128 K values leave 2.5e-7.  (The plain product, whose two terms leave 2e-6 of x, in chunks of
// 1024: 1 to 128 tokens by 18944 x 18944 are 2.6e-6 off, 1.5e-5 undrained, in 143 to 168 us against 141 to
// 163.)
// Measured on 7B-shaped QK-norm prompts: of 512,000 K and as many V elements of a block, 67 and 54 land
// beside the bf16 that 64 bits round to (84 and 82 as decode steps; 2,400 with two terms, undrained);
// 200 tokens, two blocks: 11,690 us as decode steps, 798 drained, 677 undrained.
template <int MODE, int MB, bool DRAIN>
__global__ void __launch_bounds__(NW_THREADS, 1)
    prefill_narrow_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                          NarrowParams p, PrefillEpiParams ep) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_full[NW_MAX_STAGES], s_empty[NW_MAX_STAGES], s_acc_full[2], s_acc_empty[2], s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const uint32_t ring = (smem_addr(smem_raw) + 1023u) & ~1023u;
  const uint32_t x_off = (uint32_t)MB * NW_W_BYTES;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_addr(&s_full[s]), 1);
      mbar_init(smem_addr(&s_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_addr(&s_acc_full[b]), 1);
      mbar_init(smem_addr(&s_acc_empty[b]), NW_EPI_THREADS / 32);  // one arrival per epilogue warp
    }
    mbar_init(smem_addr(&s_drain), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_addr(&s_tmem), p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int *abort_flag = &s_abort;
  // the next kernel's CTAs may take the SMs that this one leaves; they wait for this whole grid
  // before they read anything but weights
  pdl_launch_dependents();

  if (warp == 0) {
    // ---- TMA producer (the whole warp, one elected lane issuing): the i-th K block of the CTA's range
    // uses stage i % S.  Weights do not depend on the previous kernel: the first round of them is
    // under way before the wait on it
    // weights that another token tile reads again stay in L2
    const uint64_t pol = p.t_tiles == 1 ? policy_evict_first() : policy_evict_normal();
    const uint32_t bytes = x_off + (uint32_t)p.tp * p.terms * 128u;
    NarrowAt w(p), x(p);  // where the next weight and the next token loads are
    int ws = 0, wuse = 0, xs = 0, xuse = 0;
    auto weights = [&]() {
      const uint32_t full = smem_addr(&s_full[ws]), dst = ring + ws * p.stage_bytes;
      if (elect_one()) {
        mbar_arrive_expect_tx(full, bytes);
#pragma unroll
        for (int m = 0; m < MB; ++m) {
          if (p.w_rows)
            tma_load_2d_hint(dst + m * NW_W_BYTES, &tm_w, w.kb * 64, (w.r_tile * MB + m) * 128, full, pol);
          else
            tma_load_4d_hint(dst + m * NW_W_BYTES, &tm_w, (w.kb & 1) * 64, 0, w.kb >> 1,
                             (w.r_tile * MB + m) * (128 / RB), full, pol);
        }
      }
      __syncwarp();
      w.next(p);
      if (++ws == p.stages) ws = 0, ++wuse;
    };
    auto tokens = [&]() {
      if (elect_one())
        tma_load_3d(ring + xs * p.stage_bytes + x_off, &tm_x, x.kb * 64, x.t0, 0, smem_addr(&s_full[xs]));
      __syncwarp();
      x.next(p);
      if (++xs == p.stages) xs = 0, ++xuse;
    };
    while (w.more && wuse == 0) weights();
    pdl_wait();
    asm volatile("fence.proxy.async;" ::: "memory");  // the previous kernel's stores, before TMA reads them
    while (x.more && xuse == 0) tokens();
    bool ok = true;
    while (w.more) {
      ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_empty[ws]), (uint32_t)(wuse - 1) & 1));
      if (!ok) break;
      weights();
      tokens();
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicOr(ep.err, ERR_TIMEOUT);
      }
      // let the copies in flight land: stage s was last filled in its use number wuse - (s >= ws)
      for (int s = 0; s < p.stages; ++s) {
        const int last = wuse - (s >= ws ? 1 : 0);
        if (last >= 0) mbar_wait(smem_addr(&s_full[s]), (uint32_t)last & 1);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer (the whole warp, one elected lane issuing): segment i of the range (one row
    // tile's share, or with DRAIN a chunk of it) accumulates into buffer i % bufs
    const uint32_t idesc = idesc_kind_f16(128, p.tp * p.terms, !ep.f16);
    TileWalk w(p.share);
    int s = 0, left = 0;  // K blocks of the segment not yet issued
    uint32_t use = 0;
    bool ok = true;
    for (int seg = 0; ok; ++seg) {
      if (left == 0) {
        if (!w.next()) break;
        left = w.kb1 - w.kb0;
      }
      const int n = DRAIN ? min(left, p.chunk) : left;
      left -= n;
      const int buf = p.bufs == 2 ? seg & 1 : 0;
      if (seg >= p.bufs) {
        const uint32_t back = (uint32_t)(p.bufs == 2 ? (seg >> 1) - 1 : seg - 1);
        ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&s_acc_empty[buf]), back & 1));
        if (!ok) break;
      }
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)(buf * MB * p.acc_cols);
      for (int i = 0; i < n; ++i) {
        ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_full[s]), use & 1));
        if (!ok) break;
        tc_fence_after();
        const uint32_t a = ring + s * p.stage_bytes;
        const uint64_t da = sdesc_k_sw128(a), db = sdesc_k_sw128(a + x_off);
        if (elect_one()) {
          // one accumulator after the other: at N = 256 an MMA takes 128 cycles behind one on the same
          // accumulator, 150 behind one on another
#pragma unroll
          for (int m = 0; m < MB; ++m)
#pragma unroll
            for (int k = 0; k < 4; ++k)  // 16 K values further: 32 bytes, 2 in the descriptor's units
              mma_bf16_ss(d + m * p.acc_cols, da + m * (NW_W_BYTES >> 4) + 2 * k, db + 2 * k, idesc, (i | k) != 0);
          mma_commit(smem_addr(&s_empty[s]));
        }
        __syncwarp();
        if (++s == p.stages) s = 0, ++use;
      }
      if (ok && elect_one()) mma_commit(smem_addr(&s_acc_full[buf]));
      __syncwarp();
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(ep.err, ERR_TIMEOUT);
    }
    if (elect_one()) mma_commit(smem_addr(&s_drain));  // every MMA issued has completed before TMEM is freed
    __syncwarp();
    mbar_wait(smem_addr(&s_drain), 0);
  } else {
    narrow_epilogue_warps<MODE, MB, DRAIN>(p, ep, tmem, s_acc_full, s_acc_empty, abort_flag);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

// ---------------------------------------------------------------------------- int4 weights
// The same product with int4 weights decoded on the way: a K unit is half an int4 tile (128 columns)
// of the tile's 256 rows, whose codes and scales (17 KiB, four row blocks) arrive by bulk copies;
// eight converter warps turn each 64-column half into the swizzled fp16 A operand of the MMAs (code x
// scale rounded to fp16, as dequant_int4_f16_kernel rounds it), while the tokens' slices arrive by TMA
// beside it.  Reads of HBM are the int4 bytes alone: dequantizing a matrix to an fp16 copy first
// costs 4.5 times its bytes (0.53 read, 2 written and 2 read again).
// 256 rows to a tile: a token slice (up to 32 KiB) is read from L2 once per 16 KiB of fp16 weights of
// two 128-row blocks, and each converter warp has two independent 16-row groups in hand.
// Measured, one 72B-shaped block: 261 us at 16 tokens, 359 at 100 and 1389 at 512, against 1207, 1228 and
// 2188 with fp16 copies made ahead on a second stream (1517 at 512 with their faster kernel of today,
// which takes over from there).  Bound by the converters at few tokens and by the MMAs from about 100.
constexpr int N4_CONV_WARPS = 8;
constexpr int N4_CONV_WARP = 10;  // the first converter warp
constexpr int N4_THREADS = (N4_CONV_WARP + N4_CONV_WARPS) * 32;
constexpr int N4_A_BYTES = 2 * NW_W_BYTES;                                   // 256 rows x 64 fp16
constexpr int N4_RB_BYTES = TILE4_CODE_BYTES / 2 + TILE4_SCALE_BYTES / 2;    // one row block's half tile
constexpr int N4_CODE_BYTES = 4 * N4_RB_BYTES;
constexpr int N4_MAX_CODE_STAGES = 8, N4_MAX_A_STAGES = 3, N4_MAX_X_STAGES = 6;

// The rings of a CTA: code stages, operand (A) stages and token stages.
struct Narrow4Params {
  const uint8_t *tiles;
  int n_rb, n_kt;
  int c_stages, a_stages, x_stages, x_bytes;
};


template <int MODE>
__global__ void __launch_bounds__(N4_THREADS, 1)
    prefill_narrow4_kernel(const Narrow4Params r, const __grid_constant__ CUtensorMap tm_x, NarrowParams p,
                           PrefillEpiParams ep) {
  constexpr int MB = 2;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_cfull[N4_MAX_CODE_STAGES], s_cempty[N4_MAX_CODE_STAGES], s_xfull[N4_MAX_X_STAGES],
      s_xempty[N4_MAX_X_STAGES], s_afull[N4_MAX_A_STAGES], s_aempty[N4_MAX_A_STAGES], s_acc_full[2], s_acc_empty[2],
      s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const uint32_t a_ring = (smem_addr(smem_raw) + 1023u) & ~1023u;
  const uint32_t x_ring = a_ring + r.a_stages * N4_A_BYTES;
  const uint32_t codes = x_ring + r.x_stages * r.x_bytes;  // [code stage][row block][codes, scales]
  if (threadIdx.x == 0) {
    for (int s = 0; s < r.c_stages; ++s) {
      mbar_init(smem_addr(&s_cfull[s]), 1);
      mbar_init(smem_addr(&s_cempty[s]), N4_CONV_WARPS);
    }
    for (int s = 0; s < r.a_stages; ++s) {
      mbar_init(smem_addr(&s_afull[s]), N4_CONV_WARPS);
      mbar_init(smem_addr(&s_aempty[s]), 1);
    }
    for (int s = 0; s < r.x_stages; ++s) {
      mbar_init(smem_addr(&s_xfull[s]), 1);
      mbar_init(smem_addr(&s_xempty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_addr(&s_acc_full[b]), 1);
      mbar_init(smem_addr(&s_acc_empty[b]), NW_EPI_THREADS / 32);
    }
    mbar_init(smem_addr(&s_drain), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) tmem_alloc(smem_addr(&s_tmem), p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int *abort_flag = &s_abort;
  pdl_launch_dependents();

  if (warp == 0) {
    // ---- producer (the whole warp, one elected lane issuing): units' codes as the code ring frees,
    // their two token slices as the token ring does
    const uint64_t pol = p.t_tiles == 1 ? policy_evict_first() : policy_evict_normal();
    NarrowAt w(p), x(p);  // where the next codes and the next token slices are
    int cs = 0, cuse = 0, xs = 0, xuse = 0, half = 0;
    auto issue_codes = [&]() {
      const uint32_t full = smem_addr(&s_cfull[cs]), dst = codes + cs * N4_CODE_BYTES;
      if (elect_one()) {
        mbar_arrive_expect_tx(full, N4_CODE_BYTES);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          // row blocks past the end repeat the last: their rows are beyond N and never stored
          const int rb = min(w.r_tile * 4 + b, r.n_rb - 1);
          const uint8_t *t = r.tiles + ((size_t)rb * r.n_kt + (w.kb >> 1)) * TILE4_BYTES;
          bulk_g2s(dst + b * N4_RB_BYTES, t + (w.kb & 1) * (TILE4_CODE_BYTES / 2), TILE4_CODE_BYTES / 2, full, pol);
          bulk_g2s(dst + b * N4_RB_BYTES + TILE4_CODE_BYTES / 2,
                   t + TILE4_CODE_BYTES + (w.kb & 1) * (TILE4_SCALE_BYTES / 2), TILE4_SCALE_BYTES / 2, full, pol);
        }
      }
      __syncwarp();
      w.next(p);
      if (++cs == r.c_stages) cs = 0, ++cuse;
    };
    auto issue_tokens = [&]() {
      const uint32_t full = smem_addr(&s_xfull[xs]);
      if (elect_one()) {
        mbar_arrive_expect_tx(full, r.x_bytes);
        tma_load_3d(x_ring + xs * r.x_bytes, &tm_x, x.kb * 128 + half * 64, x.t0, 0, full);
      }
      __syncwarp();
      if (half) x.next(p);
      half ^= 1;
      if (++xs == r.x_stages) xs = 0, ++xuse;
    };
    while (w.more && cuse == 0) issue_codes();
    pdl_wait();
    asm volatile("fence.proxy.async;" ::: "memory");  // the previous kernel's stores, before TMA reads them
    while (x.more && xuse == 0) issue_tokens();
    bool ok = true;
    // whichever ring has room goes first; one of them always will, or a wait elsewhere gives up
    for (uint32_t idle = 0; x.more || w.more;) {
      bool did = false;
      if (w.more && __any_sync(0xffffffffu, mbar_test_wait(smem_addr(&s_cempty[cs]), (uint32_t)(cuse - 1) & 1))) {
        issue_codes();
        did = true;
      }
      if (x.more && __any_sync(0xffffffffu, mbar_test_wait(smem_addr(&s_xempty[xs]), (uint32_t)(xuse - 1) & 1))) {
        issue_tokens();
        did = true;
      }
      idle = did ? 0 : idle + 1;
      if (__any_sync(0xffffffffu, *abort_flag != 0) || idle > WAIT_LIMIT) {
        ok = false;
        break;
      }
      if (idle >= WAIT_FAST_SPINS) __nanosleep(64);
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicOr(ep.err, ERR_TIMEOUT);
      }
      for (int s = 0; s < r.c_stages; ++s) {
        const int last = cuse - (s >= cs ? 1 : 0);
        if (last >= 0) mbar_wait(smem_addr(&s_cfull[s]), (uint32_t)last & 1);
      }
      for (int s = 0; s < r.x_stages; ++s) {
        const int last = xuse - (s >= xs ? 1 : 0);
        if (last >= 0) mbar_wait(smem_addr(&s_xfull[s]), (uint32_t)last & 1);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer, as in prefill_narrow_kernel; a unit is two stages
    const uint32_t idesc = idesc_kind_f16(128, p.tp * p.terms, false);
    TileWalk w(p.share);
    int as = 0, xs = 0;
    uint32_t ause = 0, xuse = 0;
    bool ok = true;
    for (int seg = 0; ok && w.next(); ++seg) {
      const int n = w.kb1 - w.kb0;
      const int buf = p.bufs == 2 ? seg & 1 : 0;
      if (seg >= p.bufs) {
        const uint32_t back = (uint32_t)(p.bufs == 2 ? (seg >> 1) - 1 : seg - 1);
        ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&s_acc_empty[buf]), back & 1));
        if (!ok) break;
      }
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)(buf * MB * p.acc_cols);
      for (int i = 0; i < 2 * n; ++i) {
        ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_xfull[xs]), xuse & 1) &&
                                         mbar_wait(smem_addr(&s_afull[as]), ause & 1));
        if (!ok) break;
        tc_fence_after();
        const uint64_t da = sdesc_k_sw128(a_ring + as * N4_A_BYTES), db = sdesc_k_sw128(x_ring + xs * r.x_bytes);
        if (elect_one()) {
#pragma unroll
          for (int m = 0; m < MB; ++m)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_bf16_ss(d + m * p.acc_cols, da + m * (NW_W_BYTES >> 4) + 2 * k, db + 2 * k, idesc, (i | k) != 0);
          mma_commit(smem_addr(&s_aempty[as]));
          mma_commit(smem_addr(&s_xempty[xs]));
        }
        __syncwarp();
        if (++as == r.a_stages) as = 0, ++ause;
        if (++xs == r.x_stages) xs = 0, ++xuse;
      }
      if (ok && elect_one()) mma_commit(smem_addr(&s_acc_full[buf]));
      __syncwarp();
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(ep.err, ERR_TIMEOUT);
    }
    if (elect_one()) mma_commit(smem_addr(&s_drain));  // every MMA issued has completed before TMEM is freed
    __syncwarp();
    mbar_wait(smem_addr(&s_drain), 0);
  } else if (warp < N4_CONV_WARP) {
    narrow_epilogue_warps<MODE, MB, false>(p, ep, tmem, s_acc_full, s_acc_empty, abort_flag);
  } else {
    // ---- converters: warp w decodes 16-row groups (row block b, r16) = (w / 4 and w / 4 + 2, w % 4)
    const int cw = warp - N4_CONV_WARP, r16 = cw & 3, gid = lane >> 2;
    // where this lane's stmatrix row goes: matrices 0..3 are rows 0-7 and 8-15 of columns 0-7, then of
    // columns 8-15 of each 16-column step j; 16-byte chunks of a 128-byte row XOR the row (mod 8)
    const int mrow = (lane & 7) + ((lane >> 3) & 1) * 8, mcol = lane >> 4;
    uint32_t off[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) off[j] = (uint32_t)((r16 * 16 + mrow) * 128 + (((2 * j + mcol) ^ (lane & 7)) << 4));
    int cs = 0, s = 0;
    uint32_t cuse = 0, use = 0;
    int total = 0;  // the CTA's units
    for (TileWalk w(p.share); w.next();) total += w.kb1 - w.kb0;
    bool ok = true;
    for (int i = 0; i < total && ok; ++i) {
      ok = __all_sync(0xffffffffu, !*abort_flag && mbar_wait(smem_addr(&s_cfull[cs]), cuse & 1));
      if (!ok) break;
      // the unit's codes and scales of this warp's rows: [half][group]
      const uint32_t src = codes + cs * N4_CODE_BYTES + (cw >> 2) * N4_RB_BYTES;
      uint4 w[2][2];
      uint32_t sc[2][2];
      bool exact = true;
#pragma unroll
      for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const uint32_t blk = src + 2 * g * N4_RB_BYTES;
          uint4 &v = w[half][g];
          asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                       : "r"(blk + r16 * 1024 + half * 512 + lane * 16));
          asm volatile("ld.shared.u32 %0, [%1];"
                       : "=r"(sc[half][g])
                       : "r"(blk + TILE4_CODE_BYTES / 2 + (((half * 8 + gid) * 4 + r16) * 4)));
        }
#pragma unroll
      for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int g = 0; g < 2; ++g) exact = exact && ScalePair(sc[half][g]).exact();
      exact = __all_sync(0xffffffffu, exact);
      __syncwarp();  // every lane's reads, before lane 0 gives the stage back (a vote orders no memory)
      if (lane == 0) mbar_arrive(smem_addr(&s_cempty[cs]));
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        ok = ok && (use == 0 || __all_sync(0xffffffffu, mbar_wait(smem_addr(&s_aempty[s]), (use - 1) & 1)));
        if (!ok) break;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          // row block b = cw / 4 + 2 g: rows 64 (b % 2) of 128-row block b / 2
          const uint32_t dst = a_ring + s * N4_A_BYTES + g * NW_W_BYTES + (cw >> 2) * (64 * 128);
          const ScalePair sp(sc[half][g]);
          const uint32_t words[4] = {w[half][g].x, w[half][g].y, w[half][g].z, w[half][g].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t c0, c1, c2, c3;
            decode_word(words[j], c0, c1, c2, c3);
            sp.apply(exact, c0, c1, c2, c3);
            stsm_x4(dst + off[j], c0, c1, c2, c3);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stores, before the MMAs read them
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_addr(&s_afull[s]));
        if (++s == r.a_stages) s = 0, ++use;
      }
      if (++cs == r.c_stages) cs = 0, ++cuse;
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicOr(ep.err, ERR_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, p.tmem_cols);
  }
}

}  // namespace

size_t narrow_ws_bytes(int n_sm, int T) {
  // NW_PARTS partials per CTA of 256 rows x tp tokens
  return (size_t)n_sm * NW_PARTS * 256 * std::min(NW_MAX_TP, (T + 15) / 16 * 16) * sizeof(float);
}
int narrow_argmax_slots(int N) { return (N + 127) / 128 * 4; }

// Opts a kernel in to a block's whole shared memory; returns its dynamic part (the rings start on
// the KiB boundary after the kernel's own barriers), or -1.
class RingOptIn {
  SmemOptIn opt_in_;
  std::atomic<int> own_{-1};  // the kernel's static shared memory

 public:
  int operator()(const void *kernel) {
    int own = own_.load(std::memory_order_relaxed);
    if (own < 0) {
      cudaFuncAttributes a;
      if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess || a.sharedSizeBytes > 1024) return -1;
      own_.store(own = (int)a.sharedSizeBytes, std::memory_order_relaxed);
    }
    const int dyn = NW_RING + 1024 - own;
    return opt_in_(kernel, dyn) == cudaSuccess ? dyn : -1;
  }
};

template <int MODE>
static cudaError_t launch_narrow_reduce(const NarrowParams &p, int mb, int grid, const PrefillEpiParams &ep,
                                        cudaStream_t s, NarrowPending *pending) {
  if (pending) pending->any = false;
  if (!p.share.cut()) return cudaSuccess;
  if (pending && MODE == PE_RESID && ep.N <= NW_NORM_MAX_D) {
    *pending = NarrowPending{true, p.share, grid, mb, p.tp, p.t_tiles, p.ws};
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.share.tail * mb * (p.tp / 16)));
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, narrow_reduce_kernel<MODE>, p, mb, grid, ep);
}

template <int MODE, int MB, bool DRAIN>
static cudaError_t launch_narrow_mode(const CUtensorMap &w, const CUtensorMap &x, const NarrowParams &p, int grid,
                                      const PrefillEpiParams &ep, cudaStream_t s, NarrowPending *pending, bool early) {
  static RingOptIn opt_in;
  const int smem = opt_in(reinterpret_cast<const void *>(prefill_narrow_kernel<MODE, MB, DRAIN>));
  if (smem < 0) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NW_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_narrow_kernel<MODE, MB, DRAIN>, w, x, p, ep);
  return e == cudaSuccess ? launch_narrow_reduce<MODE>(p, MB, grid, ep, s, pending) : e;
}

int narrow_tp(int T, int terms) {
  const int most = terms == 2 ? NW_MAX_TP : NW_DRAIN_TP;  // terms * tp <= 256 MMA columns
  const int tiles = (T + most - 1) / most;
  return ((T + tiles - 1) / tiles + 15) / 16 * 16;
}

cudaError_t launch_prefill_narrow(int mode, const CUtensorMap &w, bool w_rows, const CUtensorMap &x, int K, int terms,
                                  const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s,
                                  NarrowPending *pending, bool early) {
  if (ep.T <= 0 || ep.N <= 0) return cudaSuccess;
  NarrowParams p = {};
  p.w_rows = w_rows;
  p.terms = terms;
  p.tp = narrow_tp(ep.T, terms);
  p.t_tiles = (ep.T + p.tp - 1) / p.tp;
  const int cols = p.tp * terms;
  // Q/K/V (and its plain form): K and V are rounded to bf16 next, and every error before that moves some
  // across a rounding
  p.chunk = terms == 2 ? NW_PRODUCT_KB : mode == PE_QKV || mode == PE_STORE ? 1 : NW_DRAIN_KB;
  // wide tiles of many rows share their tokens' slices between two 128-row blocks: the slices (2 x
  // 16 KiB of terms at 128 tokens) then cost no more L2 reads than the weights
  const bool drain = terms == 3 || mode == PE_STORE;
  const int mb = !drain && cols > 128 && (ep.N + 255) / 256 * p.t_tiles >= ws.n_sm * 3 / 4 ? 2 : 1;
  const int n_kb = (K + 63) / 64, n_tiles = (ep.N + 128 * mb - 1) / (128 * mb) * p.t_tiles;
  p.acc_cols = (cols + 31) / 32 * 32;
  p.bufs = 2 * mb * p.acc_cols <= 512 ? 2 : 1;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.bufs * mb * p.acc_cols) p.tmem_cols *= 2;
  p.stage_bytes = mb * NW_W_BYTES + cols * 128;
  p.stages = std::min(NW_MAX_STAGES, NW_RING / p.stage_bytes);
  p.ws = ws.partial;
  // at least four K blocks per CTA: finer splits cost more in partial sums than they stream sooner
  const long long U = (long long)n_tiles * n_kb;
  const int grid = (int)std::min<long long>(ws.n_sm, std::max<long long>(std::min<long long>(n_tiles, ws.n_sm), U / 4));
  p.share = share_tiles(n_tiles, n_kb, grid, p.t_tiles == 1, NW_PARTS);
  auto go = [&](auto m) {
    constexpr int MODE = decltype(m)::value;
    if constexpr (MODE != PE_STORE) {
      if (!drain)
        return mb == 2 ? launch_narrow_mode<MODE, 2, false>(w, x, p, grid, ep, s, pending, early)
                       : launch_narrow_mode<MODE, 1, false>(w, x, p, grid, ep, s, pending, early);
    }
    return launch_narrow_mode<MODE, 1, true>(w, x, p, grid, ep, s, pending, early);
  };
  switch (mode) {
    case PE_STORE: return go(std::integral_constant<int, PE_STORE>());
    case PE_RESID: return go(std::integral_constant<int, PE_RESID>());
    case PE_SWIGLU: return go(std::integral_constant<int, PE_SWIGLU>());
    case PE_QKV: return go(std::integral_constant<int, PE_QKV>());
    case PE_ARGMAX: return go(std::integral_constant<int, PE_ARGMAX>());
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE>
static cudaError_t launch_narrow4_mode(const Narrow4Params &r, const CUtensorMap &x, const NarrowParams &p, int grid,
                                       const PrefillEpiParams &ep, cudaStream_t s, NarrowPending *pending) {
  static RingOptIn opt_in;
  const int smem = opt_in(reinterpret_cast<const void *>(prefill_narrow4_kernel<MODE>));
  if (smem < 0) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(N4_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_narrow4_kernel<MODE>, r, x, p, ep);
  return e == cudaSuccess ? launch_narrow_reduce<MODE>(p, 2, grid, ep, s, pending) : e;
}

cudaError_t launch_prefill_narrow4(int mode, const uint8_t *tiles, int n_rb, int n_kt, const CUtensorMap &x, int K,
                                   int terms, const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s,
                                  NarrowPending *pending) {
  if (ep.T <= 0 || ep.N <= 0) return cudaSuccess;
  NarrowParams p = {};
  p.terms = terms;
  p.tp = narrow_tp(ep.T, terms);
  p.t_tiles = (ep.T + p.tp - 1) / p.tp;
  const int cols = p.tp * terms;
  const int n_kb = (K + 127) / 128, n_tiles = (ep.N + 255) / 256 * p.t_tiles;
  p.acc_cols = (cols + 31) / 32 * 32;
  p.bufs = 4 * p.acc_cols <= 512 ? 2 : 1;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.bufs * 2 * p.acc_cols) p.tmem_cols *= 2;
  // three code stages at least (70 KiB ahead of the converters with what they hold), then the token ring
  // (slices come from L2: about a microsecond), then more codes
  Narrow4Params r = {tiles, n_rb, n_kt, 0, 0, 0, cols * 128};
  r.a_stages = r.x_bytes <= 16384 ? 3 : 2;
  r.x_stages = std::min(N4_MAX_X_STAGES, (NW_RING - r.a_stages * N4_A_BYTES - 3 * N4_CODE_BYTES) / r.x_bytes);
  r.c_stages = std::min(N4_MAX_CODE_STAGES, (NW_RING - r.a_stages * N4_A_BYTES - r.x_stages * r.x_bytes) / N4_CODE_BYTES);
  p.ws = ws.partial;
  // at least two units (2 x 128 columns) per CTA, as prefill_narrow_kernel's four K blocks of 64
  const long long U = (long long)n_tiles * n_kb;
  const int grid = (int)std::min<long long>(ws.n_sm, std::max<long long>(std::min<long long>(n_tiles, ws.n_sm), U / 2));
  p.share = share_tiles(n_tiles, n_kb, grid, p.t_tiles == 1, NW_PARTS);
  auto go = [&](auto m) {
    return launch_narrow4_mode<decltype(m)::value>(r, x, p, grid, ep, s, pending);
  };
  switch (mode) {
    case PE_RESID: return go(std::integral_constant<int, PE_RESID>());
    case PE_SWIGLU: return go(std::integral_constant<int, PE_SWIGLU>());
    case PE_QKV: return go(std::integral_constant<int, PE_QKV>());
    case PE_ARGMAX: return go(std::integral_constant<int, PE_ARGMAX>());
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_narrow_norm(const NarrowPending &pend, float *h, int ldh, int T, int d, const float *g, float eps,
                               uint16_t *x, size_t term_stride, int terms, int ldx, int f16, unsigned *err,
                               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(T);
  cfg.blockDim = dim3(std::min(NW_NORM_THREADS, (d / 4 + 31) / 32 * 32));
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, narrow_norm_kernel, pend, h, ldh, d, g, eps, x, term_stride, terms, ldx, f16, err);
}

}  // namespace kfl
