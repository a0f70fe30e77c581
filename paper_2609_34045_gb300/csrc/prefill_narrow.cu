// The prefill GEMM of few tokens (sm_103a): Y^T[N][T] = W[N][K] X[T][K]^T with the weight rows as the
// M = 128 rows of the tcgen05 products and the tokens' terms side by side as their N columns, split
// stream-K over one CTA per SM.
//
// Up to 128 tokens the product is bound by the weights' stream from HBM (2 T flops per weight
// byte and term: at T = 128 the MMAs of a 16 KiB weight slice take about 512 cycles, its share of
// the HBM bandwidth about 750).  So every SM streams an equal share of the matrix, whatever its
// shape: the K blocks of all row tiles form one sequence, CTA c takes the contiguous range
// [c U / G, (c + 1) U / G) of it, and a row tile that several CTAs share is summed from their
// partial sums in CTA order by the last of them to arrive (no CTA ever waits for another).
// The tokens' terms share each MMA: 128 weight rows x (terms x tokens) columns, so a token count
// of 16 costs an eighth of the 128-token tile of prefill_gemm_persistent, and the epilogue's lanes
// hold consecutive output columns of one token.
//
// Measured (7B-shaped block, 43 tokens): the gate/up loop streams its 272 MB in 36 us (7.0 TB/s
// after the first ring fill); a GEMM takes 17 (Q/K/V), 28 (down) and 45 us (gate/up) from its first
// CTA to its last, of which 4 to 8 us are the shared tiles' sums and epilogues at the end; clusters
// of up to 8 CTAs per 128-token tile, reducing through distributed shared memory, took 51, 39 and
// 58 us (four blocks with everything between: 954 -> 697 us).
#include <algorithm>
#include <type_traits>

#include "prefill_tc.cuh"

namespace kfl {

namespace {

constexpr int NW_WARPS = 10;             // TMA, MMA, 8 epilogue warps
constexpr int NW_THREADS = NW_WARPS * 32;
constexpr int NW_EPI_THREADS = 256;
constexpr int NW_MAX_STAGES = 12;
constexpr int NW_SMEM = 224 * 1024;      // ring + alignment slack

struct NarrowParams {
  int n_kb;         // K blocks of 64
  int n_tiles;      // row tiles (of 128 mb rows) x token tiles
  int t_tiles;
  int tp, terms;    // tokens of a tile (a multiple of 16), terms per token: tp * terms columns
  int stages, stage_bytes;
  int acc_cols;     // TMEM columns of one 128-row accumulator (tp * terms rounded up to 32)
  int bufs;         // accumulators: 1 or 2
  int tmem_cols;
  float *ws;        // partial sums: [G][2][mb][tp][128]
  unsigned *tickets;  // [n_tiles], zero between launches
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Whether `ok` holds on all n threads that meet at named barrier id.
__device__ __forceinline__ bool named_bar_and(int id, int n, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %3, 0;\n\t"
      "barrier.cta.red.and.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(id), "r"(n), "r"((uint32_t)ok)
      : "memory");
  return r != 0;
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
        uint16_t *base = is_q ? ep.out16 + (size_t)t0 * ep.ldo16 + (size_t)head * ep.hd + at
                              : ep.kcache + ((size_t)ep.slot * ep.hkv + head) * ep.max_ctx * ep.hd + at;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float other = __shfl_xor_sync(0xffffffffu, v[j], 1);
          const float y = odd ? v[j] * a[j] + other * b[j] : v[j] * a[j] - other * b[j];
          if (pos[j] >= 0 && row_ok) base[is_q ? (size_t)j * ep.ldo16 : (size_t)pos[j] * ep.hd] = f32_to_bf16_rne(y);
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

// MB: 128-row blocks per tile, 1 or 2.
template <int MODE, int MB>
__global__ void __launch_bounds__(NW_THREADS, 1)
    prefill_narrow_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
                          NarrowParams p, PrefillEpiParams ep) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t s_full[NW_MAX_STAGES], s_empty[NW_MAX_STAGES], s_acc_full[2], s_acc_empty[2], s_drain;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_last;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const uint32_t ring = (smem_addr(smem_raw) + 1023u) & ~1023u;
  const long long U = (long long)p.n_tiles * p.n_kb, G = gridDim.x;
  const long long u0 = blockIdx.x * U / G, u1 = (blockIdx.x + 1) * U / G;
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
    if (lane == 0) {
      // ---- TMA producer: the i-th K block of the CTA's range uses stage i % S.  Weights do not
      // depend on the previous kernel: the first round of them is under way before the wait on it
      const uint64_t pol = policy_evict_first();
      const uint32_t bytes = x_off + (uint32_t)p.tp * p.terms * 128u;
      // the ring position and the (tile, K block) of the next weight and token loads
      struct At {
        int s, use, kb, r, t;  // stage, its use, K block, row tile, token tile
      };
      const int tile0 = (int)(u0 / p.n_kb);
      At w = {0, 0, (int)(u0 % p.n_kb), tile0 / p.t_tiles, tile0 % p.t_tiles}, x = w;
      auto next = [&](At &a) {
        if (++a.s == p.stages) a.s = 0, ++a.use;
        if (++a.kb == p.n_kb) {
          a.kb = 0;
          if (++a.t == p.t_tiles) a.t = 0, ++a.r;
        }
      };
      auto weights = [&]() {
        const uint32_t full = smem_addr(&s_full[w.s]), dst = ring + w.s * p.stage_bytes;
        mbar_arrive_expect_tx(full, bytes);
        for (int m = 0; m < MB; ++m)
          tma_load_4d_hint(dst + m * NW_W_BYTES, &tm_w, (w.kb & 1) * 64, 0, w.kb >> 1, (w.r * MB + m) * (128 / RB),
                           full, pol);
        next(w);
      };
      auto tokens = [&]() {
        tma_load_3d(ring + x.s * p.stage_bytes + x_off, &tm_x, x.kb * 64, x.t * p.tp, 0, smem_addr(&s_full[x.s]));
        next(x);
      };
      const int total = (int)(u1 - u0), lead = min(total, p.stages);
      for (int i = 0; i < lead; ++i) weights();
      pdl_wait();
      asm volatile("fence.proxy.async;" ::: "memory");  // the previous kernel's stores, before TMA reads them
      for (int i = 0; i < lead; ++i) tokens();
      bool ok = true;
      for (int i = lead; i < total; ++i) {
        if (*abort_flag || !mbar_wait(smem_addr(&s_empty[w.s]), (uint32_t)(w.use - 1) & 1)) {
          ok = false;
          break;
        }
        weights();
        tokens();
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(ep.err, ERR_TIMEOUT);
        // let the copies in flight land: stage s was last filled in its use number w.use - (s >= w.s)
        for (int s = 0; s < p.stages; ++s) {
          const int last = w.use - (s >= w.s ? 1 : 0);
          if (last >= 0) mbar_wait(smem_addr(&s_full[s]), (uint32_t)last & 1);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---- MMA issuer (the whole warp, one elected lane issuing): segment i of the range (one row
    // tile's share) accumulates into buffer i % bufs
    const uint32_t idesc = idesc_kind_f16(128, p.tp * p.terms, !ep.f16);
    int s = 0, left = (int)(u1 - u0), n = p.n_kb - (int)(u0 % p.n_kb);
    uint32_t use = 0;
    bool ok = true;
    for (int seg = 0; left > 0 && ok; ++seg, n = p.n_kb) {
      n = min(n, left);
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
#pragma unroll
          for (int k = 0; k < 4; ++k)  // 16 K values further: 32 bytes, 2 in the descriptor's units
#pragma unroll
            for (int m = 0; m < MB; ++m)
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
    // ---- epilogue warps: TMEM lanes 32 q .. (q = warp % 4) are 32 consecutive rows of the tile;
    // the two warps of a quadrant take alternate groups of 16 tokens
    pdl_wait();  // h, the partial sums and the outputs may still be in use by the previous kernel
    const int q = warp & 3, grp = (warp - 2) >> 2, row = 32 * q + lane;
    const int groups = p.tp / 16;
    const size_t part = (size_t)MB * p.tp * 128;  // floats of one partial
    int seg = 0;
    for (long long u = u0; u < u1; ++seg) {
      const int tile = (int)(u / p.n_kb);
      const long long t_lo = (long long)tile * p.n_kb, t_hi = t_lo + p.n_kb, end = min(u1, t_hi);
      const int buf = p.bufs == 2 ? seg & 1 : 0;
      const bool ready = named_bar_and(
          1, NW_EPI_THREADS,
          !*abort_flag && mbar_wait(smem_addr(&s_acc_full[buf]), (uint32_t)(p.bufs == 2 ? seg >> 1 : seg) & 1));
      if (!ready) {
        if (lane == 0) {
          *abort_flag = 1;
          atomicOr(ep.err, ERR_TIMEOUT);
        }
        break;
      }
      tc_fence_after();
      const bool whole = u == t_lo && end == t_hi;
      const int r_tile = tile / p.t_tiles, tt0 = (tile % p.t_tiles) * p.tp;
      for (int m = 0; m < MB; ++m) {
        const int n = (r_tile * MB + m) * 128 + row;
        for (int gr = grp; gr < groups; gr += 2) {
          const int t0 = tt0 + gr * 16;
          if (t0 >= ep.T) break;
          NarrowEpilogue<MODE> e;
          if (whole) e.load(ep, n, t0, lane);
          const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((buf * MB + m) * p.acc_cols + gr * 16);
          uint32_t r0[16], r1[16], r2[16];
          tmem_ld16(ta, r0);
          tmem_ld16(ta + p.tp, r1);
          if (p.terms == 3) tmem_ld16(ta + 2 * p.tp, r2);
          tmem_wait_ld();
          float v[16];
          // the smaller terms first
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float lo = p.terms == 3 ? __uint_as_float(r1[j]) + __uint_as_float(r2[j]) : __uint_as_float(r1[j]);
            v[j] = __uint_as_float(r0[j]) + lo;
          }
          if (whole) {
            e.store(ep, n, t0, v, lane, (r_tile * MB + m) * 4 + q);
          } else {
            // this CTA's slot 0: the range starts inside the tile; slot 1: it ends inside
            float4 *w = reinterpret_cast<float4 *>(p.ws + ((size_t)blockIdx.x * 2 + (u > t_lo ? 0 : 1)) * part) +
                        (size_t)(m * groups + gr) * 4 * 128 + row;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j * 128] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_addr(&s_acc_empty[buf]));
      if (!whole) {
        // the CTAs that share the tile are first .. last; the last to take the ticket sums their
        // partials in CTA order, four partials (256 bytes a thread) in flight
        const int first = (int)(((t_lo + 1) * G - 1) / U), last = (int)((t_hi * G - 1) / U);
        const int slot0 = first * U / G > t_lo ? 0 : 1;  // of CTA `first`; the others start inside the tile
        named_bar_sync(1, NW_EPI_THREADS);
        if (threadIdx.x == 64) {
          const unsigned old = atom_add_acq_rel(p.tickets + tile, 1u);
          s_last = old == (unsigned)(last - first);
          if (s_last) p.tickets[tile] = 0;
        }
        named_bar_sync(1, NW_EPI_THREADS);
        if (s_last) {
          for (int m = 0; m < MB; ++m) {
            const int n = (r_tile * MB + m) * 128 + row;
            for (int gr = grp; gr < groups; gr += 2) {
              const int t0 = tt0 + gr * 16;
              if (t0 >= ep.T) break;
              const float4 *at = reinterpret_cast<const float4 *>(p.ws) + (size_t)(m * groups + gr) * 4 * 128 + row;
              NarrowEpilogue<MODE> e;
              e.load(ep, n, t0, lane);
              float v[16] = {};
              for (int c = first; c <= last; c += 4) {
                float4 x[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const float4 *w = at + ((size_t)(c + i) * 2 + (c + i == first ? slot0 : 0)) * (part / 4);
#pragma unroll
                  for (int j = 0; j < 4; ++j)
                    x[i][j] = c + i <= last ? __ldcg(w + j * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                  for (int j = 0; j < 4; ++j) {
                    v[4 * j] += x[i][j].x;
                    v[4 * j + 1] += x[i][j].y;
                    v[4 * j + 2] += x[i][j].z;
                    v[4 * j + 3] += x[i][j].w;
                  }
              }
              e.store(ep, n, t0, v, lane, (r_tile * MB + m) * 4 + q);
            }
          }
        }
        named_bar_sync(1, NW_EPI_THREADS);  // s_last is read by all before the next segment writes it
      }
      u = end;
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
  // two slots per CTA of 256 rows x tp tokens
  return (size_t)n_sm * 2 * 256 * std::min(NW_MAX_TP, (T + 15) / 16 * 16) * sizeof(float);
}
int narrow_max_tiles(int N) { return (N + 127) / 128; }

template <int MODE, int MB>
static cudaError_t launch_narrow_mode(const CUtensorMap &w, const CUtensorMap &x, const NarrowParams &p, int grid,
                                      const PrefillEpiParams &ep, cudaStream_t s) {
  static bool set = false;
  if (!set) {
    const cudaError_t e =
        cudaFuncSetAttribute(prefill_narrow_kernel<MODE, MB>, cudaFuncAttributeMaxDynamicSharedMemorySize, NW_SMEM);
    if (e != cudaSuccess) return e;
    set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NW_THREADS);
  cfg.dynamicSmemBytes = NW_SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  pdl_attribute(attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, prefill_narrow_kernel<MODE, MB>, w, x, p, ep);
}

int narrow_tp(int T, int terms) {
  return std::min((T + 15) / 16 * 16, terms == 2 ? NW_MAX_TP : 80);  // terms * tp <= 256 MMA columns
}

cudaError_t launch_prefill_narrow(int mode, const CUtensorMap &w, const CUtensorMap &x, int K, int terms,
                                  const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s) {
  if (ep.T <= 0 || ep.N <= 0) return cudaSuccess;
  NarrowParams p = {};
  p.terms = terms;
  p.tp = narrow_tp(ep.T, terms);
  p.t_tiles = (ep.T + p.tp - 1) / p.tp;
  if (mode == PE_ARGMAX && p.t_tiles != 1) return cudaErrorInvalidValue;
  const int cols = p.tp * terms;
  // wide tiles of many rows share their tokens' slices between two 128-row blocks: the slices (2 x
  // 16 KiB of terms at 128 tokens) then cost no more L2 reads than the weights
  const int mb = cols > 128 && (ep.N + 255) / 256 * p.t_tiles >= ws.n_sm * 3 / 4 ? 2 : 1;
  p.n_kb = (K + 63) / 64;
  p.n_tiles = (ep.N + 128 * mb - 1) / (128 * mb) * p.t_tiles;
  p.acc_cols = (cols + 31) / 32 * 32;
  p.bufs = 2 * mb * p.acc_cols <= 512 ? 2 : 1;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.bufs * mb * p.acc_cols) p.tmem_cols *= 2;
  p.stage_bytes = mb * NW_W_BYTES + cols * 128;
  p.stages = std::min(NW_MAX_STAGES, (NW_SMEM - 1024) / p.stage_bytes);
  p.ws = ws.partial;
  p.tickets = ws.tickets;
  // at least four K blocks per CTA: finer splits cost more in partial sums than they stream sooner
  const long long U = (long long)p.n_tiles * p.n_kb;
  const int grid = (int)std::min<long long>(ws.n_sm, std::max<long long>(std::min<long long>(p.n_tiles, ws.n_sm), U / 4));
  auto go = [&](auto m) {
    constexpr int MODE = decltype(m)::value;
    return mb == 2 ? launch_narrow_mode<MODE, 2>(w, x, p, grid, ep, s) : launch_narrow_mode<MODE, 1>(w, x, p, grid, ep, s);
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

}  // namespace kfl
