// Internal definitions of the dense prompt prefill (sm_103a only): a tcgen05 GEMM over the
// prompt's tokens with fused epilogues, causal attention over the cache, row RMSNorm.
#pragma once

#include <cuda.h>  // CUtensorMap (the type only; maps are encoded through the runtime's entry point)

#include <atomic>

#include "common.cuh"

namespace kfl {

// ---- the prefill GEMM: Y[T][N] = X[T][K] W[N][K]^T ------------------------------------------
// X is fp32 in meaning and given as two bf16 terms, X = Xhi + Xlo (Xhi = bf16(X), Xlo =
// bf16(X - Xhi), about 2^-16 relative error left), so that the products keep the accuracy of the
// decode path's fp32 activations; W is bf16 as stored (int4 stages: fp16 tiles dequantized from
// the int4 ones, with fp16 terms of X).  An output tile is PG_M tokens x PG_N weight rows,
// computed with tcgen05.mma (M = PG_M, N = PG_N, K = 16 per instruction; each K slice once with
// Xhi and once with Xlo against the same W slice), the fp32 accumulator in tensor memory, by a
// persistent CTA per SM with two accumulators (prefill_gemm_persistent).  Operands reach shared memory
// by TMA with the 128-byte swizzle, PG_K = 64 bf16 (one swizzle row) per pipeline stage: Xhi and Xlo
// through 2-D maps of the activation rows, W through a 4-D map of the decode path's weight tiles
// [N/RB][K/KT][RB][KT] (one box = PG_N / RB row blocks x 64 columns of one K tile), so the prefill
// streams the weights from where the decode step reads them.
constexpr int PG_M = 128;
constexpr int PG_N = 256;
constexpr int PG_K = 64;
constexpr int PG_STAGES = 3;
constexpr int PG_A_BYTES = PG_M * PG_K * 2;  // 16 KiB per term
constexpr int PG_B_BYTES = PG_N * PG_K * 2;  // 32 KiB
constexpr size_t PG_SMEM = (size_t)PG_STAGES * (2 * PG_A_BYTES + PG_B_BYTES) + 1024;  // + alignment slack

enum PrefillEpi : int {
  PE_STORE = 0,   // out[t][n] = y
  PE_RESID = 1,   // out[t][n] += y (the residual stream)
  PE_SWIGLU = 2,  // columns (2j, 2j+1) = (gate j, up j): silu(g) u as hi/lo terms -> out16, out16lo
  PE_QKV = 3,     // Q/K/V rows in the decode path's order: RoPE, q -> out16, k and v -> KV cache
  PE_ARGMAX = 4,  // per (token, column tile): the largest y and its lowest index
};

struct PrefillEpiParams {
  int T, N;                // valid tokens and columns
  int f16;                 // operands are fp16 (int4 stages: weights dequantized to fp16), else bf16
  float *out;              // PE_STORE / PE_RESID: fp32 [T][ldo]
  int ldo;
  uint16_t *out16;         // PE_SWIGLU: hi term, bf16 [T][ldo16] (N / 2 columns); PE_QKV: q, bf16 [T][ldo16]
  uint16_t *out16lo;       // PE_SWIGLU: lo term, same layout (out16 + term_stride)
  int ldo16;
  int terms;               // PE_SWIGLU: terms stored, term_stride elements apart
  size_t term_stride;
  // PE_QKV (out not NULL: q in fp32 to out [T][ldo] instead of out16): rows [0, qdim) q, [qdim, qdim +
  // kvdim) k (pairs (i, i + hd/2) adjacent per head, as the weights were loaded), then v in natural order; K/V stored at the token's position of
  // KV slot `slot` of this layer's caches [max_batch][Hkv][max_ctx][hd]
  uint16_t *kcache, *vcache;
  const int *positions;    // [T], -1 for a refused token (nothing of it is stored)
  int slot, hd, hkv, qdim, kvdim, max_ctx;
  const float *rope_cos, *rope_sin;  // [max_ctx][hd / 2]
  // PE_ARGMAX: [T][n_tiles] partial maxima (of 256 columns, or of 32 rows in the few-token GEMM) and
  // their indices
  float *amax;
  int *aidx;
  int n_tiles;
  unsigned *err;           // ERR_TIMEOUT if a pipeline wait gave up; ERR_F16_RANGE (PE_SWIGLU, fp16
                           // terms) if a value is beyond the fp16 range
};

struct PrefillAttnParams {
  const uint16_t *q;       // [T][ldq] bf16, RoPE applied, heads in natural order
  const float *q32;        // not NULL: q in fp32 instead, carried (like the softmax weights) as bf16 pairs
  int ldq;
  uint16_t *o;             // [T][ldo]: the output as 2 or 3 terms, term_stride apart (fp16 if f16, else bf16)
  int ldo, f16, terms;
  size_t term_stride;
  const uint16_t *kcache, *vcache;  // this layer's [max_batch][Hkv][max_ctx][hd]
  const int *positions;    // [T], -1: refused (output 0)
  int slot, T, n_heads, n_kv_heads, max_ctx;
  float scale_log2;        // log2(e) / sqrt(hd)
  unsigned *err;           // ERR_F16_RANGE if an fp16 output term cannot hold its value
};

// ---- the prefill GEMM of few tokens (prefill_narrow.cu): weight rows as M, the tokens' terms
// side by side as N, split stream-K over one CTA per SM
constexpr int NW_MAX_TP = 128;            // tokens of a tile (two terms: 256 MMA columns)
constexpr int NW_PARTS = 3;               // partial sums per CTA in a GEMM's workspace
constexpr int N4_MAX_TOKENS = 512;        // int4 stages: the longest passes that decode in the GEMM
constexpr int NW_W_BYTES = 128 * 64 * 2;  // a 128-row weight slice of 64 K
// How a GEMM's output tiles are shared out (share_tiles, TileWalk in prefill_tc.cuh).
struct TileShare {
  int n_kb, waves, tail, splits;
  bool cut() const { return tail > 0 && splits != 1; }
};
// Partial sums of a residual GEMM's cut tiles that nothing has added to h yet: the RMSNorm behind it does
// (launch_narrow_norm).
struct NarrowPending {
  bool any = false;
  TileShare share = {};
  int grid = 0, mb = 0, tp = 0, t_tiles = 0;
  const float *ws = nullptr;
};
struct NarrowWorkspace {
  float *partial;  // narrow_ws_bytes
  int n_sm;
};
size_t narrow_ws_bytes(int n_sm, int T);  // for passes of up to T tokens
int narrow_argmax_slots(int N);  // PE_ARGMAX: partial maxima per token (n_tiles of PrefillEpiParams)
int narrow_tp(int T, int terms);  // tokens of a tile
// w: encode_tiles_map with 2 row blocks per box, or (w_rows) encode_rows_map with 128 rows; x:
// encode_terms_map with narrow_tp rows per box.  early: w was written by nothing later than the kernel
// before the last, so that the kernel may read it before it waits for the last.
cudaError_t launch_prefill_narrow(int mode, const CUtensorMap &w, bool w_rows, const CUtensorMap &x, int K, int terms,
                                  const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s,
                                  NarrowPending *pending = nullptr, bool early = true);
// The same over int4 tiles [n_rb][n_kt][TILE4_BYTES], decoded in the kernel (fp16 terms).
cudaError_t launch_prefill_narrow4(int mode, const uint8_t *tiles, int n_rb, int n_kt, const CUtensorMap &x, int K,
                                   int terms, const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s,
                                   NarrowPending *pending = nullptr);
// RMSNorm (as launch_prefill_rmsnorm) of h after adding the pending sums to it.  d up to NW_NORM_MAX_D.
constexpr int NW_NORM_MAX_D = 32768;
cudaError_t launch_narrow_norm(const NarrowPending &pend, float *h, int ldh, int T, int d, const float *g, float eps,
                               uint16_t *x, size_t term_stride, int terms, int ldx, int f16, unsigned *err,
                               cudaStream_t s);

// Host side (prefill.cu).
// cudaMalloc, once more without what kfl_matmul_bf16w keeps if there is no memory.
bool device_alloc(void **p, size_t bytes);
int encode_act_map(CUtensorMap *map, const uint16_t *base, int K, int rows, int ld);
// The terms of activation rows [term][rows][K] (row stride ld, term stride term_stride elements):
// boxes of 64 columns x box_rows rows x every term.
int encode_terms_map(CUtensorMap *map, const uint16_t *base, int K, int rows, int ld, int terms, size_t term_stride,
                     int box_rows);
int encode_tiles_map(CUtensorMap *map, const uint8_t *tiles, int n_kt, int n_rb, int box_rb);
// A row-major bf16 matrix [N][K] (K a multiple of 8, 16-byte aligned): boxes of 64 columns x box_rows rows.
int encode_rows_map(CUtensorMap *map, const uint16_t *w, int K, int N, int box_rows);
// Opts a kernel in to its dynamic shared memory before a launch.  The attribute holds for the device it
// was set on, so it is set once on each (a bit per device; beyond 64, at every launch); a failure is not
// remembered.  One per kernel, shared by every thread.
class SmemOptIn {
  std::atomic<uint64_t> done_{0};

 public:
  cudaError_t operator()(const void *kernel, int bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;
    if (done_.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_relaxed);
    return e;
  }
};
// The launch attribute of a kernel that waits (griddepcontrol.wait) for the kernel before it.
inline void pdl_attribute(cudaLaunchAttribute &a) {
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
}
// b: encode_tiles_map with PG_N / RB row blocks per box, or (w_rows) encode_rows_map with PG_N rows.
cudaError_t launch_prefill_gemm(int mode, const CUtensorMap &a_hi, const CUtensorMap &a_lo, const CUtensorMap &b,
                                bool w_rows, int K,
                                const NarrowWorkspace &ws, const PrefillEpiParams &ep, cudaStream_t s);
cudaError_t launch_prefill_attention(const PrefillAttnParams &p, int hd, int n_sm, cudaStream_t s);
cudaError_t launch_prefill_input(const int *ids, const float *hidden_in, const int *positions_in, int T,
                                 const uint16_t *embed, int vocab, int d, int ldh, float *h, int *positions,
                                 int max_ctx, int user, int *slots, unsigned *err, cudaStream_t s);
cudaError_t launch_prefill_rmsnorm(const float *h, int ldh, int T, int d, const float *g, float eps, uint16_t *x,
                                   size_t term_stride, int terms, int ldx, int f16, unsigned *err, cudaStream_t s);
// int4 group-64 tiles [n_rb][n_kt][TILE4_BYTES] -> fp16 tiles [n_rb][2 n_kt][RB][KT] of code x scale.
cudaError_t launch_dequant_int4_f16(const uint8_t *tiles4, int n_rb, int n_kt, uint16_t *dst, int n_sm,
                                    cudaStream_t s);
// fp32 rows [T][K] (stride ldx) as hi and lo bf16 terms (stride ld); *err = 0.
cudaError_t launch_split_bf16(const float *x, int T, int K, int ldx, uint16_t *hi, uint16_t *lo, int ld, unsigned *err,
                              cudaStream_t s);
cudaError_t launch_prefill_argmax(const float *amax, const int *aidx, int n_tiles, int T, int *next_ids,
                                  cudaStream_t s);

}  // namespace kfl
