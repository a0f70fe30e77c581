// tcgen05 / TMA building blocks of the prefill kernels (sm_103a): tensor memory, shared-memory and
// instruction descriptors, tensor copies, and activations as 16-bit terms.
#pragma once

#include <cmath>

#include "prefill.cuh"

namespace kfl {

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Tensor-memory allocation by one whole warp; the base address is written to shared memory.
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// Shared-memory matrix descriptor of a K-major operand in the 128-byte swizzled layout: rows of
// 128 bytes (64 bf16 of K), groups of 8 rows 1024 bytes apart (the stride byte offset); the
// leading byte offset is unused in this layout (1 by convention); descriptor version 1; swizzle
// mode 2 (128 bytes).  A slice of 16 K values starts 32 bytes further within the row.
__device__ __forceinline__ uint64_t sdesc_k_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of kind::f16: fp32 accumulator (bits 4-5 = 1), A and B both bf16 (bits
// 7-9 and 10-12 = 1) or both fp16 (0), both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22,
// M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_kind_f16(int m, int n, bool bf16) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16_ss(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive on an mbarrier of this CTA once every MMA this thread issued before has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

// 32 consecutive fp32 columns of this thread's tensor-memory lane (warp w reads lanes 32 w ..).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 columns; the registers are there after tmem_wait_ld.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

// The same with an L2 policy.
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                                 uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  return (uint32_t)f32_to_bf16_rne(lo) | ((uint32_t)f32_to_bf16_rne(hi) << 16);
}

// x as two bf16 terms: hi = bf16(x), lo = bf16(x - hi) (the difference is exact in fp32).
__device__ __forceinline__ void split_bf16(float x, uint16_t &hi, uint16_t &lo) {
  hi = f32_to_bf16_rne(x);
  lo = f32_to_bf16_rne(x - bf16_to_f32(hi));
}
// The same with fp16 terms (about 2^-22 relative left; |x| must stay below 65504).
__device__ __forceinline__ void split_f16(float x, uint16_t &hi, uint16_t &lo) {
  hi = f32_to_f16_rn(x);
  lo = f32_to_f16_rn(x - f16_to_f32(hi));
}
__device__ __forceinline__ void split_term(float x, uint16_t &hi, uint16_t &lo, int f16) {
  if (f16)
    split_f16(x, hi, lo);
  else
    split_bf16(x, hi, lo);
}
// x as `terms` (2 or 3) terms: each the rounding of what the ones before left over.
__device__ __forceinline__ void split_terms(float x, uint16_t (&t)[3], int terms, int f16) {
  split_term(x, t[0], t[1], f16);
  if (terms == 3) {
    const float r = f16 ? x - f16_to_f32(t[0]) - f16_to_f32(t[1]) : x - bf16_to_f32(t[0]) - bf16_to_f32(t[1]);
    t[2] = f16 ? f32_to_f16_rn(r) : f32_to_bf16_rne(r);
  }
}
// ---- int4 weights as fp16 MMA operands
__device__ __forceinline__ void stsm_x4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2),
               "r"(r3)
               : "memory");
}
__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t hfma2(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// The eight codes of an A-fragment word as exact fp16 pairs: rows gid and gid + 8 of columns 2 tig,
// 2 tig + 1 (c0, c1) and of columns 2 tig + 8, 2 tig + 9 (c2, c3).  The nibbles, top bit flipped, become
// 1024 + u or 1024 + 16 u (u = code + 8): integers placed in the mantissa of fp16 1024, as published by
// Kim, Henry, Fahim and Awadalla, "Who Says Elephants Can't Run" (arXiv 2211.10017).
__device__ __forceinline__ void decode_word(uint32_t w, uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3) {
  const uint32_t w8 = w >> 8;
  asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(c0) : "r"(w), "r"(0x000F000Fu), "r"(0x64086408u));
  asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(c1) : "r"(w8), "r"(0x000F000Fu), "r"(0x64086408u));
  asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(c2) : "r"(w), "r"(0x00F000F0u), "r"(0x64806480u));
  asm("lop3.b32 %0, %1, %2, %3, 0x6A;" : "=r"(c3) : "r"(w8), "r"(0x00F000F0u), "r"(0x64806480u));
  c0 = hfma2(c0, 0x3C003C00u, 0xE408E408u);  // - 1032
  c1 = hfma2(c1, 0x3C003C00u, 0xE408E408u);
  c2 = hfma2(c2, 0x2C002C00u, 0xD480D480u);  // / 16 - 72
  c3 = hfma2(c3, 0x2C002C00u, 0xD480D480u);
}

// fp16 pair of codes times an fp32 scale, rounded once.
__device__ __forceinline__ uint32_t scale_pair_f32(uint32_t c, float sc) {
  return (uint32_t)f32_to_f16_rn(f16_to_f32((uint16_t)c) * sc) |
         ((uint32_t)f32_to_f16_rn(f16_to_f32((uint16_t)(c >> 16)) * sc) << 16);
}

// The bf16 scales of rows gid and gid + 8 of a weight group, applied to decode_word's codes.
struct ScalePair {
  float s0, s1;
  uint32_t p0, p1;
  __device__ __forceinline__ explicit ScalePair(uint32_t sc) : s0(bf16_lo(sc)), s1(bf16_hi(sc)) {
    p0 = f32_to_f16_rn(s0) * 0x10001u;
    p1 = f32_to_f16_rn(s1) * 0x10001u;
  }
  // scales that fp16 holds exactly: the fp16 product of code and scale is rounded as the fp32 product
  // would be; others (below 2^-14, or too large) go through fp32
  __device__ __forceinline__ bool exact() const {
    return f16_to_f32((uint16_t)p0) == s0 && f16_to_f32((uint16_t)p1) == s1;
  }
  __device__ __forceinline__ void apply(bool exact, uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3) const {
    if (exact) {
      c0 = hmul2(c0, p0), c1 = hmul2(c1, p1), c2 = hmul2(c2, p0), c3 = hmul2(c3, p1);
    } else {
      c0 = scale_pair_f32(c0, s0), c1 = scale_pair_f32(c1, s1);
      c2 = scale_pair_f32(c2, s0), c3 = scale_pair_f32(c3, s1);
    }
  }
};

// How the CTAs of a GEMM share its output tiles (each n_kb K blocks long).  Whole tiles first, tile
// c + i G to CTA c, for `waves` rounds: the CTAs at work together then read few weight rows and few
// tokens, at the same K, from L2.  The `tail` tiles left over would leave SMs idle in a last round:
//  - splits = 0 (one token tile: the weights pass through L2 once, whatever the order): as one
//    sequence of K blocks of which CTA c takes [c U / G, (c + 1) U / G), an equal share to the block; the
//    last whole round joins it, so that no tile is cut more than about twice more than it must be;
//  - splits = S: every tail tile's K in S parts, part p of all tiles before part p + 1 of any, so that
//    CTAs at work together still read the same K (the sequence had each at a K of its own: 2048
//    tokens' down projection, 290 MB of weights and tokens, went from 201 to 281 us).
// A cut tile is summed from its partial sums, in K order, by a kernel behind the GEMM.
// parts_per_cta: how many partial sums per CTA the workspace holds (2 for the sequence).
inline TileShare share_tiles(int tiles, int n_kb, int grid, bool sequence, int parts_per_cta) {
  TileShare s = {n_kb, tiles / grid, tiles % grid, 1};
  if (s.tail == 0) return s;
  // (the device's arithmetic on the sequence is 32-bit: a 64-bit division is a microsecond's start)
  if (sequence && (long long)(tiles % grid + grid) * n_kb * grid < (1ll << 31)) {
    s.splits = 0;
    if (s.waves > 0) --s.waves, s.tail += grid;
    return s;
  }
  // in K blocks' time: rounds of parts, a few blocks' worth of ring refill per round, and for cut tiles
  // the kernel that sums them (its launch, and 256 KB written and read per part)
  double best = 1e30;
  for (int S = 1; S <= 8 && S * 4 <= n_kb && (S == 1 || S * s.tail <= parts_per_cta * grid); ++S) {
    const int rounds = (s.tail * S + grid - 1) / grid;
    const double t = rounds * ((n_kb + S - 1) / S + 2.0) + (S > 1 ? 10.0 + s.tail * S / 12.0 : 0.0);
    if (t < best) best = t, s.splits = S;
  }
  return s;
}
// One CTA's segments in order: K blocks [kb0, kb1) of `tile`; `part`: its place among the partial sums.
struct TileWalk {
  TileShare s;
  int i, tile, kb0, kb1, part;
  unsigned u, u1;
  __device__ __forceinline__ explicit TileWalk(const TileShare &share) : s(share), i(0) {
    const unsigned U = s.splits == 0 ? s.tail * s.n_kb : 0;
    u = blockIdx.x * U / gridDim.x;
    u1 = (blockIdx.x + 1) * U / gridDim.x;
  }
  __device__ __forceinline__ bool next() {
    if (i < s.waves) {
      tile = blockIdx.x + i * gridDim.x;
      kb0 = 0;
      kb1 = s.n_kb;
    } else if (s.splits > 0) {
      part = blockIdx.x + (i - s.waves) * gridDim.x;
      if (part >= s.tail * s.splits) return false;
      const int sp = part / s.tail;
      tile = s.waves * gridDim.x + part - sp * s.tail;
      kb0 = sp * s.n_kb / s.splits;
      kb1 = (sp + 1) * s.n_kb / s.splits;
    } else {
      if (u >= u1) return false;
      const unsigned t = u / (unsigned)s.n_kb;
      tile = s.waves * gridDim.x + t;
      kb0 = (int)(u - t * s.n_kb);
      kb1 = min(s.n_kb, kb0 + (int)(u1 - u));
      part = blockIdx.x * 2 + (kb0 > 0 ? 0 : 1);
      u += kb1 - kb0;
    }
    ++i;
    return true;
  }
  __device__ __forceinline__ bool whole() const { return kb0 == 0 && kb1 == s.n_kb; }
};
// The partial sums of tail tile k, in K order.
struct TileParts {
  int n, at, step, rest;  // part i: i == 0 ? at : rest + i * step
  TileParts() = default;
  __device__ __forceinline__ TileParts(const TileShare &s, int k, int grid) {
    if (s.splits > 0) {
      n = s.splits;
      at = rest = k;
      step = s.tail;
    } else {
      // the CTAs first .. last meet the tile; every one but the first starts inside it (partial 0), the
      // first comes to its start (partial 1)
      const unsigned U = s.tail * s.n_kb, G = grid, lo = k * s.n_kb;
      const int first = (int)(((lo + 1) * G - 1) / U), last = (int)(((lo + s.n_kb) * G - 1) / U);
      n = last - first + 1;
      at = first * 2 + 1;
      rest = first * 2;
      step = 2;
    }
  }
  __device__ __forceinline__ int part(int i) const { return i == 0 ? at : rest + i * step; }
};

// Two values as packed pairs of their hi and lo terms.  fp16 terms of a value that fp16 cannot
// hold (|x| >= 65520 rounds to infinity, or not finite) set ERR_F16_RANGE in *err.
__device__ __forceinline__ void split_pack(float x0, float x1, uint32_t &hi, uint32_t &lo, int f16 = 0,
                                           unsigned *err = nullptr) {
  if (f16 && err && !(fabsf(x0) < 65520.f && fabsf(x1) < 65520.f)) atomicOr(err, ERR_F16_RANGE);
  uint16_t h0, l0, h1, l1;
  split_term(x0, h0, l0, f16);
  split_term(x1, h1, l1, f16);
  hi = (uint32_t)h0 | ((uint32_t)h1 << 16);
  lo = (uint32_t)l0 | ((uint32_t)l1 << 16);
}

// What rounding leaves out of the fp32 product a * b * c (to first order).
__device__ __forceinline__ float product3_rest(float a, float b, float c) {
  const float p = a * b;
  return fmaf(fmaf(a, b, -p), c, fmaf(p, c, -(p * c)));
}

// The block's sum of v (whole warps; red: a float per warp).
__device__ __forceinline__ float block_sum(float v, float *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
  __syncthreads();
  v = threadIdx.x % 32 < blockDim.x / 32 ? red[threadIdx.x % 32] : 0.f;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Four consecutive normalised values v * inv * g as 16-bit terms, term_stride elements apart (x 8-byte
// aligned).
__device__ __forceinline__ void store_normed(float4 v, float inv, float4 g, uint16_t *x, size_t term_stride, int terms,
                                             int f16, unsigned *err) {
  uint2 hi, lo;
  const float y0 = v.x * inv * g.x, y1 = v.y * inv * g.y, y2 = v.z * inv * g.z, y3 = v.w * inv * g.w;
  split_pack(y0, y1, hi.x, lo.x, f16, err);
  split_pack(y2, y3, hi.y, lo.y, f16, err);
  *reinterpret_cast<uint2 *>(x) = hi;
  *reinterpret_cast<uint2 *>(x + term_stride) = lo;
  if (terms == 3)  // bf16 terms: what the first two, and the products' roundings, leave
    *reinterpret_cast<uint2 *>(x + 2 * term_stride) =
        make_uint2(pack_bf16(y0 - bf16_lo(hi.x) - bf16_lo(lo.x) + product3_rest(v.x, inv, g.x),
                             y1 - bf16_hi(hi.x) - bf16_hi(lo.x) + product3_rest(v.y, inv, g.y)),
                   pack_bf16(y2 - bf16_lo(hi.y) - bf16_lo(lo.y) + product3_rest(v.z, inv, g.z),
                             y3 - bf16_hi(hi.y) - bf16_hi(lo.y) + product3_rest(v.w, inv, g.w)));
}

}  // namespace kfl
