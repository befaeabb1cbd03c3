// GEMM epilogues: TMEM -> registers -> fused element-wise work -> global memory.
// Each epilogue thread owns one accumulator row (TMEM lane) of a 128 x BN tile and walks its
// columns 32 at a time.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <utility>

#include "tc_gemm.cuh"

namespace still {

// Element offset of (batch b, row r, column c) as an affine function of their div/mod parts.
struct AffineMap {
  int32_t bdiv = 1, rdiv = 1 << 30, cdiv = 1 << 30;
  int64_t b1 = 0, b0 = 0, r1 = 0, r0 = 0, c1 = 0, c0 = 0, k = 0;
  __device__ __forceinline__ int64_t at(int b, int r, int c) const {
    return (int64_t)(b / bdiv) * b1 + (int64_t)(b % bdiv) * b0 + (int64_t)(r / rdiv) * r1 +
           (int64_t)(r % rdiv) * r0 + (int64_t)(c / cdiv) * c1 + (int64_t)(c % cdiv) * c0 + k;
  }
};

// OUT_HILO: bf16 hi and lo = bf16(x - hi); OUT_HILO16: the same in fp16 (about 22 bits).
enum OutKind : int32_t { OUT_F32 = 0, OUT_BF16 = 1, OUT_HILO = 2, OUT_HILO16 = 3 };

__device__ __forceinline__ void split_hilo(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// GELU with the exact (erf) form, 0.5 x (1 + erf(x / sqrt 2)) (App. A, Feed-forward).
__device__ __forceinline__ float gelu_erf(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);  // a -> low half, b -> high half
  return *reinterpret_cast<uint32_t*>(&v);
}

// hi/lo split of two values, packed: hi = bf16(x), lo = bf16(x - hi)
__device__ __forceinline__ void split_pack(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// hi/lo split of two values in fp16 (11-bit significands: about 22 bits together):
// hi = fp16(x), lo = fp16(x - hi), packed.
__device__ __forceinline__ void split_pack_f16(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// The same of a packed fp32 pair, in fp16 or bf16.
template <bool F16>
__device__ __forceinline__ void split2(uint64_t v, uint32_t& hi, uint32_t& lo) {
  float a, b;
  unpack2(v, a, b);
  if constexpr (F16)
    split_pack_f16(a, b, hi, lo);
  else
    split_pack(a, b, hi, lo);
}

// 32 floats -> 32 bf16 packed in 4 x uint4
__device__ __forceinline__ void pack_bf16x32(const float (&v)[32], uint4 (&o)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    o[q] = make_uint4(pack_bf16x2(v[8 * q], v[8 * q + 1]), pack_bf16x2(v[8 * q + 2], v[8 * q + 3]),
                      pack_bf16x2(v[8 * q + 4], v[8 * q + 5]),
                      pack_bf16x2(v[8 * q + 6], v[8 * q + 7]));
}

// 32 floats -> hi and lo bf16, each packed in 4 x uint4
__device__ __forceinline__ void pack_hilo_x32(const float (&v)[32], uint4 (&h4)[4],
                                              uint4 (&l4)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) split_pack(v[8 * q + 2 * k], v[8 * q + 2 * k + 1], h[k], l[k]);
    h4[q] = make_uint4(h[0], h[1], h[2], h[3]);
    l4[q] = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

__device__ __forceinline__ void pack_hilo16_x32(const float (&v)[32], uint4 (&h4)[4],
                                                uint4 (&l4)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) split_pack_f16(v[8 * q + 2 * k], v[8 * q + 2 * k + 1], h[k], l[k]);
    h4[q] = make_uint4(h[0], h[1], h[2], h[3]);
    l4[q] = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

// 16 floats -> 4 x uint4 (fp32 bits)
__device__ __forceinline__ void pack_f32x16(const float* v, uint4 (&o)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    o[q] = make_uint4(__float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                      __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
}

// General epilogue: v = acc * alpha [* colscale(c)] [* rowscale(r)] [+ bias(c)]
//   -> [sum-of-squares partial] -> [GELU] -> [+ residual] -> store (f32/bf16/hi-lo)
// colscale / rowscale are read from vectors of ready factors (see launch_inv_norms).
// Sums of squares are written as partials, never accumulated atomically, so that results do
// not depend on scheduling: per (vector, tile, half-warp) one slot, ss_parts slots per vector.
// Host contract: csm, resm and (when vec_ok) om are contiguous in c (c0 == 1) with cdiv a
// multiple of 32, so every 32-column chunk maps to 32 consecutive elements; ss_seg is a
// multiple of the tile width.
// kChunkSums: one slot per 32-column chunk, so that a tile's chunks may lie in several CTAs, at the
// price of more partials. A type of its own: as a run-time choice it cost the other projections
// 1% to 4%.
template <bool kChunkSums>
struct EpiAffineT {
  static constexpr int kWarps = 8;  // two per lane quarter: alternating 32-column chunks
  static constexpr int kStages = 0;  // default pipeline depth
  int32_t kind = OUT_F32;
  void* out = nullptr;
  int64_t lo_off = 0;  // OUT_HILO: lo element offset from hi
  AffineMap om;
  float alpha = 1.f;
  const float* bias = nullptr;  // indexed by column
  const float* col_scale = nullptr;
  AffineMap csm;  // (b, 0, c) -> index
  const float* row_scale = nullptr;
  AffineMap rsm;  // (b, r, 0) -> index
  int32_t gelu = 0;
  int32_t res_kind = 0;  // 0 none, 1 f32, 2 bf16
  const void* res = nullptr;
  AffineMap resm;
  float* sumsq = nullptr;  // partial sums of v^2 over segments of ss_seg columns
  AffineMap ssm;           // (b, r, c / ss_seg) -> vector index
  int32_t ss_seg = 1 << 30;
  int32_t ss_parts = 2;    // slots per vector: 2 * ss_seg / tile width, kChunkSums ss_seg / 32
  // Vectors in blocks of ss_block consecutive indices, stored part-major (see launch_inv_norms),
  // so that a warp's 32 rows write 32 consecutive floats of one part.
  int64_t ss_block = 1;
  int32_t vec_ok = 0;  // host: om.c0 == 1, cdiv % 32 == 0, 16-B aligned rows
  // OUT_F32 through TMA stores: the output is the 3-D view (col, row, batch) given to the
  // launcher (boxes of 32 x 32 fp32, 128-byte swizzled staging); rows / columns past the view
  // are clipped by the copy engine.
  int32_t tma_f32 = 0;
  // Columns [N, pad_n) of the last tile are stored as zeros (vec_ok outputs only; pad_n a multiple
  // of 32): a last chunk that N ends in then goes out in vectors too. 0: nothing past N.
  int32_t pad_n = 0;
  int32_t tile_cols_ = 256;  // the tile width BN, set by the launcher
  bool can_split() const { return sumsq == nullptr || kChunkSums; }
  static constexpr bool kAnyTile = true;  // its 32-column chunks are independent
  static constexpr bool kPairs = !kChunkSums;  // has a 2-SM form, of these tile widths:
  using Widths = std::integer_sequence<int, 256>;
  // Clocks of the 2-SM form (see gemm2_cost): 720 measured at t = 1024, d_l = 1024.
  static constexpr int pair_wave(int) { return 720; }
  static constexpr int pair_start(int) { return 0; }

  // The residual rows of this warp's columns are pulled into L2 while the main loop runs.
  template <class Src>
  __device__ void prefetch(const GemmParams& p, const TileCoord& tc, int row, const Src& src,
                           int half) const {
    if (res_kind == 0) return;
    const int r = tc.tm * kBM + row;
    if (r >= p.M) return;
    const int esz = res_kind == 1 ? 4 : 2;
    for (int cc = src.first(half); cc < tile_cols_; cc += src.step()) {
      const int c0 = tc.tn * tile_cols_ + cc;
      if (c0 >= p.N) break;
      const char* base = static_cast<const char*>(res) + resm.at(tc.b, r, c0) * esz;
      for (int off = 0; off < 32 * esz; off += 32) prefetch_l2(base + off);  // per 32-B sector
    }
  }

  template <class Src>
  __device__ void operator()(const GemmParams& p, const TileCoord& tc, int row, const Src& src,
                             int half, uint4* stage, const CUtensorMap* tmc) const {
    // A warp whose 32 rows all lie past M has nothing to do. In the warp that M ends in, the
    // lanes past it repeat the last row and store nothing, so that the warp stays converged (on a
    // path of their own they doubled the epilogue of the last row of tiles: q/k projection of
    // 1,000 rows 112 us, of 992 or 1,024 rows 68).
    const int tr = tc.tm * kBM + row;
    if (tr - (int)(threadIdx.x & 31) >= p.M) return;
    const bool rvalid = tr < p.M;
    const int r = min(tr, p.M - 1);
    float rscale = alpha;
    if (row_scale != nullptr) rscale *= row_scale[rsm.at(tc.b, r, 0)];
    float ss = 0.f;
    for (int cc = src.first(half); cc < tile_cols_; cc += src.step()) {
      const int c0 = tc.tn * tile_cols_ + cc;
      if (c0 >= max(p.N, pad_n)) continue;  // uniform across the warp
      float v[32];
      src.load(cc, v);
      const int nv = min(32, p.N - c0);
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] *= rscale;
      if (nv < 32 && pad_n > 0) {
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = e < nv ? v[e] : 0.f;
      }
      // Residual rows read coalesced by the whole warp. Not on the TMA-store path, whose
      // staging area may still be in use.
      const bool res_vec = res_kind != 0 && vec_ok && !tma_f32 && nv == 32;
      float resv[32];
      if (res_vec) {
        const int64_t o = resm.at(tc.b, r, c0);
        if (res_kind == 1) {
          uint4 u[8];
          warp_load_rows<8>(stage, static_cast<const float*>(res) + o, rvalid, u);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            resv[4 * q] = __uint_as_float(u[q].x);
            resv[4 * q + 1] = __uint_as_float(u[q].y);
            resv[4 * q + 2] = __uint_as_float(u[q].z);
            resv[4 * q + 3] = __uint_as_float(u[q].w);
          }
        } else {
          uint4 u[4];
          warp_load_rows<4>(stage, static_cast<const __nv_bfloat16*>(res) + o, rvalid, u);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t w[4] = {u[q].x, u[q].y, u[q].z, u[q].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[k]));
              resv[8 * q + 2 * k] = f.x;
              resv[8 * q + 2 * k + 1] = f.y;
            }
          }
        }
      }
      if (col_scale != nullptr) {
        float cs[32];
        load_cols(col_scale + csm.at(tc.b, 0, c0), nv, 1.f, cs);
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] *= cs[e];
      }
      if (bias != nullptr) {
        float add[32];
        load_cols(bias + c0, nv, 0.f, add);
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] += add[e];
      }
      if (sumsq != nullptr) {
#pragma unroll
        for (int e = 0; e < 32; ++e)
          if (e < nv) ss += v[e] * v[e];
        if constexpr (kChunkSums) {
          if (rvalid) store_sum(tc.b, r, c0, (c0 % ss_seg) / 32, ss);
          ss = 0.f;
        }
      }
      if (gelu) {
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = gelu_erf(v[e]);
      }
      if (res_vec) {
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] += resv[e];
      } else if (res_kind != 0) {
        const int64_t o = resm.at(tc.b, r, c0);
        if (res_kind == 1) {
          const float* rp = static_cast<const float*>(res) + o;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (e < nv) v[e] += rp[e];
        } else {
          const __nv_bfloat16* rp = static_cast<const __nv_bfloat16*>(res) + o;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (e < nv) v[e] += __bfloat162float(rp[e]);
        }
      }
      if (tma_f32)
        store32_tma(tc, row, c0, v, stage, tmc);
      else
        store32(p, tc.b, r, c0, v, rvalid, stage);
    }
    if (!kChunkSums && sumsq != nullptr && rvalid) {
      const int c_tile = tc.tn * tile_cols_;
      store_sum(tc.b, r, c_tile, ((c_tile % ss_seg) / tile_cols_) * 2 + half, ss);
    }
  }

  __device__ __forceinline__ void store_sum(int b, int r, int c, int slot, float ss) const {
    const int64_t vec = ssm.at(b, r, c / ss_seg);
    sumsq[(vec / ss_block) * ss_parts * ss_block + slot * ss_block + vec % ss_block] = ss;
  }

  // 32 values of a per-column vector (the same in every lane), `fill` past the nv valid ones.
  static __device__ __forceinline__ void load_cols(const float* src, int nv, float fill,
                                                   float (&o)[32]) {
    if (nv == 32 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 x = reinterpret_cast<const float4*>(src)[q];
        o[4 * q] = x.x;
        o[4 * q + 1] = x.y;
        o[4 * q + 2] = x.z;
        o[4 * q + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 32; ++e) o[e] = e < nv ? src[e] : fill;
    }
  }

  // Warp-collective: this warp's 32 rows x 32 fp32 columns as one TMA box.
  __device__ __forceinline__ void store32_tma(const TileCoord& tc, int row, int c0,
                                              const float (&v)[32], uint4* stage,
                                              const CUtensorMap* tmc) const {
    const int lane = threadIdx.x & 31;
    if (lane == 0) bulk_wait_read();  // the previous box has left the staging area
    __syncwarp();
    uint4* my = stage + lane * 8;  // 128 B per row; 16-B chunk q lands at q ^ (row & 7)
#pragma unroll
    for (int q = 0; q < 8; ++q)
      my[q ^ (lane & 7)] = make_uint4(__float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                                      __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3]));
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_3d(tmc, stage, c0, tc.tm * kBM + row, tc.b);
      bulk_commit();
    }
  }

  // Warp-collective on the vector path (every lane calls it; invalid rows store nothing).
  __device__ __forceinline__ void store32(const GemmParams& p, int b, int r, int c0,
                                          const float (&v)[32], bool rvalid,
                                          uint4* stage) const {
    const bool full = vec_ok && (c0 + 32 <= max(p.N, pad_n));  // uniform across the warp
    if (full) {
      const int64_t o = om.at(b, r, c0);
      uint4 a4[4], b4[4];
      if (kind == OUT_F32) {
        float* dst = static_cast<float*>(out) + o;
        pack_f32x16(v, a4);
        pack_f32x16(v + 16, b4);
        warp_store64(stage, a4, dst, rvalid);
        warp_store64(stage, b4, dst + 16, rvalid);
      } else if (kind == OUT_HILO || kind == OUT_HILO16) {
        __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(out) + o;
        if (kind == OUT_HILO)
          pack_hilo_x32(v, a4, b4);
        else
          pack_hilo16_x32(v, a4, b4);
        warp_store64(stage, a4, dst, rvalid);
        warp_store64(stage, b4, dst + lo_off, rvalid);
      } else {
        pack_bf16x32(v, a4);
        warp_store64(stage, a4, static_cast<__nv_bfloat16*>(out) + o, rvalid);
      }
      return;
    }
    if (!rvalid) return;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      const int c = c0 + e;
      if (c >= p.N) break;
      const int64_t o = om.at(b, r, c);
      if (kind == OUT_F32) {
        static_cast<float*>(out)[o] = v[e];
      } else if (kind == OUT_BF16) {
        static_cast<__nv_bfloat16*>(out)[o] = __float2bfloat16_rn(v[e]);
      } else if (kind == OUT_HILO16) {
        const __half hh = __float2half_rn(v[e]);
        const __half ll = __float2half_rn(v[e] - __half2float(hh));
        reinterpret_cast<__half*>(out)[o] = hh;
        reinterpret_cast<__half*>(out)[o + lo_off] = ll;
      } else {
        __nv_bfloat16 h, l;
        split_hilo(v[e], h, l);
        static_cast<__nv_bfloat16*>(out)[o] = h;
        static_cast<__nv_bfloat16*>(out)[o + lo_off] = l;
      }
    }
  }
};

using EpiAffine = EpiAffineT<false>;

// Cache positions given as segments: position of token idx = start[k] + (idx - begin[k]) * step[k].
struct PosSegs {
  int32_t n = 0;
  int64_t begin[9] = {0};
  double start[8] = {0};
  double step[8] = {0};
};

__device__ __forceinline__ double seg_position(const PosSegs& s, int64_t idx) {
  int k = 0;
#pragma unroll 1
  while (k + 1 < s.n && idx >= s.begin[k + 1]) ++k;
  return s.start[k] + (double)(idx - s.begin[k]) * s.step[k];
}

// Positions between two rows of the coarse compactor-RoPE table (see keyproj.cuh).
constexpr int kPosGrain = 32;

// sin and cos of |x| <= 1 from their Taylor series about 0, through x^11 and x^12 (the first
// omitted terms are below 2e-10), by Horner's rule in fp32: no range reduction needed.
__device__ __forceinline__ void sincos_taylor(float x, float* s, float* c) {
  const float x2 = x * x;
  float ps = 1.f / 39916800.f;                  // 1/11!
  ps = fmaf(ps, -x2, 1.f / 362880.f);           // 1/9!
  ps = fmaf(ps, -x2, 1.f / 5040.f);             // 1/7!
  ps = fmaf(ps, -x2, 1.f / 120.f);              // 1/5!
  ps = fmaf(ps, -x2, 1.f / 6.f);                // 1/3!
  ps = fmaf(ps, -x2, 1.f);
  float pc = 1.f / 479001600.f;                 // 1/12!
  pc = fmaf(pc, -x2, 1.f / 3628800.f);          // 1/10!
  pc = fmaf(pc, -x2, 1.f / 40320.f);            // 1/8!
  pc = fmaf(pc, -x2, 1.f / 720.f);              // 1/6!
  pc = fmaf(pc, -x2, 1.f / 24.f);               // 1/4!
  pc = fmaf(pc, -x2, 0.5f);                     // 1/2!
  *s = x * ps;
  *c = fmaf(pc, -x2, 1.f);
}

// Output heads: columns [0, d) = Z_out W_key, re-rotated by the base RoPE at the output
// position of latent j; columns [d, 2d) = Z_out W_val. Rows r = h * t + j. bf16 stores into
// the caller's C_k / C_v with element strides (st, sh). rot[j][m] = (cos, sin)(p_j * omega_m),
// a table formed once per call with the angle reduced modulo 2 pi in fp64.
// Folded key path (no compactor RoPE): |k~_n|^2 = x~_n G x~_n^T with G = W~ W~^T. The GEMM
// gives Y = x~ G (rows = tokens of one KV-head, columns = the Kp entries of one cross head);
// the epilogue dots each 32-column chunk of Y with the same columns of x~ (hi + lo, read back
// from global memory) and stores the partial, part-major: part[(b * Kp/32 + chunk) * Ntok + n].
struct EpiQuad {
  static constexpr int kWarps = 8;   // two per lane quarter: alternating 32-column chunks
  static constexpr int kStages = 0;
  float* part = nullptr;
  const __nv_bfloat16* xt = nullptr;  // x~ rows [hi | lo], pitch 2 Kp, of the group's first KV-head
  int64_t Ntok = 0;
  int32_t Kp = 0;
  int32_t tile_cols_ = 256;
  bool can_split() const { return true; }
  static constexpr bool kAnyTile = true;
  static constexpr bool kPairs = true;
  // Kp is 320, two tiles of 160, or 192. Measured on both kernels (us, 1-SM then pairs; 4 KV-heads of
  // 8 cross heads): Kp 320, 896 tokens 33.1, 32.6; 1,152 38.9, 37.8; 2,688 69.5, 63.5; 8,192 176.7,
  // 151.8 (158.3 in two tiles of 192). Kp 192, 1,024 tokens 21.0, 22.5; 2,048 31.4, 31.4; 2,432
  // 32.6, 35.9 (4 waves against 5); 4,864 52.8, 51.1; 8,192 81.3, 78.5. A line through each column
  // over its waves gives the clocks.
  using Widths = std::integer_sequence<int, 160, 192>;
  static constexpr int pair_wave(int bn) { return bn == 160 ? 745 : 800; }
  static constexpr int pair_start(int bn) { return bn == 160 ? -480 : 240; }

  template <class Src>
  __device__ void prefetch(const GemmParams&, const TileCoord&, int, const Src&, int) const {}

  template <class Src>
  __device__ void operator()(const GemmParams& p, const TileCoord& tc, int row, const Src& src,
                             int half, uint4*, const CUtensorMap*) const {
    const int r = tc.tm * kBM + row;
    const bool rvalid = r < p.M;
    const int parts = Kp / 32;
    const __nv_bfloat16* xr =
        xt + ((int64_t)(tc.b / p.bdiv) * Ntok + (rvalid ? r : 0)) * 2 * Kp;
    for (int cc = src.first(half); cc < tile_cols_; cc += src.step()) {
      float v[32];
      src.load(cc, v);
      const int c0 = tc.tn * tile_cols_ + cc;
      if (c0 >= p.N) continue;
      const uint4* hp = reinterpret_cast<const uint4*>(xr + c0);
      const uint4* lp = reinterpret_cast<const uint4*>(xr + Kp + c0);
      float acc = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 hq = hp[q], lq = lp[q];
        const uint32_t hw[4] = {hq.x, hq.y, hq.z, hq.w}, lw[4] = {lq.x, lq.y, lq.z, lq.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 h2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hw[k]));
          const float2 l2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&lw[k]));
          acc = fmaf(v[8 * q + 2 * k], h2.x + l2.x, acc);
          acc = fmaf(v[8 * q + 2 * k + 1], h2.y + l2.y, acc);
        }
      }
      if (rvalid) part[((int64_t)tc.b * parts + c0 / 32) * Ntok + r] = acc;
    }
  }
};

struct EpiHeads {
  static constexpr int kWarps = 8;
  static constexpr int kStages = 0;
  __nv_bfloat16* ck = nullptr;
  __nv_bfloat16* cv = nullptr;
  int64_t st = 0, sh = 0;  // element strides of [t, H, d]; d is contiguous, rows 16-B aligned
  int32_t t = 0, d = 0;
  const float2* rot = nullptr;  // [t][d/2]
  int32_t tile_cols_ = 256;
  bool can_split() const { return true; }
  static constexpr bool kPairs = false;
  static constexpr bool kAnyTile = false;  // a RoPE pair of C_k lies in one tile

  template <class Src>
  __device__ void prefetch(const GemmParams&, const TileCoord&, int, const Src&, int) const {}

  template <class Src>
  __device__ void operator()(const GemmParams& p, const TileCoord& tc, int row, const Src& src,
                             int half, uint4* stage, const CUtensorMap*) const {
    const int r = tc.tm * kBM + row;
    const bool rvalid = r < p.M;
    const int h = rvalid ? r / t : 0, j = rvalid ? r % t : 0;
    const int c_tile = tc.tn * tile_cols_;
    const float2* rrow = rot + (int64_t)j * (d / 2);
    const int64_t obase = (int64_t)j * st + (int64_t)h * sh;
    const int hd = d / 2;
    for (int cc = src.first(half); cc < tile_cols_; cc += src.step()) {
      const int c0 = c_tile + cc;
      if (c0 >= p.N) break;
      if (c0 < d) {
        // key columns: process pairs (m, m + d/2) when visiting the first half
        if (c0 >= hd) continue;
        float a[32], b[32];
        src.load(cc, a);
        src.load(cc + hd, b);
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const float2 cs = rrow[c0 + e];
          const float cw = cs.x, sw = cs.y;
          const float x = a[e], y = b[e];
          a[e] = x * cw - y * sw;
          b[e] = x * sw + y * cw;
        }
        uint4 o4[4];
        pack_bf16x32(a, o4);
        warp_store64(stage, o4, ck + obase + c0, rvalid);
        pack_bf16x32(b, o4);
        warp_store64(stage, o4, ck + obase + c0 + hd, rvalid);
      } else {
        float v[32];
        src.load(cc, v);
        uint4 o4[4];
        pack_bf16x32(v, o4);
        warp_store64(stage, o4, cv + obase + (c0 - d), rvalid);
      }
    }
  }
};

}  // namespace still
