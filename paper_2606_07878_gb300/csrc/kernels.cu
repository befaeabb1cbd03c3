// Memory-bound kernels of the compactor path: RoPE-fix strip, RoPE tables, query rotation,
// softmax, hi/lo conversion, RMSNorm, weight re-layout.
#include <algorithm>
#include <type_traits>

#include "kernels.cuh"
#include "launch.cuh"

namespace still {

namespace {

constexpr double kTwoPi = 6.283185307179586;
constexpr double kInvTwoPi = 0.15915494309189535;
constexpr float kLog2e = 1.4426950408889634f;

// angle reduced to [-pi, pi] in fp64, then sin/cos in fp32 (|error| ~1e-7)
__device__ __forceinline__ void sincos_reduced(double ang, float* s, float* c) {
  ang -= kTwoPi * rint(ang * kInvTwoPi);
  sincosf((float)ang, s, c);
}

constexpr int kStripTok = 32;

__device__ __forceinline__ int64_t kv_offset(const KVSource& src, int64_t n, int h, bool& second) {
  second = n >= src.n_split;
  return second ? (n - src.n_split) * src.sN2 + (int64_t)h * src.sH2
                : n * src.sN + (int64_t)h * src.sH;
}

// Eight consecutive bf16 of a K / V row (one 16-byte load when aligned).
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* p, bool vec) {
  if (vec) return *reinterpret_cast<const uint4*>(p);
  const uint16_t* q = reinterpret_cast<const uint16_t*>(p);
  uint32_t w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = q[2 * k] | (uint32_t)q[2 * k + 1] << 16;
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void widen8(const uint4& u, float (&v)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[k]));
    v[2 * k] = f.x;
    v[2 * k + 1] = f.y;
  }
}

// One CTA = 32 tokens x the KV-heads of its share (blockIdx.y of gridDim.y). A thread handles the
// same tokens and pairs of every head: it forms its base-RoPE angles once (fp64, reduced mod
// 2 pi) and keeps them in registers. Keys: inverse rotation of pairs (m, m + d/2) (Sec. 2.2,
// RoPE-fix); values pass through. Writes X (bf16 hi | key lo) and XT (fp16 hi for all 2d features,
// fp16 lo for the key half; the value half's lo is exactly zero and is never read). Rows are
// moved in 16-byte pieces; the transpose for XT goes through shared memory with an odd word pitch
// (conflict-free column reads). The next head's rows are loaded while this head's XT is written.
// Kp > 0 writes X in the layout of the folded key path instead: rows of 2 Kp elements,
// [x~ hi | x~ lo] with x~ = [unRoPE(K) | V | 1 | 0 ...] (Kp >= 2d + 1, a multiple of 64).
//
// Bound by memory (long caches) or by one CTA's chain of heads and the fp64 rate of its angles
// (short ones). Measured before (angles in shared memory,
// no load ahead, no shares) and now: 131,072 tokens of 8 heads of 256 channels 1291 -> 719 us
// (4.8 GB: 6.7 TB/s), 65,536 of 8 x 128 268 -> 189, 8,003 of 4 x 128 33 -> 25, three windows of
// 1,024 of 8 x 128 33 -> 14 each.
template <int HD>
__global__ void __launch_bounds__(256, HD == 256 ? 2 : 3)
    strip_kernel(KVSource src, int64_t N, int H, PosSegs segs, const double* __restrict__ omega,
                 int rope_fix, int vec, int x16, int Kp, __nv_bfloat16* __restrict__ X,
                 __half* __restrict__ XT, int64_t Np, float2* __restrict__ gd, double origin,
                 int G) {
  constexpr int half = HD / 2;
  constexpr int ph = 2 * HD + 2, pl = HD + 2;  // pitches (halves) of the transpose tiles
  constexpr int kg = half / 8, vg = HD / 8;    // 8-element groups per token: key pairs, values
  constexpr int kK = (kStripTok * kg + 255) / 256, kV = kStripTok * vg / 256;  // per thread
  __shared__ double tpos[kStripTok];
  extern __shared__ __align__(16) uint8_t sm[];
  __half* thi = reinterpret_cast<__half*>(sm);  // [kStripTok][ph]
  __half* tlo = thi + kStripTok * ph;           // [kStripTok][pl]
  const int64_t n0 = (int64_t)blockIdx.x * kStripTok;
  const int h0 = H * blockIdx.y / gridDim.y, h1 = H * (blockIdx.y + 1) / gridDim.y;
  uint4 ka[kK], kb[kK], va[kV];
  auto load = [&](int h) {
    bool second;
#pragma unroll
    for (int q = 0; q < kK; ++q) {
      const int it = threadIdx.x + 256 * q, m0 = 8 * (it % kg);
      const int64_t n = n0 + it / kg;
      ka[q] = kb[q] = make_uint4(0, 0, 0, 0);
      if (it < kStripTok * kg && n < N) {
        const int64_t off = kv_offset(src, n, h, second);
        const __nv_bfloat16* kr = (second ? src.K2 : src.K) + off;
        ka[q] = load8(kr + m0, vec);
        kb[q] = load8(kr + half + m0, vec);
      }
    }
#pragma unroll
    for (int q = 0; q < kV; ++q) {
      const int it = threadIdx.x + 256 * q;
      const int64_t n = n0 + it / vg;
      va[q] = make_uint4(0, 0, 0, 0);
      if (n < N) {
        const int64_t off = kv_offset(src, n, h, second);
        va[q] = load8((second ? src.V2 : src.V) + off + 8 * (it % vg), vec);
      }
    }
  };
  load(h0);
  if (threadIdx.x < kStripTok) {
    // token position (fp64) once per token; also the compactor-RoPE coarse index and residual
    const int64_t n = n0 + threadIdx.x;
    const double pos = n < N ? seg_position(segs, n) : origin;
    tpos[threadIdx.x] = pos;
    if (n < N && blockIdx.y == 0) {
      int g = (int)floor((pos - origin) / (double)kPosGrain);
      g = max(0, min(g, G - 1));
      gd[n] = make_float2((float)g, (float)(pos - (origin + (double)g * kPosGrain)));
    }
  }
  __syncthreads();
  float2 rot[kK][8];  // (cos, sin)
#pragma unroll
  for (int q = 0; q < kK; ++q) {
    const int it = threadIdx.x + 256 * q, tok = it / kg, m0 = 8 * (it % kg);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float sw = 0.f, cw = 1.f;
      if (rope_fix && it < kStripTok * kg && n0 + tok < N)
        sincos_reduced(tpos[tok] * omega[m0 + e], &sw, &cw);
      rot[q][e] = make_float2(cw, sw);
    }
  }
  const int d3 = Kp > 0 ? 2 * Kp : 3 * HD;  // X row pitch
  const int lo0 = Kp > 0 ? Kp : 2 * HD;     // column of the key lo part
  const int64_t ld = 2 * Np;
  for (int h = h0; h < h1; ++h) {
    // keys: group g holds pairs m = 8g .. 8g + 7
#pragma unroll
    for (int q = 0; q < kK; ++q) {
      const int it = threadIdx.x + 256 * q, tok = it / kg, m0 = 8 * (it % kg);
      if (kStripTok * kg % 256 != 0 && it >= kStripTok * kg) break;
      const int64_t n = n0 + tok;
      float a[8], b[8], xa[8], xb[8];
      widen8(ka[q], xa);
      widen8(kb[q], xb);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float2 cs = rot[q][e];
        a[e] = xa[e] * cs.x + xb[e] * cs.y;
        b[e] = -xa[e] * cs.y + xb[e] * cs.x;
      }
      if (n < N) {
        uint32_t ah[4], al[4], bh[4], bl[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (x16) {
            split_pack_f16(a[2 * k], a[2 * k + 1], ah[k], al[k]);
            split_pack_f16(b[2 * k], b[2 * k + 1], bh[k], bl[k]);
          } else {
            split_pack(a[2 * k], a[2 * k + 1], ah[k], al[k]);
            split_pack(b[2 * k], b[2 * k + 1], bh[k], bl[k]);
          }
        }
        __nv_bfloat16* xr = X + ((int64_t)h * N + n) * d3;
        *reinterpret_cast<uint4*>(xr + m0) = make_uint4(ah[0], ah[1], ah[2], ah[3]);
        *reinterpret_cast<uint4*>(xr + half + m0) = make_uint4(bh[0], bh[1], bh[2], bh[3]);
        *reinterpret_cast<uint4*>(xr + lo0 + m0) = make_uint4(al[0], al[1], al[2], al[3]);
        *reinterpret_cast<uint4*>(xr + lo0 + half + m0) = make_uint4(bl[0], bl[1], bl[2], bl[3]);
      }
      __half* hr = thi + tok * ph;
      __half* lr = tlo + tok * pl;
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const __half2 ha = __floats2half2_rn(a[e], a[e + 1]);
        const __half2 hb = __floats2half2_rn(b[e], b[e + 1]);
        const float2 fa = __half22float2(ha), fb = __half22float2(hb);
        *reinterpret_cast<__half2*>(hr + m0 + e) = ha;
        *reinterpret_cast<__half2*>(hr + half + m0 + e) = hb;
        *reinterpret_cast<__half2*>(lr + m0 + e) = __floats2half2_rn(a[e] - fa.x, a[e + 1] - fa.y);
        *reinterpret_cast<__half2*>(lr + half + m0 + e) =
            __floats2half2_rn(b[e] - fb.x, b[e + 1] - fb.y);
      }
    }
    // values: group g holds features 8g .. 8g + 7 (bf16 values are exact in fp16)
#pragma unroll
    for (int q = 0; q < kV; ++q) {
      const int it = threadIdx.x + 256 * q, tok = it / vg, f0 = 8 * (it % vg);
      const int64_t n = n0 + tok;
      float v[8];
      widen8(va[q], v);
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const __half2 x = __floats2half2_rn(v[2 * k], v[2 * k + 1]);
        w[k] = *reinterpret_cast<const uint32_t*>(&x);
        *reinterpret_cast<uint32_t*>(thi + tok * ph + HD + f0 + 2 * k) = w[k];
      }
      if (n < N)  // x16: values in fp16 (bf16 values in the fp16 range convert exactly)
        *reinterpret_cast<uint4*>(X + ((int64_t)h * N + n) * d3 + HD + f0) =
            x16 ? make_uint4(w[0], w[1], w[2], w[3]) : va[q];
    }
    if (Kp > 0) {  // folded layout: [.. | 1 | 0 ...] after the values, zeros after the key lo
      const int nc = (Kp - 2 * HD) / 8, nz = (Kp - HD) / 8;  // 16-byte groups per token
      for (int it = threadIdx.x; it < kStripTok * (nc + nz); it += blockDim.x) {
        const int tok = it / (nc + nz), q = it % (nc + nz);
        const int64_t n = n0 + tok;
        if (n >= N) continue;
        __nv_bfloat16* xr = X + ((int64_t)h * N + n) * d3;
        uint4 val = make_uint4(0, 0, 0, 0);
        if (q == 0) val.x = x16 ? 0x3C00u : 0x3F80u;  // 1.0 in the first element (fp16 / bf16)
        *reinterpret_cast<uint4*>(xr + (q < nc ? 2 * HD + 8 * q : Kp + HD + 8 * (q - nc))) = val;
      }
    }
    __syncthreads();
    if (h + 1 < h1) load(h + 1);
    // XT: feature rows of 32 tokens, 8 tokens (16 B) per store; hi rows [0, 2d), lo rows [0, d)
    constexpr int kTg = kStripTok / 8;
    constexpr int nhi = 2 * HD * kTg;
#pragma unroll 2
    for (int it = threadIdx.x; it < 3 * HD * kTg; it += 256) {
      const bool lo = it >= nhi;
      const int q = lo ? it - nhi : it;
      const int f = q / kTg, t0 = 8 * (q % kTg);
      const __half* col = lo ? tlo + f : thi + f;
      const int pitch = lo ? pl : ph;
      uint32_t w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const __half x0 = col[(t0 + 2 * k) * pitch], x1 = col[(t0 + 2 * k + 1) * pitch];
        const __half2 pr = __halves2half2(x0, x1);
        w[k] = *reinterpret_cast<const uint32_t*>(&pr);
      }
      __half* dst = XT + ((int64_t)h * 2 * HD + f) * ld + (lo ? Np : 0) + n0 + t0;
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    __syncthreads();
  }
}

// The call's angle tables (see RopeTables): coarse rows, then the fine table, then the output heads'
// rotations, an entry per thread. Angles formed and reduced in fp64, whose rate bounds it. One
// launch for all three; in CTAs of the strip launch they held up its token tiles (8,003 tokens:
// the call 953 -> 961 us).
__global__ void rope_tables_kernel(const RopeTables tb) {
  griddep_wait();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int quarter = tb.D / 4;
  const int64_t ncoarse = (int64_t)tb.G * quarter, nkey = ncoarse + (int64_t)kPosGrain * quarter;
  if (idx < nkey) {
    const int g = (int)(idx / quarter);
    const int64_t f = idx - ncoarse;  // index into the fine table when >= 0
    const int q = g < tb.G ? (int)(idx % quarter) : (int)(f / kPosGrain);
    float s[2], c[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const double w = tb.omega_c[2 * q + e];
      const double ang =
          g < tb.G ? (tb.origin + (double)g * kPosGrain) * w : (double)(f % kPosGrain) * w;
      sincos_reduced(ang, &s[e], &c[e]);
      if (g == 0) tb.omega[2 * q + e] = (float)w;
    }
    tb.coarse[idx] = make_float4(c[0], c[1], s[0], s[1]);
  } else if (idx - nkey < (int64_t)tb.t * tb.hd) {
    const int64_t r = idx - nkey;
    const int j = (int)(r / tb.hd), m = (int)(r % tb.hd);
    float s = 0.f, c = 1.f;
    if (tb.use_rope) sincos_reduced((tb.qstart + (double)j * tb.qstep) * tb.omega_b[m], &s, &c);
    tb.hrot[r] = make_float2(c, s);
  }
}

// Thread = (latent j, 4 consecutive pairs m) x a share of the batches (blockIdx.y); the angles are
// formed once and reused for every batch of the share. Columns are in pair-chunk order: pair m
// sits at f1 = (m / 128) * 256 + m % 128 and its partner at f1 + 128, so four consecutive pairs
// are four consecutive columns. Bound by memory once enough rows are in flight. Measured with one
// share and now: 64 batches of 164 x 1024 51 -> 26 us, 32 of 251 x 1024 32 -> 25; from t = 655 up
// unchanged at 87% of the memory rate (one share).
__global__ void q_rope_kernel(const float* __restrict__ qhat, const float* __restrict__ scale,
                              int t_max, int b0, int nb, int t, int D, double qstart,
                              double qstep, const double* omega_c, int use_rope,
                              __nv_bfloat16* __restrict__ qhl, int fp16, float qscale) {
  griddep_wait();
  const int half = D / 2, q4 = half / 4;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)t * q4) return;
  const int j = (int)(idx / q4), m0 = 4 * (int)(idx % q4);
  float s[4], c[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    s[e] = 0.f;
    c[e] = 1.f;
    if (use_rope) sincos_reduced((qstart + (double)j * qstep) * omega_c[m0 + e], &s[e], &c[e]);
  }
  const int f1 = (m0 / 128) * 256 + (m0 % 128), f2 = f1 + 128;
  const int bb1 = (int)((int64_t)nb * (blockIdx.y + 1) / gridDim.y);
#pragma unroll 2
  for (int bb = (int)((int64_t)nb * blockIdx.y / gridDim.y); bb < bb1; ++bb) {
    const float* q = qhat + ((int64_t)(b0 + bb) * t_max + j) * D;
    const float4 x4 = *reinterpret_cast<const float4*>(q + f1);
    const float4 y4 = *reinterpret_cast<const float4*>(q + f2);
    float x[4] = {x4.x, x4.y, x4.z, x4.w}, y[4] = {y4.x, y4.y, y4.z, y4.w};
    if (scale != nullptr) {
      const float f = scale[(int64_t)bb * t + j];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        x[e] *= f;
        y[e] *= f;
      }
    }
    float a[4], b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      a[e] = x[e] * c[e] - y[e] * s[e];
      b[e] = x[e] * s[e] + y[e] * c[e];
    }
    uint32_t ah[2], al[2], bh[2], bl[2];
    if (fp16) {
      split_pack_f16(a[0] * qscale, a[1] * qscale, ah[0], al[0]);
      split_pack_f16(a[2] * qscale, a[3] * qscale, ah[1], al[1]);
      split_pack_f16(b[0] * qscale, b[1] * qscale, bh[0], bl[0]);
      split_pack_f16(b[2] * qscale, b[3] * qscale, bh[1], bl[1]);
    } else {
      split_pack(a[0], a[1], ah[0], al[0]);
      split_pack(a[2], a[3], ah[1], al[1]);
      split_pack(b[0], b[1], bh[0], bl[0]);
      split_pack(b[2], b[3], bh[1], bl[1]);
    }
    __nv_bfloat16* o = qhl + ((int64_t)bb * t + j) * 2 * D;
    *reinterpret_cast<uint2*>(o + f1) = make_uint2(ah[0], ah[1]);
    *reinterpret_cast<uint2*>(o + D + f1) = make_uint2(al[0], al[1]);
    *reinterpret_cast<uint2*>(o + f2) = make_uint2(bh[0], bh[1]);
    *reinterpret_cast<uint2*>(o + D + f2) = make_uint2(bl[0], bl[1]);
  }
}

__device__ __forceinline__ void ml_combine(float& m, float& l, float m2, float l2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2;
    l = l2;
    return;
  }
  const float M = fmaxf(m, m2);
  l = l * exp2f((m - M) * kLog2e) + l2 * exp2f((m2 - M) * kLog2e);
  m = M;
}

template <typename OutT>
__global__ void __launch_bounds__(256) softmax_kernel(const float* __restrict__ S, int64_t ncols,
                                                      int64_t ldS, OutT* __restrict__ P,
                                                      int64_t ldP) {
  griddep_wait();
  __shared__ float red_m[8], red_l[8];
  const int64_t row = blockIdx.x;
  const float* s = S + row * ldS;
  float m = -INFINITY, l = 0.f;
  for (int64_t c = threadIdx.x; c < ncols; c += blockDim.x) {
    const float x = s[c];
    if (x > m) {
      l = (m == -INFINITY ? 0.f : l * exp2f((m - x) * kLog2e)) + 1.f;
      m = x;
    } else {
      l += exp2f((x - m) * kLog2e);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
    ml_combine(m, l, m2, l2);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red_m[warp] = m;
    red_l[warp] = l;
  }
  __syncthreads();
  if (warp == 0) {
    m = lane < 8 ? red_m[lane] : -INFINITY;
    l = lane < 8 ? red_l[lane] : 0.f;
    for (int o = 4; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
      const float l2 = __shfl_xor_sync(0xffffffffu, l, o);
      ml_combine(m, l, m2, l2);
    }
    if (lane == 0) {
      red_m[0] = m;
      red_l[0] = l;
    }
  }
  __syncthreads();
  const float M = red_m[0], inv = 1.f / red_l[0];
  OutT* p = P + row * ldP;
  for (int64_t c = threadIdx.x; c < ldP; c += blockDim.x) {
    const float v = c < ncols ? exp2f((s[c] - M) * kLog2e) * inv : 0.f;
    if constexpr (sizeof(OutT) == 2 && std::is_same<OutT, __half>::value)
      p[c] = __float2half_rn(v);
    else
      p[c] = __float2bfloat16_rn(v);
  }
}

// Row softmax with the row held in registers: 256 threads, PER columns each (float4 groups).
// HILO: the row is written as hi at [0, ldP) and lo = OutT(p - hi) at [ldP, 2 ldP) of a row of
// pitch 2 ldP (bf16 or fp16 parts).
template <typename OutT, int PER, bool HILO = false>
__global__ void __launch_bounds__(256) softmax_reg_kernel(const float* __restrict__ S,
                                                          int64_t ncols, int64_t ldS,
                                                          OutT* __restrict__ P, int64_t ldP) {
  griddep_wait();
  __shared__ float red[8];
  const int64_t row = blockIdx.x;
  const float* s = S + row * ldS;
  constexpr int G = PER / 4;
  float v[PER];
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const int64_t c = (int64_t)(i * 256 + threadIdx.x) * 4;
    float4 x = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (c + 3 < ncols) {
      x = *reinterpret_cast<const float4*>(s + c);
    } else if (c < ncols) {
      x.x = s[c];
      if (c + 1 < ncols) x.y = s[c + 1];
      if (c + 2 < ncols) x.z = s[c + 2];
    }
    v[4 * i] = x.x;
    v[4 * i + 1] = x.y;
    v[4 * i + 2] = x.z;
    v[4 * i + 3] = x.w;
    m = fmaxf(m, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) red[warp] = m;
  __syncthreads();
  m = red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = fmaxf(m, red[w]);
  __syncthreads();
  float l = 0.f;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    v[k] = exp2f((v[k] - m) * kLog2e);  // exp(-inf) = 0 for padding
    l += v[k];
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (lane == 0) red[warp] = l;
  __syncthreads();
  l = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) l += red[w];
  const float inv = 1.f / l;
  OutT* prow = P + row * (HILO ? 2 * ldP : ldP);
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const int64_t c = (int64_t)(i * 256 + threadIdx.x) * 4;
    if (c < ldP) {
      OutT o4[4], l4[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float y = v[4 * i + k] * inv;
        if constexpr (std::is_same<OutT, __half>::value) {
          o4[k] = __float2half_rn(y);
          if constexpr (HILO) l4[k] = __float2half_rn(y - __half2float(o4[k]));
        } else {
          o4[k] = __float2bfloat16_rn(y);
          if constexpr (HILO) l4[k] = __float2bfloat16_rn(y - __bfloat162float(o4[k]));
        }
      }
      *reinterpret_cast<uint2*>(prow + c) = *reinterpret_cast<const uint2*>(o4);
      if constexpr (HILO) *reinterpret_cast<uint2*>(prow + ldP + c) = *reinterpret_cast<const uint2*>(l4);
    }
  }
}

// Failure-detection self-test: waits on an mbarrier that nothing arrives on, with a short
// bound. The wait expires, the kernel records DEV_WAIT_TIMEOUT in the error record and returns.
__global__ void wait_timeout_selftest_kernel(int* err, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t a = smem_u32(&bar);
    const uint64_t t0 = globaltimer_ns();
    bool done = false;
    while (!done && globaltimer_ns() - t0 < limit_ns) done = mbar_try_wait(a, 0) != 0;
    if (!done) dev_set_error(err, DEV_WAIT_TIMEOUT, 900);
  }
}

__global__ void omega_kernel(double* out, int half, int width, double base) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < half) out[m] = pow(base, -2.0 * m / width);
}

// Key-split merge of the fused cross-attention. Split s holds, per row, the unnormalised
// O_s = sum_k 2^(v_k - m_s) X_k and l_s = sum_k 2^(v_k - m_s) (v, m in log2 units). With
// M = max_s m_s:  O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s, summed in split order.
// One warp per row; lane k holds the weight of split k (at most 32), and each lane owns G groups
// of 4 columns (16-byte loads, those of several splits in flight). Measured with the statistics
// read and the weights formed again per column group, and now: 131,072 tokens, t = 655 198 -> 129
// us, 65,536 tokens, t = 1311 37 -> 27, 8,003 tokens, t = 251 21 -> 15.
template <int G>
__global__ void __launch_bounds__(256) ca_merge_kernel(const float* __restrict__ O,
                                                       const float2* __restrict__ stats,
                                                       int nsplit, int b0, int nb, int n, int t,
                                                       int f16, __nv_bfloat16* __restrict__ PX) {
  griddep_wait();
  constexpr int d2 = 128 * G;
  const int64_t rows = (int64_t)nb * t;
  const int64_t rj = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (rj >= rows) return;
  const float2 st = lane < nsplit ? stats[lane * rows + rj] : make_float2(-INFINITY, 0.f);
  float M = st.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  const float wl = exp2f(st.x - M);
  float4 acc[G];
#pragma unroll
  for (int g = 0; g < G; ++g) acc[g] = make_float4(0.f, 0.f, 0.f, 0.f);
  float L = 0.f;
#pragma unroll 4
  for (int k = 0; k < nsplit; ++k) {
    const float4* orow = reinterpret_cast<const float4*>(O + (k * rows + rj) * d2) + lane;
    const float w = __shfl_sync(0xffffffffu, wl, k);
    L += w * __shfl_sync(0xffffffffu, st.y, k);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float4 o = orow[32 * g];
      acc[g].x += w * o.x;
      acc[g].y += w * o.y;
      acc[g].z += w * o.z;
      acc[g].w += w * o.w;
    }
  }
  const float invL = 1.f / L;
  const int j = (int)(rj % t), bb = (int)(rj / t);
  const int b = b0 + bb, h = b / n, i = b % n;
  const int64_t ld = 2 * (int64_t)n * d2;
  __nv_bfloat16* row = PX + ((int64_t)h * t + j) * ld + (int64_t)i * d2;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int c = 4 * lane + 128 * g;
    uint32_t h01, l01, h23, l23;
    if (f16) {  // fp16 hi | lo
      split_pack_f16(acc[g].x * invL, acc[g].y * invL, h01, l01);
      split_pack_f16(acc[g].z * invL, acc[g].w * invL, h23, l23);
    } else {
      split_pack(acc[g].x * invL, acc[g].y * invL, h01, l01);
      split_pack(acc[g].z * invL, acc[g].w * invL, h23, l23);
    }
    *reinterpret_cast<uint2*>(row + c) = make_uint2(h01, h23);
    *reinterpret_cast<uint2*>(row + (int64_t)n * d2 + c) = make_uint2(l01, l23);
  }
}

__global__ void __launch_bounds__(256) rmsnorm_kernel(const void* __restrict__ in, int in_bf16,
                                                      int64_t rows, int D, int64_t ldi, float eps,
                                                      __nv_bfloat16* __restrict__ out,
                                                      int64_t ldo, int hilo) {
  griddep_wait();
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  auto ld = [&](int c) -> float {
    return in_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(in)[row * ldi + c])
                   : static_cast<const float*>(in)[row * ldi + c];
  };
  float ss = 0.f;
  for (int c = lane; c < D; c += 32) {
    const float x = ld(c);
    ss += x * x;
  }
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float scale = 1.f / sqrtf(ss / (float)D + eps);
  __nv_bfloat16* o = out + row * ldo;
  for (int c = lane; c < D; c += 32) {
    const float y = ld(c) * scale;
    if (hilo == 2) {  // fp16 hi | lo
      const __half hi = __float2half_rn(y);
      const __half lo = __float2half_rn(y - __half2float(hi));
      reinterpret_cast<__half*>(o)[c] = hi;
      reinterpret_cast<__half*>(o)[D + c] = lo;
    } else if (hilo) {
      __nv_bfloat16 hi, lo;
      split_hilo(y, hi, lo);
      o[c] = hi;
      o[D + c] = lo;
    } else {
      o[c] = __float2bfloat16_rn(y);
    }
  }
}

__global__ void bf16_to_f16_kernel(uint16_t* p, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const __nv_bfloat16 b = *reinterpret_cast<const __nv_bfloat16*>(&p[i]);
  const __half h = __float2half_rn(__bfloat162float(b));
  p[i] = *reinterpret_cast<const uint16_t*>(&h);
}

__global__ void scale_rows_kernel(float* x, const float* inv, int64_t rows, int D) {
  griddep_wait();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * D) return;
  x[idx] *= inv[idx / D];
}

__global__ void inv_norms_kernel(const float* __restrict__ parts, int64_t nvec, int nparts,
                                 int64_t block, float eps, float alpha, float* __restrict__ out) {
  griddep_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nvec) return;
  const float* p = parts + (i / block) * nparts * block + i % block;
  float s = 0.f;
  for (int k = 0; k < nparts; ++k) s += p[k * block];  // fixed order
  out[i] = alpha / fmaxf(sqrtf(fmaxf(s, 0.f)), eps);  // a quadratic form may round below 0
}

__global__ void transpose_kernel(const __nv_bfloat16* __restrict__ in, int64_t R, int64_t C,
                                 __nv_bfloat16* __restrict__ out, int perm_D,
                                 int key_rows) {
  __shared__ __nv_bfloat16 tile[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32, r0 = (int64_t)blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t r = r0 + k, c = c0 + threadIdx.x;
    if (r < R && c < C) {
      const int pos = key_rows ? key_row_source((int)c) : (int)c;
      const int64_t src = perm_D > 0 ? pair_chunk_src(pos, perm_D) : c;
      tile[k][threadIdx.x] = in[r * C + src];
    }
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t c = c0 + k, r = r0 + threadIdx.x;
    if (r < R && c < C) out[c * R + r] = tile[threadIdx.x][k];
  }
}

__global__ void bias_kernel(const __nv_bfloat16* in, const __nv_bfloat16* in2, int64_t C,
                            float* out, int perm_D) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const int64_t src = perm_D > 0 ? pair_chunk_src((int)c, perm_D) : c;
  out[c] = __bfloat162float(in[src]);
  if (in2 != nullptr) out[C + c] = __bfloat162float(in2[src]);
}

// ---------------------------------------------------------------- folded key projection

// Wt[i][c][j] = W_K,i[c][j] (c < 2d), b_K,i[j] (c = 2d), 0 (2d < c < Kp): the rows of
// W~_i = [W_K,i ; b_K,i], from the pair-chunk-ordered transposed copy WkT[i D + j][c] and
// bias bk[i D + j] (fp32 copies of bf16 values, so the conversion back is exact).
__global__ void fold_weights_kernel(const __nv_bfloat16* __restrict__ WkT,
                                    const float* __restrict__ bk, int n, int D, int d2, int Kp,
                                    __nv_bfloat16* __restrict__ Wt) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n * Kp * D) return;
  const int j = (int)(idx % D);
  const int c = (int)((idx / D) % Kp);
  const int i = (int)(idx / ((int64_t)D * Kp));
  const int64_t col = (int64_t)i * D + j;
  __nv_bfloat16 v = __float2bfloat16_rn(0.f);
  if (c < d2)
    v = WkT[col * d2 + c];
  else if (c == d2)
    v = __float2bfloat16_rn(bk[col]);
  Wt[idx] = v;
}

// out[r] = [bf16 hi(x) | bf16 lo(x)] of fp32 rows x of width C.
__global__ void f32_hilo_kernel(const float* __restrict__ x, int64_t rows, int C,
                                __nv_bfloat16* __restrict__ out) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= rows * C) return;
  const int64_t r = idx / C;
  const int c = (int)(idx % C);
  __nv_bfloat16 hi, lo;
  split_hilo(x[idx], hi, lo);
  out[r * 2 * C + c] = hi;
  out[r * 2 * C + C + c] = lo;
}

// ----------------------------------------------------------------------- beta channel

// beta[j][h] of latent row (h, j): Z_out (hi + lo) . w, then saturation and the mass-matching
// offset (App. A, output projections and optional beta shaping). One warp per row.
__global__ void beta_kernel(const __nv_bfloat16* __restrict__ Z, int64_t rows, int t, int H,
                            int D, const float* __restrict__ w, float beta_max, float offset,
                            float* __restrict__ beta) {
  griddep_wait();
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const __nv_bfloat16* z = Z + row * 2 * D;
  float acc = 0.f;
  for (int c = lane; c < D; c += 32)
    acc += (__bfloat162float(z[c]) + __bfloat162float(z[D + c])) * w[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    if (beta_max > 0.f) acc = beta_max * tanhf(acc / beta_max);
    const int h = (int)(row / t), j = (int)(row % t);
    beta[(int64_t)j * H + h] = acc + offset;
  }
}

// ----------------------------------------------------------------- biased decode attention
//
// Attention of query rows over the entries [C (t compact slots, logit bias beta) ; F (S
// uncompacted entries, bias 0)] (App. B, "Bias semantics in attention"). Each entry's K and V
// row is read once and takes part in G = nq Hq / H query rows: HBM bounds the kernel as long as
// the work per entry stays small, so the inner loop is built for few instructions per entry and
// several independent warps per scheduler.
//
// Grid (slot x row block, KV-head, layer). The entries of a KV-head are cut into batches (of one
// part each: the last batch of either part may be short), the batches into slots; the warps of
// a CTA take the batches of its slot in turn and never wait for one another until the slot
// ends. Per batch of a warp:
//   S^T = K q^T  mma.m16n8k16 (16 entries x 8 query rows; bf16 products, fp32 sums). The order
//                of the d dimensions inside the contraction is free as long as K and q agree, so
//                the 16 contiguous bytes of a K row that a lane loads are the A fragments of two
//                steps: K goes from global memory to the tensor core without shared memory.
//   P            online softmax per query row in fp32, exchanged through a few hundred bytes of
//                the warp's shared memory
//   O += P V     fp32 FMAs in packed pairs (fma.rn.f32x2): a lane owns 8 dimensions of the V
//                rows of its lane group's entries, so P stays fp32 and a V row is unpacked once
//                for all query rows
// The next batch's K loads are issued when S is formed and its V loads when O is: each lane's
// registers hold them in flight. The row states (m, l, O) of the warps are combined once per
// slot; decode_merge_kernel combines the slots in order (with one slot the CTA writes the output
// itself). Query rows beyond 8 go to further row blocks, which read the entries again through
// L2.
//
// Measured on 36 layers, 1 token, 32 query heads over 8 KV-heads, d = 128, t = 1311 + 4096
// (799 MB): 155 us with the merge, 5.2 TB/s; 148 us and 69% of the DRAM's cycles for this kernel
// alone. 444 us with the kernel it replaced, whose warps formed every logit by FMAs and warp sums
// and met at two block barriers per 128 entries. A shared-memory ring filled by cp.async (205 us;
// 211 us with a persistent grid) costs more instructions per entry than the register form.
template <int D>
struct DecShape {
  static constexpr int kWarps = 4;
  static constexpr int kBatch = D == 64 ? 32 : D == 128 ? 16 : 8;  // entries: 32 registers of K
  static constexpr int kRows = kBatch / 8;       // K rows per lane group (entries lg + 8 i)
  static constexpr int kChunks = D / 32;         // 16-byte K pieces per lane and row
  static constexpr int kGroups = 32 / (D / 8);   // lane groups that split a batch's V rows
  static constexpr int kVRows = kBatch / kGroups;
};

// c (16 entries x 8 rows) += a (16 x 16 bf16) b (16 x 8 bf16)
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Read-once data: past L1, first to leave L2.
__device__ __forceinline__ uint4 ld_stream(const __nv_bfloat16* p) {
  return __ldcs(reinterpret_cast<const uint4*>(p));
}

// R: query rows per row block (4 or 8).
template <int D, int R>
__global__ void __launch_bounds__(32 * DecShape<D>::kWarps, R == 4 ? 3 : 2)
    decode_chunk_kernel(const __grid_constant__ DecodeStack st, int nslots, int nrb,
                        float* __restrict__ part_o, float2* __restrict__ part_ml) {
  using S = DecShape<D>;
  constexpr int kW = S::kWarps, kBatch = S::kBatch, kRows = S::kRows;
  __shared__ __align__(16) float wts[kW][(kBatch + 1) * R];  // weights, then rescale factors
  __shared__ __align__(16) float red[kW][4][D + 2];          // O, m, l of four rows per warp
  const DecodeArgs& a = st.layer[blockIdx.z];
  const int h = blockIdx.y, slot = blockIdx.x / nrb, rb = blockIdx.x % nrb;
  const int g = a.Hq / a.H;   // query heads per KV-head
  const int G = a.nq * g;     // query rows of this KV-head
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lg = lane >> 2, lj = lane & 3;             // MMA fragment coordinates
  const int kg = lane / (D / 8), dc = lane % (D / 8);  // V: lane group, 8-dimension piece
  float* pw = wts[warp];
  // batches: nbc of the compact part, then those of the other part; this slot's [b0, b1)
  const int nbc = (int)((a.t + kBatch - 1) / kBatch);
  const int nbt = nbc + (int)((a.S + kBatch - 1) / kBatch);
  const int b0 = (int)((int64_t)nbt * slot / nslots) + warp;
  const int b1 = (int)((int64_t)nbt * (slot + 1) / nslots);
  const int64_t pitch = a.cst;  // entry pitch (the same in both parts)
  const int64_t hoff = (int64_t)h * D;

  // Entry range of batch b: first entry, entries left in its part, the part.
  auto locate = [&](int b, bool& comp, int64_t& e0, int& left) {
    comp = b < nbc;
    e0 = (int64_t)(comp ? b : b - nbc) * kBatch;
    left = (int)min((int64_t)kBatch, (comp ? a.t : a.S) - e0);
  };
  uint4 kx[kRows][S::kChunks], vx[S::kVRows];
  float bias[kRows];
  // Entries past the end of the part load its last entry (its weight is 0, its V zeroed).
  auto load_k = [&](int b) {
    bool comp;
    int64_t e0;
    int left;
    locate(b, comp, e0, left);
    const __nv_bfloat16* base = (comp ? a.Ck : a.Kf) + e0 * pitch + hoff + 8 * lj;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = min(lg + 8 * i, left - 1);
      const __nv_bfloat16* p = base + r * pitch;
#pragma unroll
      for (int c = 0; c < S::kChunks; ++c) kx[i][c] = ld_stream(p + 32 * c);
      bias[i] = comp && a.beta != nullptr ? a.beta[(e0 + r) * a.H + h] : 0.f;
    }
  };
  auto load_v = [&](int b) {
    bool comp;
    int64_t e0;
    int left;
    locate(b, comp, e0, left);
    const __nv_bfloat16* base = (comp ? a.Cv : a.Vf) + e0 * pitch + hoff + 8 * dc;
#pragma unroll
    for (int v = 0; v < S::kVRows; ++v)
      vx[v] = ld_stream(base + min(v * S::kGroups + kg, left - 1) * pitch);
  };

  if (b0 < b1) {
    load_k(b0);
    load_v(b0);
  }
  // q as B fragments: row lg of the block, the same order of dimensions as K
  uint4 qf[S::kChunks];
  {
    const int r = rb * R + lg;
    const bool ok = lg < R && r < G;
    const int n = ok ? r / g : 0, qh = ok ? h * g + r % g : 0;
    const __nv_bfloat16* qp = a.q + ((int64_t)n * a.Hq + qh) * D + 8 * lj;
#pragma unroll
    for (int c = 0; c < S::kChunks; ++c)
      qf[c] = ok ? *reinterpret_cast<const uint4*>(qp + 32 * c) : make_uint4(0u, 0u, 0u, 0u);
  }
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;  // rows 2 lj and 2 lj + 1
  uint64_t acc[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = 0ull;

#pragma unroll 1
  for (int b = b0; b < b1; b += kW) {
    float c[kRows == 4 ? 2 : 1][4], c2[kRows == 4 ? 2 : 1][4];
#pragma unroll
    for (int i = 0; i < (kRows == 4 ? 2 : 1); ++i) {
#pragma unroll
      for (int e = 0; e < 4; ++e) c[i][e] = c2[i][e] = 0.f;
#pragma unroll
      for (int s = 0; s < S::kChunks; ++s) {
        const uint4 ka = kx[kRows == 1 ? 0 : 2 * i][s];
        const uint4 kb = kRows == 1 ? make_uint4(0u, 0u, 0u, 0u) : kx[kRows == 1 ? 0 : 2 * i + 1][s];
        mma_16816(c[i], ka.x, kb.x, ka.y, kb.y, qf[s].x, qf[s].y);
        mma_16816(c2[i], ka.z, kb.z, ka.w, kb.w, qf[s].z, qf[s].w);
      }
    }
    bool comp;
    int64_t e0;
    int left;
    locate(b, comp, e0, left);
    float s0[kRows], s1[kRows], x0 = -INFINITY, x1 = -INFINITY;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const float t0 = c[i / 2][2 * (i & 1)] + c2[i / 2][2 * (i & 1)];
      const float t1 = c[i / 2][2 * (i & 1) + 1] + c2[i / 2][2 * (i & 1) + 1];
      const bool ok = lg + 8 * i < left;
      s0[i] = ok ? t0 * a.scale + bias[i] : -INFINITY;
      s1[i] = ok ? t1 * a.scale + bias[i] : -INFINITY;
      x0 = fmaxf(x0, s0[i]);
      x1 = fmaxf(x1, s1[i]);
    }
    if (b + kW < b1) load_k(b + kW);
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) {
      x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
      x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
    }
    const float n0 = fmaxf(m0, x0), n1 = fmaxf(m1, x1);
    const bool moved = __any_sync(0xffffffffu, n0 != m0 || n1 != m1);
    if (moved) {
      const float f0 = n0 == m0 ? 1.f : __expf(m0 - n0), f1 = n1 == m1 ? 1.f : __expf(m1 - n1);
      l0 *= f0;
      l1 *= f1;
      m0 = n0;
      m1 = n1;
      if (lg == 0 && 2 * lj < R)
        *reinterpret_cast<float2*>(pw + kBatch * R + 2 * lj) = make_float2(f0, f1);
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const bool ok = lg + 8 * i < left;
      const float p0 = ok ? __expf(s0[i] - m0) : 0.f, p1 = ok ? __expf(s1[i] - m1) : 0.f;
      l0 += p0;
      l1 += p1;
      if (2 * lj < R) *reinterpret_cast<float2*>(pw + (lg + 8 * i) * R + 2 * lj) = make_float2(p0, p1);
    }
    __syncwarp();
    if (moved) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float f = pw[kBatch * R + r];
        const uint64_t f2 = pack2(f, f);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[r][i] = mul2(acc[r][i], f2);
      }
    }
    if (left < kBatch) {  // 0 * inf of a repeated entry would be NaN
#pragma unroll
      for (int v = 0; v < S::kVRows; ++v)
        if (v * S::kGroups + kg >= left) vx[v] = make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int v = 0; v < S::kVRows; ++v) {
      const uint64_t x[4] = {bf16_pair(vx[v].x), bf16_pair(vx[v].y), bf16_pair(vx[v].z),
                             bf16_pair(vx[v].w)};
      const float4* pr = reinterpret_cast<const float4*>(pw + (v * S::kGroups + kg) * R);
#pragma unroll
      for (int rq = 0; rq < R / 4; ++rq) {
        const float4 p = pr[rq];
        const float ps[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t p2 = pack2(ps[k], ps[k]);
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[4 * rq + k][i] = fma2(p2, x[i], acc[4 * rq + k][i]);
        }
      }
    }
    if (b + kW < b1) load_v(b + kW);
    __syncwarp();  // the weights are overwritten next
  }
  // ---- the slot's end: the warps' row states, four rows at a time
#pragma unroll
  for (int o = 4; o <= 16; o <<= 1) {
    l0 += __shfl_xor_sync(0xffffffffu, l0, o);
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  }
  const int64_t lrows = (int64_t)blockIdx.z * a.nq * a.Hq * nslots;  // this layer's partials
#pragma unroll
  for (int r0 = 0; r0 < R; r0 += 4) {
    if (r0 > 0 && rb * R + r0 >= G) break;  // uniform in the CTA
    if (r0 > 0) __syncthreads();
    if (lg == 0 && 2 * lj >= r0 && 2 * lj < r0 + 4) {
      float* mr = red[warp][2 * lj - r0];
      mr[D] = m0;
      mr[D + 1] = l0;
      mr[D + 2 + D] = m1;
      mr[D + 2 + D + 1] = l1;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float x, y;
        unpack2(acc[r0 + r][i], x, y);
#pragma unroll
        for (int o = D / 8; o < 32; o <<= 1) {  // lane groups hold different entries
          x += __shfl_xor_sync(0xffffffffu, x, o);
          y += __shfl_xor_sync(0xffffffffu, y, o);
        }
        if (kg == 0) *reinterpret_cast<float2*>(&red[warp][r][8 * dc + 2 * i]) = make_float2(x, y);
      }
    }
    __syncthreads();
    const int nr = min(4, G - rb * R - r0);
    for (int it = threadIdx.x; it < nr * D; it += 32 * kW) {
      const int r = it / D, col = it % D;
      float M = -INFINITY;
#pragma unroll
      for (int v = 0; v < kW; ++v) M = fmaxf(M, red[v][r][D]);
      float L = 0.f, O = 0.f;
#pragma unroll
      for (int v = 0; v < kW; ++v) {  // fixed order
        const float* sw = red[v][r];
        const float wt = sw[D] == -INFINITY ? 0.f : __expf(sw[D] - M);
        L += wt * sw[D + 1];
        O += wt * sw[col];
      }
      const int rr = rb * R + r0 + r;
      const int64_t orow = (int64_t)(rr / g) * a.Hq + h * g + rr % g;
      if (nslots == 1) {
        a.out[orow * D + col] = __float2bfloat16_rn(O / L);
      } else {
        part_o[(lrows + orow * nslots + slot) * D + col] = O;
        if (col == 0) part_ml[lrows + orow * nslots + slot] = make_float2(M, L);
      }
    }
  }
}

// Output row (query n, query head qh): sum_s e^(m_s - M) O_s / sum_s e^(m_s - M) l_s over the
// chunk partials, in chunk order. One CTA of d threads per row, one column per thread.
__global__ void decode_merge_kernel(const __grid_constant__ DecodeStack st,
                                    const float* __restrict__ part_o,
                                    const float2* __restrict__ part_ml, int64_t rows, int nch,
                                    int d) {
  griddep_wait();
  extern __shared__ float2 mls[];  // the row's (m, l) per chunk, then (weight, -)
  const int64_t row = blockIdx.x;
  const int c = threadIdx.x;
  __nv_bfloat16* __restrict__ out = st.layer[blockIdx.y].out;
  part_o += (int64_t)blockIdx.y * rows * nch * d;  // layer blockIdx.y's partials
  part_ml += (int64_t)blockIdx.y * rows * nch;
  for (int s = c; s < nch; s += blockDim.x) mls[s] = part_ml[row * nch + s];  // coalesced
  __syncthreads();
  float M = -INFINITY;
  for (int s = 0; s < nch; ++s) M = fmaxf(M, mls[s].x);
  float L = 0.f, o = 0.f;
  const float* po = part_o + row * nch * d + c;
#pragma unroll 8
  for (int s = 0; s < nch; ++s) {
    const float2 m = mls[s];
    const float w = m.x != -INFINITY ? __expf(m.x - M) : 0.f;
    L += w * m.y;
    o += w * po[(int64_t)s * d];
  }
  out[row * d + c] = __float2bfloat16_rn(o / L);
}

}  // namespace

namespace {

inline unsigned blocks_for(int64_t n, int per) { return (unsigned)((n + per - 1) / per); }

}  // namespace

// Slots of a KV-head's entries: one CTA per SM and layer over all KV-heads, of 128 entries or
// more (a shorter slot is all pipeline fill and combination). It depends on one layer's shape
// only, so that a layer's result does not depend on the layers it is launched with.
int decode_slots(int64_t entries, int H, int num_sms) {
  return (int)std::max<int64_t>(
      1, std::min<int64_t>((entries + 127) / 128, (int64_t)num_sms / std::max(1, H)));
}

size_t decode_workspace_bytes(int64_t rows, int nslots, int d, int layers) {
  if (nslots == 1) return 0;  // the chunk kernel writes the output itself
  const size_t r = (size_t)rows * layers * nslots;
  return r * d * 4 + 256 + r * 8 + 256;
}

template <int D, int R>
static cudaError_t launch_decode_chunks(const DecodeStack& st, int nslots, int nrb, float* part_o,
                                        float2* part_ml, cudaStream_t s) {
  const dim3 grid(nslots * nrb, st.layer[0].H, st.n);
  decode_chunk_kernel<D, R><<<grid, 32 * DecShape<D>::kWarps, 0, s>>>(st, nslots, nrb, part_o,
                                                                      part_ml);
  return cudaGetLastError();
}

cudaError_t launch_decode_biased(const DecodeStack& st, void* ws, int num_sms, cudaStream_t s,
                                 int* launches) {
  *launches = 0;
  if (st.n < 1 || st.n > kDecodeMaxLayers) return cudaErrorInvalidValue;
  const DecodeArgs& a = st.layer[0];  // every layer has the same shape
  const int64_t E = a.t + a.S;
  const int nslots = decode_slots(E, a.H, num_sms);
  const int G = a.nq * (a.Hq / a.H);
  const int R = G <= 4 ? 4 : 8;  // query rows per row block
  const int nrb = (G + R - 1) / R;
  const int64_t rows = (int64_t)a.nq * a.Hq;
  float* part_o = static_cast<float*>(ws);
  float2* part_ml = reinterpret_cast<float2*>(
      static_cast<uint8_t*>(ws) +
      (((size_t)rows * st.n * nslots * a.d * 4 + 255) & ~size_t(255)));
  auto launch = [&](auto r8) -> cudaError_t {
    constexpr int RR = decltype(r8)::value ? 8 : 4;
    switch (a.d) {
      case 64: return launch_decode_chunks<64, RR>(st, nslots, nrb, part_o, part_ml, s);
      case 128: return launch_decode_chunks<128, RR>(st, nslots, nrb, part_o, part_ml, s);
      case 256: return launch_decode_chunks<256, RR>(st, nslots, nrb, part_o, part_ml, s);
    }
    return cudaErrorInvalidValue;
  };
  cudaError_t e = R == 4 ? launch(std::false_type{}) : launch(std::true_type{});
  if (e != cudaSuccess) return e;
  *launches = 1;
  if (nslots == 1) return cudaSuccess;
  launch_chained(decode_merge_kernel, dim3((unsigned)rows, st.n), a.d, nslots * sizeof(float2), s,
                 1, st, part_o, part_ml, rows, nslots, a.d);
  *launches = 2;
  return cudaGetLastError();
}

cudaError_t launch_fold_weights(const __nv_bfloat16* WkT, const float* bk, int n, int D, int d2,
                                int Kp, __nv_bfloat16* Wt, cudaStream_t s) {
  const int64_t total = (int64_t)n * Kp * D;
  fold_weights_kernel<<<blocks_for(total, 256), 256, 0, s>>>(WkT, bk, n, D, d2, Kp, Wt);
  return cudaGetLastError();
}

cudaError_t launch_f32_hilo(const float* x, int64_t rows, int C, __nv_bfloat16* out,
                            cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  f32_hilo_kernel<<<blocks_for(rows * C, 256), 256, 0, s>>>(x, rows, C, out);
  return cudaGetLastError();
}

cudaError_t launch_beta(const __nv_bfloat16* Z, int t, int H, int D, const float* w,
                        float beta_max, float offset, float* beta, cudaStream_t s) {
  const int64_t rows = (int64_t)H * t;
  if (rows == 0) return cudaSuccess;
  launch_chained(beta_kernel, blocks_for(rows, 8), 256, 0, s, 1, Z, rows, t, H, D, w, beta_max,
                 offset, beta);
  return cudaGetLastError();
}

template <int HD>
static cudaError_t launch_strip_d(const KVSource& src, int64_t N, int H, const PosSegs& segs,
                                  const double* omega, int rope_fix, int vec, int x16, int Kp,
                                  __nv_bfloat16* X, __half* XT, int64_t Np, float2* gd,
                                  double origin, int G, const KernelTable& dev, cudaStream_t s) {
  constexpr int smem = kStripTok * (2 * HD + 2 + HD + 2) * 2;
  const cudaError_t ready = dev.of<KernelId<strip_kernel<HD>, 256, smem>>().status;
  if (ready != cudaSuccess) return ready;
  // Shares of the heads only while the token tiles leave SMs without two CTAs: each share forms
  // the tile's angles again, at the fp64 rate.
  const int64_t tiles = Np / kStripTok;
  const int shares = (int)std::max<int64_t>(1, std::min<int64_t>(H, 2 * dev.num_sms / tiles));
  strip_kernel<HD><<<dim3((unsigned)tiles, shares), 256, smem, s>>>(
      src, N, H, segs, omega, rope_fix, vec, x16, Kp, X, XT, Np, gd, origin, G);
  return cudaGetLastError();
}

cudaError_t launch_strip(const KVSource& src, int64_t N, int H, int d, const PosSegs& segs,
                         const double* omega, int rope_fix, __nv_bfloat16* X, __half* XT,
                         int64_t Np, float2* gd, double origin, int G, int x16, int Kp,
                         const KernelTable& dev, cudaStream_t s) {
  if (Np < kStripTok || Np % kStripTok != 0 || (Kp != 0 && (Kp % 64 != 0 || Kp < 2 * d + 1)))
    return cudaErrorInvalidValue;
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const bool second = src.n_split < N;
  const int vec = al16(src.K) && al16(src.V) && src.sN % 8 == 0 && src.sH % 8 == 0 &&
                  (!second || (al16(src.K2) && al16(src.V2) && src.sN2 % 8 == 0 &&
                               src.sH2 % 8 == 0));
  auto launch = [&](auto hd) {
    return launch_strip_d<decltype(hd)::value>(src, N, H, segs, omega, rope_fix, vec, x16, Kp, X,
                                               XT, Np, gd, origin, G, dev, s);
  };
  switch (d) {
    case 64: return launch(std::integral_constant<int, 64>{});
    case 128: return launch(std::integral_constant<int, 128>{});
    case 256: return launch(std::integral_constant<int, 256>{});
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_rope_tables(const RopeTables& tb, cudaStream_t s) {
  const int64_t n = ((int64_t)tb.G + kPosGrain) * (tb.D / 4) + (int64_t)tb.t * tb.hd;
  launch_chained(rope_tables_kernel, blocks_for(n, 256), 256, 0, s, 1, tb);
  return cudaGetLastError();
}

cudaError_t launch_q_rope(const float* qhat, const float* scale, int t_max, int b0, int nb, int t,
                          int D, double qstart, double qstep, const double* omega_c, int use_rope,
                          __nv_bfloat16* qhl, int fp16, float qscale, int num_sms,
                          cudaStream_t s) {
  if (D % 256 != 0) return cudaErrorInvalidValue;
  const int64_t n = (int64_t)t * (D / 8);
  const unsigned tiles = blocks_for(n, 256);
  // shares of the batches until each SM has three CTAs
  const unsigned shares = std::max(1u, std::min((unsigned)nb, 3u * num_sms / tiles));
  launch_chained(q_rope_kernel, dim3(tiles, shares), 256, 0, s, 1, qhat, scale, t_max, b0, nb,
                 t, D, qstart, qstep, omega_c, use_rope, qhl, fp16, qscale);
  return cudaGetLastError();
}

template <typename OutT, bool HILO = false>
static bool softmax_reg(const float* S, int64_t rows, int64_t ncols, int64_t ldS, void* P,
                        int64_t ldP, cudaStream_t s) {
  const int64_t need = std::max(ldP, ncols);
  OutT* Pt = static_cast<OutT*>(P);
  if ((ldS % 4) != 0 || (ldP % 4) != 0) return false;
  if (need <= 1024)
    launch_chained(softmax_reg_kernel<OutT, 4, HILO>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   Pt, ldP);
  else if (need <= 2048)
    launch_chained(softmax_reg_kernel<OutT, 8, HILO>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   Pt, ldP);
  else if (need <= 4096)
    launch_chained(softmax_reg_kernel<OutT, 16, HILO>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   Pt, ldP);
  else if (need <= 8192)
    launch_chained(softmax_reg_kernel<OutT, 32, HILO>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   Pt, ldP);
  else if (need <= 16384)
    launch_chained(softmax_reg_kernel<OutT, 64, HILO>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   Pt, ldP);
  else
    return false;
  return true;
}

cudaError_t launch_wait_timeout_selftest(int* err, unsigned long long limit_ns, cudaStream_t s) {
  wait_timeout_selftest_kernel<<<1, 32, 0, s>>>(err, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_omega(double* out, int half, int width, double base, cudaStream_t s) {
  omega_kernel<<<blocks_for(half, 256), 256, 0, s>>>(out, half, width, base);
  return cudaGetLastError();
}

cudaError_t launch_softmax(const float* S, int64_t rows, int64_t ncols, int64_t ldS, void* P,
                           int64_t ldP, int out_fp16, cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  if (out_fp16 == 2 || out_fp16 == 3) {  // bf16 (2) or fp16 (3) hi | lo rows
    if (!(out_fp16 == 2 ? softmax_reg<__nv_bfloat16, true>(S, rows, ncols, ldS, P, ldP, s)
                        : softmax_reg<__half, true>(S, rows, ncols, ldS, P, ldP, s)))
      return cudaErrorInvalidValue;
    return cudaGetLastError();
  }
  if (out_fp16 ? softmax_reg<__half>(S, rows, ncols, ldS, P, ldP, s)
               : softmax_reg<__nv_bfloat16>(S, rows, ncols, ldS, P, ldP, s))
    return cudaGetLastError();
  if (out_fp16)
    launch_chained(softmax_kernel<__half>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   static_cast<__half*>(P), ldP);
  else
    launch_chained(softmax_kernel<__nv_bfloat16>, (unsigned)rows, 256, 0, s, 1, S, ncols, ldS,
                   static_cast<__nv_bfloat16*>(P), ldP);
  return cudaGetLastError();
}

cudaError_t launch_ca_merge(const float* O, const float2* stats, int nsplit, int b0, int nb,
                            int n, int t, int d2, int f16, __nv_bfloat16* PX, cudaStream_t s) {
  const int64_t total = (int64_t)nb * t * d2;
  if (total == 0) return cudaSuccess;
  if (nsplit < 1 || nsplit > 32) return cudaErrorInvalidValue;
  auto launch = [&](auto groups) {
    launch_chained(ca_merge_kernel<decltype(groups)::value>, blocks_for((int64_t)nb * t, 8), 256,
                   0, s, 1, O, stats, nsplit, b0, nb, n, t, f16, PX);
    return cudaGetLastError();
  };
  switch (d2) {
    case 128: return launch(std::integral_constant<int, 1>{});
    case 256: return launch(std::integral_constant<int, 2>{});
    case 512: return launch(std::integral_constant<int, 4>{});
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_rmsnorm(const void* in, int in_bf16, int64_t rows, int D, int64_t ldi,
                           float eps, __nv_bfloat16* out, int64_t ldo, int hilo, cudaStream_t s) {
  launch_chained(rmsnorm_kernel, blocks_for(rows, 8), 256, 0, s, 1, in, in_bf16, rows, D, ldi, eps,
                 out, ldo, hilo);
  return cudaGetLastError();
}

cudaError_t launch_bf16_to_f16(void* p, int64_t n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  bf16_to_f16_kernel<<<blocks_for(n, 256), 256, 0, s>>>(static_cast<uint16_t*>(p), n);
  return cudaGetLastError();
}

cudaError_t launch_scale_rows(float* x, const float* inv, int64_t rows, int D, cudaStream_t s) {
  launch_chained(scale_rows_kernel, blocks_for(rows * D, 256), 256, 0, s, 1, x, inv, rows, D);
  return cudaGetLastError();
}

cudaError_t launch_inv_norms(const float* parts, int64_t nvec, int nparts, int64_t block, float eps,
                             float alpha, float* out, cudaStream_t s) {
  if (block < 1) return cudaErrorInvalidValue;
  launch_chained(inv_norms_kernel, blocks_for(nvec, 256), 256, 0, s, 1, parts, nvec, nparts, block,
                 eps, alpha, out);
  return cudaGetLastError();
}

cudaError_t launch_transpose(const __nv_bfloat16* in, int64_t R, int64_t C, __nv_bfloat16* out,
                             int perm_D, cudaStream_t s, int key_rows) {
  dim3 grid(blocks_for(C, 32), blocks_for(R, 32));
  transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(in, R, C, out, perm_D, key_rows);
  return cudaGetLastError();
}

cudaError_t launch_bias(const __nv_bfloat16* in, const __nv_bfloat16* in2, int64_t C,
                        float* out, int perm_D, cudaStream_t s) {
  bias_kernel<<<blocks_for(C, 256), 256, 0, s>>>(in, in2, C, out, perm_D);
  return cudaGetLastError();
}

}  // namespace still
