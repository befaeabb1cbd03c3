// Key projection of one compactor layer, for sm_103a (App. A, "Cross-attention" keys):
//
//   k~ = X W_K,i + b_K,i ;  |k~|^2 partials ;  k = RoPE_c(k~, p_n) -> hi | lo
//
// X rows are [X hi (2d) | lo of the key half (d)], W rows W_K^T [2d]: K = 3d, so a 256 x 256
// output tile costs little tensor work for its 256 KB of k. The kernel is bound by its epilogue
// and by the bytes it moves, and both are what its layout is for.
//
// CTA pairs (clusters of two) with 2-SM MMAs (cta_group::2, M = 256, issued by the even CTA):
// CTA x holds the A rows of m-tile 2 m + x and rows [128 x, +128) of the 256-column W tile.
//   W resident  the 2d / 64 chunks of the pair's W tile stay in shared memory while the pair
//               walks m-tiles; the key-half chunks serve both the hi and the lo pass. Per tile
//               and SM that leaves the 3d / 64 chunks of X to load: 96 KB at d = 128 and 192 KB
//               at d = 256, half of what streaming both operands takes.
//   order       (KV-head, band of kBand m-tile pairs, W tile, m-tile pair), each pair of CTAs a
//               contiguous range: X is read from HBM about once (a band of X stays in L2 while
//               the W tiles pass), and W, with the bias and the 32 KB slice of the RoPE offset
//               table that go with it, changes once per band.
//   epilogue    8 warps (each thread may hold 168 registers), each 32 rows x 64 RoPE pairs of a
//               tile. tcgen05.ld.16x256b gives a thread two neighbouring columns of every 8; the
//               rows of W are ordered (key_row_source) so that those are 8 neighbouring columns
//               of k: the 4 threads of a row write 64 contiguous bytes straight from registers,
//               8 rows per store instruction, with no transpose, fence or copy engine. A thread
//               holds 4 rows of the same columns, so the coarse angles and the bias are read
//               once for all four. Rotation in packed fp32 pairs; streaming stores (k is larger
//               than L2).
//
// Measured (one layer): 32k tokens, d = 128, 64 (h, i) pairs of width 1024: 2.67 -> 2.2 ms (8.6 GB of
// k: 3.9 TB/s); 128k tokens, d = 256, 128 pairs of width 2048: 52.3 -> 44 ms; against the generic
// 2-SM GEMM with an epilogue that transposed through shared memory and stored 32-byte rows by
// TMA. At d = 128 what is left is the LSU pipe (two thirds busy: offset-angle reads and stores
// that span 8 rows); at d = 256 the X ring's depth (64 KB next to 128 KB of W): with no tables
// and six slots a copy of the kernel took 37 ms. Measured and dropped: 16 epilogue warps with 104
// registers each (2.32 ms), 12 with 128 (2.55 ms), a 3-slot ring with the coarse angles brought
// to shared memory (2.38 and 51 ms), offset angles in registers with coarse rows every 8
// positions read by LDG (2.70 and 48 ms).
//
// Every wait is bounded; a wait that runs out is recorded and the CTA drains and leaves.
#pragma once
#include "gemm_host.cuh"

namespace still {

// Key positions: the compactor angle p_n * omega_m is split as G_g * omega_m + i * omega_m +
// f * omega_m with delta = p_n - G_g in [0, kPosGrain), i = floor(delta) and f = delta - i: the
// first two rotations come from tables built per call in fp64 (coarse, fine), the third (only
// for fractional positions, |f * omega_m| < 1) from Taylor series; the three are combined by the
// angle-addition formulas. Every rotation is thus accurate to fp32 rounding; forming
// delta * omega_m in fp32 instead would leave angle errors near 2e-6 rad at delta ~ 31. The
// per-token (g, delta) come from a table formed once per call in fp64, so the epilogue itself
// does no fp64 arithmetic.
struct KeyProjParams {
  __nv_bfloat16* out = nullptr;     // [heads * nh][N][2D]: hi at [0, D), lo at [D, 2D)
  float* sumsq = nullptr;           // [heads * nh][kKeyParts * D / 256][N] partials (part-major)
  const float* bias = nullptr;      // [nh * D], pair-chunk order
  const float4* coarse = nullptr;   // [G][D / 4]: (c, c, s, s) of pairs 2 q, 2 q + 1 at G_g
  const float4* fine = nullptr;     // [D / 4][kPosGrain]: the same at offset i, i fastest
  const float* omega = nullptr;     // [D / 2] fp32
  const float2* gd = nullptr;       // [N]: (coarse index g as float, delta)
  int32_t N = 0;                    // tokens per KV-head
  int32_t D = 0, nh = 0, heads = 0; // width of a head, cross heads and KV-heads of this launch
  int32_t ncoarse = 0;
  int32_t pbands = 1;               // bands per phase (see KeyWalk); set by the launcher
  int32_t a_row0 = 0, b_row0 = 0;   // first X row (KV-head h0) and first W row (cross head i0)
  uint32_t idesc = 0;
  int* err = nullptr;
};

constexpr int kKeyParts = 2;   // |k~|^2 partials per 256 columns

// m-tile pairs per band: 4096 tokens, 3 MB of X at d = 128 and 6 MB at d = 256 (43.4 ms a layer of
// 128k tokens at d = 256; 45.2 with 64 and 32 MB phases, where X is read from HBM more often).
constexpr int kBand = 16;
constexpr int64_t kPhaseBytes = 7 << 20;  // X of a phase
constexpr int kKeyEpiWarps = 8;  // two per TMEM lane quarter
constexpr int kKeyThreads = 64 + 32 * kKeyEpiWarps;

template <int NB>  // W chunks of 64 (2d / 64)
struct KeyProjSmem {
  static constexpr int kSlots = NB + NB / 2;               // A chunks per tile: X hi, X lo
  static constexpr int kChunkBytes = kBM * kBK * 2;        // 128 rows x 64, 16 KB
  static constexpr int kStages = NB == 8 ? 4 : 6;          // A ring
  static constexpr int kAOffset = NB * kChunkBytes;
  static constexpr int kFineOffset = kAOffset + kStages * kChunkBytes;  // [64][kPosGrain] float4
  static constexpr int kBiasOffset = kFineOffset + 64 * kPosGrain * 16;  // [256] float
  static constexpr int kBarOffset = kBiasOffset + 1024;
  static constexpr int kBytes = kBarOffset + 256 + 1024;
  static_assert(kBytes <= 232448, "shared memory budget");
};

// The tiles of a pair of CTAs. The order of all tiles is (KV-head, band, W tile, m-tile pair); a
// phase is `pbands` consecutive bands, and each pair takes a contiguous range of every phase
// (which pair takes which range rotates, so that ranges one tile longer even out). All pairs
// are thus in the same few bands of X at a time.
struct KeyWalk {
  int mp, tiles_n, heads, nbands, pbands;  // m-tile pairs and bands per KV-head, bands per phase
  int ph, left;                            // phase, tiles left in it
  int hd, band, tn, m, mb;                 // current tile; m: m-tile pair inside the band of mb
  bool new_w;                              // the W tile differs from the previous tile's

  __device__ __forceinline__ void init(const KeyProjParams& p) {
    mp = (p.N + 2 * kBM - 1) / (2 * kBM);
    tiles_n = p.nh * p.D / 256;
    heads = p.heads;
    nbands = (mp + kBand - 1) / kBand;
    pbands = p.pbands;
    ph = -1;
    left = 0;
    tn = -1;
  }
  // tiles before band b of all bands (KV-head b / nbands)
  __device__ __forceinline__ int64_t before(int b) const {
    return (int64_t)tiles_n * ((int64_t)(b / nbands) * mp + (b % nbands) * kBand);
  }
  __device__ __forceinline__ void enter(int64_t tile) {
    const int64_t per_head = (int64_t)tiles_n * mp;
    hd = (int)(tile / per_head);
    int64_t r = tile % per_head;
    band = (int)(r / ((int64_t)kBand * tiles_n));
    r -= (int64_t)band * kBand * tiles_n;
    mb = min(kBand, mp - band * kBand);
    tn = (int)(r / mb);
    m = (int)(r % mb);
  }
  __device__ __forceinline__ bool next(int cid, int ncl) {
    if (left > 0) {
      --left;
      const int was = tn;
      if (++m == mb) {
        m = 0;
        if (++tn == tiles_n) {
          tn = 0;
          if (++band == nbands) {
            band = 0;
            ++hd;
          }
          mb = min(kBand, mp - band * kBand);
        }
      }
      new_w = tn != was;
      return true;
    }
    for (;;) {
      ++ph;
      if (ph * pbands >= heads * nbands) return false;
      const int64_t c0 = before(ph * pbands);
      const int64_t n = before(min((ph + 1) * pbands, heads * nbands)) - c0;
      const int64_t who = ((int64_t)cid + (int64_t)ph * (ncl * 3 / 8)) % ncl;
      const int64_t t0 = c0 + n * who / ncl, t1 = c0 + n * (who + 1) / ncl;
      if (t1 == t0) continue;
      const int was = tn;
      enter(t0);
      left = (int)(t1 - t0) - 1;
      new_w = tn != was;
      return true;
    }
  }
  __device__ __forceinline__ int m_pair() const { return band * kBand + m; }
};

// kFrac: some key positions are fractional (the sub-unit rotation is compiled in only then, so
// the integer-position kernel keeps its registers). kF16: k as fp16 hi | lo instead of bf16.
template <int NB, bool kFrac, bool kF16>
__global__ void __launch_bounds__(kKeyThreads, 1)
    key_proj_kernel(const __grid_constant__ CUtensorMap tmA,
                    const __grid_constant__ CUtensorMap tmB, const KeyProjParams p) {
  using S = KeyProjSmem<NB>;
  constexpr int kStages = S::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* afull = reinterpret_cast<uint64_t*>(smem + S::kBarOffset);  // even CTA's
  uint64_t* aempty = afull + kStages;
  uint64_t* bfull = aempty + kStages;  // [NB], even CTA's: chunk c of the W tile loaded
  uint64_t* bempty = bfull + NB;       // the W tile's last MMA is done
  uint64_t* tfull = bempty + 1;        // [2]
  uint64_t* tempty = tfull + 2;        // [2], even CTA's
  uint64_t* slice = tempty + 2;        // the epilogue warps' meeting point at a new W tile
  uint64_t* drain = slice + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int x = (int)(rank & 1u);
  const bool leader = x == 0;
  const uint16_t pair_mask = (uint16_t)((1u << rank) | (1u << (rank ^ 1u)));
  const int cid = (int)cluster_id_x(), ncl = (int)cluster_count_x();

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);
    }
    for (int c = 0; c < NB; ++c) mbar_init(&bfull[c], 1);
    mbar_init(bempty, 1);
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 2 * kKeyEpiWarps);
    }
    mbar_init(slice, kKeyEpiWarps);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) {
    tmem_alloc_2sm(tmem_slot, 512);
    tmem_relinquish_2sm();
  }
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  griddep_wait();
  const uint32_t l_afull = cluster_map(smem_u32(afull), rank & ~1u);
  const uint32_t l_bfull = cluster_map(smem_u32(bfull), rank & ~1u);
  const uint32_t l_tempty = cluster_map(smem_u32(tempty), rank & ~1u);

  if (warp == 0) {
    if (lane == 0) {
      // ------------------------------------------------------------ TMA producer
      int stage = 0;
      uint32_t phase = 0, nb = 0;  // nb: W tiles loaded
      uint32_t armed = 0, armed_par = 0;
      bool bad = false;
      auto fail = [&](int where) {
        dev_set_error(p.err, DEV_WAIT_TIMEOUT, where);
        *abort_flag = 1;
        bad = true;
      };
      auto load_w = [&](int tn) {
        if (!mbar_wait(bempty, (nb & 1) ^ 1)) {
          fail(120);
          return;
        }
        ++nb;
        for (int c = 0; c < NB; ++c) {
          if (leader) mbar_arrive_expect_tx(&bfull[c], 2 * S::kChunkBytes);
          tma_load_2d_2sm(smem + c * S::kChunkBytes, &tmB, l_bfull + 8u * (uint32_t)c, c * kBK,
                          p.b_row0 + tn * 256 + 128 * x);
        }
      };
      KeyWalk k;
      k.init(p);
      while (!bad && !*abort_flag && k.next(cid, ncl)) {
        const int32_t row = p.a_row0 + k.hd * p.N + (2 * k.m_pair() + x) * kBM;
        for (int s = 0; s < S::kSlots && !bad; ++s) {
          if (!mbar_wait(&aempty[stage], phase ^ 1)) {
            fail(121);
            break;
          }
          if (leader) {
            mbar_arrive_expect_tx(&afull[stage], 2 * S::kChunkBytes);
            armed |= 1u << stage;
            armed_par = (armed_par & ~(1u << stage)) | (phase << stage);
          }
          tma_load_2d_2sm(smem + S::kAOffset + stage * S::kChunkBytes, &tmA,
                          l_afull + 8u * (uint32_t)stage, s * kBK, row);
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1;
          }
          // A new W tile overwrites the old one after its last MMA: first fill the ring with
          // the tile's X chunks, which need no W to arrive.
          if (k.new_w && s + 1 == min(kStages, S::kSlots)) load_w(k.tn);
        }
      }
      // every slot released by the even CTA's MMAs before the CTA may leave
      for (int i = 0; i < kStages && !bad && !*abort_flag; ++i) {
        if (!mbar_wait(&aempty[stage], phase ^ 1)) {
          fail(122);
          break;
        }
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (*abort_flag && leader) {  // copies in flight land before the CTA leaves
        for (int s = 0; s < kStages; ++s)
          if (armed & (1u << s)) (void)mbar_wait_cluster(&afull[s], (armed_par >> s) & 1);
        if (nb > 0)
          for (int c = 0; c < NB; ++c) (void)mbar_wait_cluster(&bfull[c], (nb - 1) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ------------------------------------------------------------ MMA issuer (2-SM)
      int stage = 0;
      uint32_t phase = 0, nb = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool issued = false, bad = false;
      auto fail = [&](int where) {
        dev_set_error(p.err, DEV_WAIT_TIMEOUT, where);
        *abort_flag = 1;
        bad = true;
      };
      KeyWalk k;
      k.init(p);
      while (!bad && !*abort_flag && k.next(cid, ncl)) {
        if (k.new_w && issued) tc_commit_2sm_mc(bempty, pair_mask);  // the previous W tile's MMAs
        if (!mbar_wait_cluster(&tempty[acc], acc_phase ^ 1)) {
          fail(123);
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 256);
        for (int s = 0; s < S::kSlots; ++s) {
          const int c = s < NB ? s : s - NB;  // X hi chunk s, then X lo chunk s - NB
          if (k.new_w && s < NB && !mbar_wait_cluster(&bfull[c], nb & 1)) {
            fail(124);
            break;
          }
          if (!mbar_wait_cluster(&afull[stage], phase)) {
            fail(125);
            break;
          }
          tc_fence_after();
          const uint64_t ad =
              sdesc_k_sw128(smem_u32(smem + S::kAOffset + stage * S::kChunkBytes));
          const uint64_t bd = sdesc_k_sw128(smem_u32(smem + c * S::kChunkBytes));
#pragma unroll
          for (int q = 0; q < kBK / 16; ++q)
            tc_mma_f16_2sm(d_tmem, ad + 2 * q, bd + 2 * q, p.idesc, (s > 0 || q > 0) ? 1u : 0u);
          issued = true;
          tc_commit_2sm_mc(&aempty[stage], pair_mask);
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (bad) break;
        tc_commit_2sm_mc(&tfull[acc], pair_mask);
        if (++acc == 2) {
          acc = 0;
          acc_phase ^= 1;
        }
        if (k.new_w) ++nb;
      }
      if ((bad || *abort_flag) && issued) {
        tc_commit_2sm_mc(drain, (uint16_t)(1u << rank));
        (void)mbar_wait(drain, 0);
      }
    }
  } else {
    // -------------------------------------------------------------- epilogue (warps 2..9)
    const int ew = warp - 2;
    const int quarter = warp & 3;  // TMEM lanes [32 quarter, +32)
    const int half = ew >> 2;      // RoPE pairs [64 half, +64) of the tile's 128
    const int lr = lane >> 2, l4 = lane & 3;  // rows lr + 8 i, columns 8 l4 .. + 7 of every 32
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    float4* fine = reinterpret_cast<float4*>(smem + S::kFineOffset);
    float4* bias = reinterpret_cast<float4*>(smem + S::kBiasOffset);
    int acc = 0;
    uint32_t acc_phase = 0, n_meet = 0;
    bool bad = false;
    auto wait_all = [&](uint64_t* bar, uint32_t parity) {
      bool ok = mbar_wait(bar, parity);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) {
          dev_set_error(p.err, DEV_WAIT_TIMEOUT, 126);
          *abort_flag = 1;
        }
        bad = true;
      }
      return ok;
    };
    auto meet = [&]() {  // every epilogue warp has come this far
      __syncwarp();
      if (lane == 0) mbar_arrive(slice);
      return wait_all(slice, n_meet++ & 1);
    };
    auto load_gd = [&](int r0) {  // lane = row
      return r0 + lane < p.N ? p.gd[r0 + lane] : make_float2(0.f, 0.f);
    };
    // this thread's pair of pairs (columns 8 l4 of block blk) of W tile tn, inside its head
    auto quad0 = [&](int tn, int blk) {
      return (((tn * 256) % p.D) >> 2) + 16 * (2 * half + blk) + 4 * l4;
    };
    auto load_coarse = [&](float4 (&cv)[4], int g, int q) {
      const float4* cr = p.coarse + (int64_t)g * (p.D / 4) + q;
#pragma unroll
      for (int j = 0; j < 4; ++j) cv[j] = cr[j];
    };
    // (g, i) of a row: g in the upper bits, i below kPosGrain
    auto pack_gi = [&](float2 v) {
      return (max(0, min((int)v.x, p.ncoarse - 1)) << 5) | max(0, min((int)v.y, kPosGrain - 1));
    };
    static_assert(kPosGrain == 32, "pack_gi");
    KeyWalk k;
    k.init(p);
    bool more = k.next(cid, ncl);
    auto token0 = [&]() {  // first token of this warp's rows
      return (2 * k.m_pair() + x) * kBM + quarter * 32;
    };
    float2 gnext = more ? load_gd(token0()) : make_float2(0.f, 0.f);
    float4 cnext[4];  // the next tile's first coarse row, in flight during this tile
    if (more)
      load_coarse(cnext, __shfl_sync(0xffffffffu, pack_gi(gnext), lr) >> 5, quad0(k.tn, 0));
    bool met = false;
    while (more && !bad) {
      const int row0 = token0(), hd = k.hd, tn = k.tn;
      const float2 gdr = gnext;
      const bool reload = k.new_w;
      more = k.next(cid, ncl);
      if (more) gnext = load_gd(token0());
      const int c_tile = tn * 256;
      const int head = c_tile / p.D, f_tile = c_tile - head * p.D;
      if (reload) {  // this W tile's offset-table slice and bias
        if (met && !meet()) break;  // nobody reads the old ones any more
        met = true;
        // entry i of quad q sits at i + 2 (q / 4 % 4): the four threads of a row then read from
        // different banks
        const float4* src = p.fine + (int64_t)(f_tile >> 2) * kPosGrain;
        for (int e = threadIdx.x - 64; e < 64 * kPosGrain; e += 32 * kKeyEpiWarps)
          fine[(e & ~31) | ((e + 2 * (e >> 7 & 3)) & 31)] = src[e];
        if (threadIdx.x - 64 < 64)
          bias[threadIdx.x - 64] = reinterpret_cast<const float4*>(p.bias + c_tile)[threadIdx.x - 64];
        if (!meet()) break;
      }
      // (g, i) of this thread's rows lr + 8 r, from the lanes that hold them
      const int gi = pack_gi(gdr);
      const float frac = gdr.y - (float)(gi & 31);  // exact; 0 for integer positions
      const bool any_frac = kFrac && __any_sync(0xffffffffu, frac != 0.f);
      int rgi[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) rgi[r] = __shfl_sync(0xffffffffu, gi, lr + 8 * r);
      const bool one_g =
          __all_sync(0xffffffffu, ((rgi[0] ^ rgi[1]) | (rgi[0] ^ rgi[2]) | (rgi[0] ^ rgi[3])) < 32);
      const int64_t z = (int64_t)hd * p.nh + head;
      float ss[4] = {0.f, 0.f, 0.f, 0.f};
      if (!wait_all(&tfull[acc], acc_phase)) break;
      if (warp_flag(abort_flag)) break;
      tc_fence_after();
      float4 cv[4], cblk[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) cv[j] = cnext[j];
      load_coarse(cblk, rgi[0] >> 5, quad0(tn, 1));
#pragma unroll
      for (int blk = 0; blk < 2; ++blk) {
        const int part = 2 * half + blk;  // pairs [32 part, +32) of the tile
        const int qh = quad0(tn, blk);    // this thread's first pair of pairs, in the head
        if (blk == 1) {
#pragma unroll
          for (int j = 0; j < 4; ++j) cv[j] = cblk[j];
          if (more)
            load_coarse(cnext, __shfl_sync(0xffffffffu, pack_gi(gnext), lr) >> 5, quad0(k.tn, 0));
        }
        float4 ba[2], bb[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          ba[e] = bias[8 * part + 2 * l4 + e];
          bb[e] = bias[32 + 8 * part + 2 * l4 + e];
        }
        const float4* fq = fine + (16 * part + 4 * l4) * kPosGrain;
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // rows 16 h + 8 s + lr
          uint32_t a[16], b[16];
          const uint32_t ta = lane_base + ((uint32_t)(16 * h) << 16) + (uint32_t)(acc * 256 + 32 * part);
          tmem_ld_16x256b_x4_2(ta, ta + 128u, a, b);
          if (blk == 1 && h == 1) {  // the accumulator is free
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_relaxed(l_tempty + 8u * (uint32_t)acc);
          }
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            const int r = 2 * h + s;
            if (!one_g && r > 0) load_coarse(cv, rgi[r] >> 5, qh);
            const float4* fr = fq + ((rgi[r] + 2 * l4) & 31);
            float fs = 0.f;
            if constexpr (kFrac) fs = __shfl_sync(0xffffffffu, frac, lr + 8 * r);
            uint64_t ss2 = 0ull;  // (0.f, 0.f)
            uint32_t ha[4], la[4], hb[4], lb[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // columns 8 l4 + 2 j, + 1 of the 32, and 128 further
              const float4 fv = fr[j * kPosGrain];
              const float4 b4 = bb[j >> 1], a4 = ba[j >> 1];
              const uint64_t cc = pack2(cv[j].x, cv[j].y), sc = pack2(cv[j].z, cv[j].w);
              const uint64_t cf = pack2(fv.x, fv.y), sf = pack2(fv.z, fv.w);
              const uint64_t xx =
                  add2(pack2(__uint_as_float(a[4 * j + 2 * s]), __uint_as_float(a[4 * j + 2 * s + 1])),
                       (j & 1) ? pack2(a4.z, a4.w) : pack2(a4.x, a4.y));
              const uint64_t yy =
                  add2(pack2(__uint_as_float(b[4 * j + 2 * s]), __uint_as_float(b[4 * j + 2 * s + 1])),
                       (j & 1) ? pack2(b4.z, b4.w) : pack2(b4.x, b4.y));
              ss2 = fma2(xx, xx, fma2(yy, yy, ss2));
              uint64_t cw = fma2(cc, cf, neg2(mul2(sc, sf)));  // cos(G w + i w)
              uint64_t sw = fma2(sc, cf, mul2(cc, sf));        // sin(G w + i w)
              if constexpr (kFrac) {
                if (any_frac) {  // + f w, |f w| < 1
                  const float2 w2 = *reinterpret_cast<const float2*>(p.omega + 2 * (qh + j));
                  float s3[2], c3[2];
                  sincos_taylor(fs * w2.x, &s3[0], &c3[0]);
                  sincos_taylor(fs * w2.y, &s3[1], &c3[1]);
                  const uint64_t s32 = pack2(s3[0], s3[1]), c32 = pack2(c3[0], c3[1]);
                  const uint64_t c2 = fma2(cw, c32, neg2(mul2(sw, s32)));
                  sw = fma2(sw, c32, mul2(cw, s32));
                  cw = c2;
                }
              }
              split2<kF16>(fma2(xx, cw, neg2(mul2(yy, sw))), ha[j], la[j]);
              split2<kF16>(fma2(xx, sw, mul2(yy, cw)), hb[j], lb[j]);
            }
            float s0, s1;
            unpack2(ss2, s0, s1);
            ss[r] += s0 + s1;
            const int row = row0 + lr + 8 * r;
            if (row < p.N) {
              __nv_bfloat16* o = p.out + (z * p.N + row) * (2 * (int64_t)p.D) + f_tile + 32 * part +
                                 8 * l4;
              __stcs(reinterpret_cast<uint4*>(o), make_uint4(ha[0], ha[1], ha[2], ha[3]));
              __stcs(reinterpret_cast<uint4*>(o + p.D), make_uint4(la[0], la[1], la[2], la[3]));
              __stcs(reinterpret_cast<uint4*>(o + 128), make_uint4(hb[0], hb[1], hb[2], hb[3]));
              __stcs(reinterpret_cast<uint4*>(o + p.D + 128), make_uint4(lb[0], lb[1], lb[2], lb[3]));
            }
          }
        }
      }
      if (++acc == 2) {
        acc = 0;
        acc_phase ^= 1;
      }
      const int parts = kKeyParts * (p.D / 256);
      float* sq = p.sumsq + (z * parts + (f_tile / 256) * kKeyParts + half) * p.N + row0 + lr;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float v = ss[r];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (l4 == r && row0 + lr + 8 * r < p.N) sq[8 * r] = v;
      }
    }
  }

  tc_fence_before();
  // No CTA frees its TMEM while the even CTA's MMAs may still write it, nor leaves while the
  // other may still copy into or arrive on its shared memory.
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_2sm(tmem_base, 512);
  }
}

// X: [H * N][3d] (hi | key lo), W: [n D][2d] rows in key_row_source order, both ab_fmt (1 bf16, 0
// fp16); d of 64, 128 or 256, D a multiple of 256.
template <int NB, bool kFrac, bool kF16>
inline cudaError_t launch_key_proj_as(const KernelTable& dev, const Operand2D& X,
                                      const Operand2D& W, KeyProjParams p, int ab_fmt,
                                      cudaStream_t stream) {
  using S = KeyProjSmem<NB>;
  if (p.N <= 0 || p.D <= 0 || p.D % 256 != 0 || p.nh <= 0 || p.heads <= 0 || X.cols != 96 * NB ||
      W.cols != 64 * NB || p.ncoarse < 1)
    return cudaErrorInvalidValue;
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, X, kBM) || !make_tmap(&tb, W, kBM)) return cudaErrorInvalidValue;
  p.idesc = idesc_f16(2 * kBM, 256, ab_fmt);
  using Id = KernelId<key_proj_kernel<NB, kFrac, kF16>, kKeyThreads, S::kBytes, 2>;
  if (dev.of<Id>().status != cudaSuccess) return dev.of<Id>().status;
  const int clusters = dev.persistent_clusters<Id>(2);
  const int mp = (p.N + 2 * kBM - 1) / (2 * kBM);
  const int64_t total = (int64_t)mp * (p.nh * (p.D / 256)) * p.heads;
  if (total > 0x7fffffff) return cudaErrorInvalidValue;
  // the X bands of a phase stay in L2 next to W and the k that passes through
  const int64_t band_bytes = (int64_t)std::min(mp, kBand) * 2 * kBM * X.pitch * 2;
  // and a phase gives every pair several tiles
  const int64_t band_tiles = (int64_t)kBand * (p.nh * (p.D / 256));
  p.pbands = (int)std::max<int64_t>({1, kPhaseBytes / band_bytes, 4 * clusters / band_tiles});
  return launch_chained(key_proj_kernel<NB, kFrac, kF16>,
                        2 * (int)std::min<int64_t>(total, clusters), kKeyThreads, S::kBytes, stream,
                        2, ta, tb, p);
}

inline cudaError_t launch_key_proj(const KernelTable& dev, const Operand2D& X, const Operand2D& W,
                                   const KeyProjParams& p, int d, bool frac, bool f16, int ab_fmt,
                                   cudaStream_t s) {
  auto pick = [&](auto nb) -> cudaError_t {
    constexpr int NB = decltype(nb)::value;
    if (frac)
      return f16 ? launch_key_proj_as<NB, true, true>(dev, X, W, p, ab_fmt, s)
                 : launch_key_proj_as<NB, true, false>(dev, X, W, p, ab_fmt, s);
    return f16 ? launch_key_proj_as<NB, false, true>(dev, X, W, p, ab_fmt, s)
               : launch_key_proj_as<NB, false, false>(dev, X, W, p, ab_fmt, s);
  };
  switch (d) {
    case 64: return pick(std::integral_constant<int, 2>{});
    case 128: return pick(std::integral_constant<int, 4>{});
    case 256: return pick(std::integral_constant<int, 8>{});
  }
  return cudaErrorInvalidValue;
}

}  // namespace still
