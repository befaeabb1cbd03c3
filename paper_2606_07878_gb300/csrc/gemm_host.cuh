// Host side of the tcgen05 GEMM: TMA descriptors, tile/split bookkeeping, launch.
#pragma once
#include <algorithm>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <utility>

#include "epilogues.cuh"
#include "kernel_table.cuh"
#include "launch.cuh"

namespace still {

// A 2-D row-major 16-bit operand as TMA sees it: `rows` rows of `cols` elements, row pitch
// `pitch` elements (pitch * 2 must be a multiple of 16 and ptr 16-byte aligned).
struct Operand2D {
  const void* ptr = nullptr;
  int64_t rows = 0, cols = 0, pitch = 0;
};

inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

// A 3-D destination for TMA stores: element (x, y, z) at base + z * zstride + y * ystride + x
// (elements), extents (nx, ny, nz); boxes of bx x 32 x 1, optionally 128-byte swizzled.
struct StoreView3D {
  void* ptr = nullptr;
  int elem_bytes = 2;
  int64_t nx = 0, ny = 0, nz = 1, ystride = 0, zstride = 0;
  int bx = 32;
  bool swizzle128 = false;
};

inline bool make_store_tmap(CUtensorMap* m, const StoreView3D& v) {
  auto enc = tensor_map_encoder();
  if (enc == nullptr) return false;
  const int64_t eb = v.elem_bytes;
  if ((reinterpret_cast<uintptr_t>(v.ptr) & 15) != 0 || (v.ystride * eb) % 16 != 0 ||
      (v.zstride * eb) % 16 != 0 || (v.bx * eb) % 16 != 0)
    return false;
  cuuint64_t dims[3] = {(cuuint64_t)v.nx, (cuuint64_t)v.ny, (cuuint64_t)v.nz};
  cuuint64_t strides[2] = {(cuuint64_t)(v.ystride * eb), (cuuint64_t)(v.zstride * eb)};
  cuuint32_t box[3] = {(cuuint32_t)v.bx, 32, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, eb == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                   3, v.ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   v.swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Box = box_rows x 64 elements, 128-byte swizzle, zero fill out of bounds.
inline bool make_tmap(CUtensorMap* m, const Operand2D& op, int box_rows) {
  auto enc = tensor_map_encoder();
  if (enc == nullptr) return false;
  if ((reinterpret_cast<uintptr_t>(op.ptr) & 15) != 0 || (op.pitch * 2) % 16 != 0) return false;
  cuuint64_t dims[2] = {(cuuint64_t)op.cols, (cuuint64_t)op.rows};
  cuuint64_t strides[1] = {(cuuint64_t)(op.pitch * 2)};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(op.ptr), dims,
                   strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Fills the derived fields of p. Returns false on an invalid description.
template <int BN>
inline bool finalize_gemm(GemmParams& p, int ab_fmt) {
  if (p.M <= 0 || p.N <= 0 || p.batch <= 0 || p.npass < 1 || p.npass > 3 || p.bdiv < 1)
    return false;
  int iters = 0;
  for (int i = 0; i < p.npass; ++i) {
    if (p.pass[i].klen <= 0 || p.pass[i].klen % kBK != 0) return false;
    if (p.pass[i].a_koff % 8 != 0 || p.pass[i].b_koff % 8 != 0) return false;
    iters += p.pass[i].klen / kBK;
  }
  if ((p.a_k0 | p.a_k1 | p.b_k0 | p.b_k1) % 8 != 0) return false;
  p.iters_total = iters;
  p.tiles_m = (p.M + kBM - 1) / kBM;
  p.tiles_n = (p.N + BN - 1) / BN;
  const int64_t nt = (int64_t)p.tiles_m * p.tiles_n * p.batch;
  if (nt > 0x7fffffff) return false;
  p.ntiles = (int)nt;
  p.idesc = idesc_f16(kBM, BN, ab_fmt);
  return true;
}

// The kernels' places in the context's table.
template <int BN, class Epi, int kRole>
using SingleId =
    KernelId<tc_gemm_kernel<BN, Epi, kRole>, gemm_threads<Epi>(), GemmSmem<BN, Epi>::kBytes>;
template <int BN, class Epi>
using PairId =
    KernelId<tc_gemm2_kernel<BN, Epi>, gemm_threads<Epi>(), Gemm2Smem<BN, Epi>::kBytes, 2>;
constexpr int kMaxSplit = 8;
template <int BN, class Epi>
using SplitId = KernelId<tc_gemm_split_kernel<BN, Epi>, gemm_threads<Epi>(),
                         GemmSmem<BN, Epi>::kBytes, 2, kMaxSplit>;

// ------------------------------------------------------------------------------ which form
//
// A GEMM takes one of three kernels (tc_gemm.cuh): tiles of 128 x BN on single SMs, 256 x W on CTA
// pairs, or tiles shared by a cluster that splits K. choose_gemm decides by the shape and the
// device's table alone.
enum GemmForm : int32_t { GEMM_SINGLE = 1, GEMM_PAIRS = 2, GEMM_SPLIT = 3 };
struct GemmChoice {
  int32_t form = GEMM_SINGLE;
  int32_t width = 0;  // tile columns
  int32_t ranks = 1;  // CTAs per tile (GEMM_SPLIT)
};

inline int64_t gemm_tiles(const GemmParams& p, int width) {
  return (int64_t)p.tiles_m * ((p.N + width - 1) / width) * p.batch;
}

// Most tiles that the split kernel takes at tile width BN: half of the SMs hold a cluster of two
// per tile, or fewer where the device's GPCs leave single SMs over.
template <int BN, class Epi>
inline int most_split_tiles(const KernelTable& dev) {
  return std::min(dev.num_sms / 2, dev.of<SplitId<BN, Epi>>().clusters[2]);
}

// CTAs per tile of the split kernel at tile width BN: the count, two or more, that is fastest by the
// clocks of its parts (measured on 128-row tiles at about 1.9 GHz: 384 / 512 / 768 per K iteration
// at BN = 64 / 128 / 256, where a stage's bytes bound it; 16000 to read all but one of the partials
// of 256 columns through DSMEM, 1400 to write one; 2500 per 32 columns in the epilogue; 4000 to
// start), with all clusters resident at once. 1: too many tiles, or a single K iteration. *cost:
// its clocks, which order the counts and the two widths but not the forms (see choose_gemm).
template <int BN, class Epi>
inline int split_ranks(const KernelTable& dev, int64_t ntiles, int iters, double* cost) {
  *cost = 1e30;
  if (ntiles > most_split_tiles<BN, Epi>(dev)) return 1;
  const int* resident = dev.of<SplitId<BN, Epi>>().clusters;
  int best = 1;
  for (int s = 2; s <= std::min(kMaxSplit, iters); ++s) {
    if (ntiles > resident[s]) continue;
    const int blocks = (BN / 8 + s * Epi::kWarps - 1) / (s * Epi::kWarps);
    const double c = 4000 + (double)((iters + s - 1) / s) * (256 + 2 * BN) +
                     (1400 + 16000.0 * (s - 1) / s) * BN / 256 + 2500.0 * blocks;
    if (c < *cost) {
      *cost = c;
      best = s;
    }
  }
  return best;
}

// Time of a GEMM on pairs, in clocks per K iteration beside 860 for a wave of the 1-SM kernel's
// 128 x 256 tiles: waves of its tiles, and what its start adds or saves.
template <int BN, class Epi>
inline int64_t gemm2_cost(const KernelTable& dev, const GemmParams& p) {
  if (dev.of<PairId<BN, Epi>>().status != cudaSuccess) return INT64_MAX;
  const int clusters = dev.persistent_clusters<PairId<BN, Epi>>(2);
  const int64_t pairs = (int64_t)((p.tiles_m + 1) / 2) * ((p.N + BN - 1) / BN) * p.batch;
  return (pairs + clusters - 1) / clusters * Epi::pair_wave(BN) + Epi::pair_start(BN);
}

// The width of Epi::Widths at which the 2-SM kernel is fastest, if that is faster than the 1-SM
// kernel, else 0.
// An odd number of m-tiles or a bad last wave can make the pairs slower: t = 617, d_l = 2048, P v
// 488 us on single SMs, 584 on pairs. For the latent GEMMs widths of 192 and 224 gave the call 0.4%
// at t = 617 (better last waves) and nothing elsewhere, and are not offered.
template <class Epi, int... W>
inline int pair_width(const KernelTable& dev, std::integer_sequence<int, W...>,
                      const GemmParams& p) {
  int width = 0;
  int64_t best = ((int64_t)p.ntiles + dev.num_sms - 1) / dev.num_sms * 860;
  auto consider = [&](int64_t cost, int bn) {
    if (cost < best) {
      best = cost;
      width = bn;
    }
  };
  (consider(gemm2_cost<W, Epi>(dev, p), W), ...);
  return width;
}

// p: finalized at BN. Few tiles split first: up to most_split_tiles the other two forms leave half
// of the SMs idle. Measured in calls replayed from a graph, forms forced one GEMM at a time, against
// the split count that is taken. One SM per 128 x 256 tile: the GEMMs of a layer of t = 128,
// d_l = 256, H = 2 cost the call 2 to 18 us more (of 123), also where the clocks above say about
// even (8 K iterations: 2 to 8 us); those of t = 251, d_l = 1024, H = 4 up to 65 us (of 954). Pairs:
// within 2 us of that at t = 128, up to 9 us less at t = 251. One CTA per 128 x 64 tile is within 2 us
// of the split at t = 128; at t = 300, H = 2 it gains 4 us (of 180) in each of two GEMMs whose
// 64-column tiles outnumber most_split_tiles but not the SMs, and is not offered.
template <int BN, class Epi>
inline GemmChoice choose_gemm(const KernelTable& dev, const GemmParams& p, bool can_split) {
  if (can_split) {
    double cost = 0, cost64 = 1e30;
    const int ranks = split_ranks<BN, Epi>(dev, p.ntiles, p.iters_total, &cost);
    if constexpr (Epi::kAnyTile && BN != 64) {  // narrower tiles: less to reduce per CTA
      const int ranks64 = split_ranks<64, Epi>(dev, gemm_tiles(p, 64), p.iters_total, &cost64);
      if (ranks64 > 1 && cost64 < cost) return {GEMM_SPLIT, 64, ranks64};
    }
    if (ranks > 1) return {GEMM_SPLIT, BN, ranks};
  }
  if constexpr (BN == 256 && Epi::kPairs) {
    const int width = pair_width<Epi>(dev, typename Epi::Widths(), p);
    if (width != 0) return {GEMM_PAIRS, width, 1};
  }
  return {GEMM_SINGLE, BN, 1};
}

// ------------------------------------------------------------------------------ launches

template <int BN, class Epi>
inline cudaError_t launch_split(const CUtensorMap& ta, const Operand2D& B, const CUtensorMap& tc,
                                GemmParams p, Epi epi, int ab_fmt, int ranks,
                                cudaStream_t stream) {
  CUtensorMap tb;
  if (!finalize_gemm<BN>(p, ab_fmt) || !make_tmap(&tb, B, BN)) return cudaErrorInvalidValue;
  epi.tile_cols_ = BN;
  p.ranks = ranks;
  return launch_chained(tc_gemm_split_kernel<BN, Epi>, ranks * p.ntiles, gemm_threads<Epi>(),
                        GemmSmem<BN, Epi>::kBytes, stream, ranks, ta, tb, tc, p, epi);
}

template <int BN, class Epi>
inline cudaError_t launch_pairs(const KernelTable& dev, const CUtensorMap& ta, const Operand2D& B,
                                const CUtensorMap& tc, GemmParams p, Epi epi, int ab_fmt,
                                cudaStream_t stream) {
  CUtensorMap tb;
  if (!finalize_gemm<BN>(p, ab_fmt) || !make_tmap(&tb, B, BN / 2)) return cudaErrorInvalidValue;
  epi.tile_cols_ = BN;
  const int64_t pairs = (int64_t)((p.tiles_m + 1) / 2) * p.tiles_n * p.batch;
  const int clusters =
      (int)std::min<int64_t>(pairs, dev.persistent_clusters<PairId<BN, Epi>>(2));
  return launch_chained(tc_gemm2_kernel<BN, Epi>, 2 * clusters, gemm_threads<Epi>(),
                        Gemm2Smem<BN, Epi>::kBytes, stream, 2, ta, tb, tc, p, epi);
}
template <class Epi, int... W>
inline cudaError_t launch_pairs_at(const KernelTable& dev, int width,
                                   std::integer_sequence<int, W...>, const CUtensorMap& ta,
                                   const Operand2D& B, const CUtensorMap& tc, const GemmParams& p,
                                   const Epi& epi, int ab_fmt, cudaStream_t stream) {
  cudaError_t e = cudaErrorInvalidValue;
  ((width == W ? (void)(e = launch_pairs<W, Epi>(dev, ta, B, tc, p, epi, ab_fmt, stream))
               : (void)0),
   ...);
  return e;
}

// taken: the form that is launched.
template <int BN, int kRole, class Epi>
inline cudaError_t launch_gemm(const KernelTable& dev, const Operand2D& A, const Operand2D& B,
                               GemmParams p, Epi epi, int ab_fmt, cudaStream_t stream,
                               const StoreView3D* out_view, GemmChoice* taken) {
  if (!finalize_gemm<BN>(p, ab_fmt)) return cudaErrorInvalidValue;
  CUtensorMap ta, tb, tc;
  if (!make_tmap(&ta, A, kBM)) return cudaErrorInvalidValue;
  std::memset(&tc, 0, sizeof(tc));
  if (out_view != nullptr && !make_store_tmap(&tc, *out_view)) return cudaErrorInvalidValue;
  const GemmChoice c = choose_gemm<BN, Epi>(dev, p, epi.can_split());
  *taken = c;
  if (c.form == GEMM_SPLIT) {
    if constexpr (Epi::kAnyTile && BN != 64)
      if (c.width == 64) return launch_split<64, Epi>(ta, B, tc, p, epi, ab_fmt, c.ranks, stream);
    return launch_split<BN, Epi>(ta, B, tc, p, epi, ab_fmt, c.ranks, stream);
  }
  if constexpr (BN == 256 && Epi::kPairs)
    if (c.form == GEMM_PAIRS)
      return launch_pairs_at<Epi>(dev, c.width, typename Epi::Widths(), ta, B, tc, p, epi, ab_fmt,
                                  stream);
  if (!make_tmap(&tb, B, BN)) return cudaErrorInvalidValue;
  epi.tile_cols_ = BN;
  const cudaError_t ready = dev.of<SingleId<BN, Epi, kRole>>().status;
  if (ready != cudaSuccess) return ready;
  const int grid = p.ntiles < dev.num_sms ? p.ntiles : dev.num_sms;
  return launch_chained(tc_gemm_kernel<BN, Epi, kRole>, grid, gemm_threads<Epi>(),
                        GemmSmem<BN, Epi>::kBytes, stream, 1, ta, tb, tc, p, epi);
}

}  // namespace still
