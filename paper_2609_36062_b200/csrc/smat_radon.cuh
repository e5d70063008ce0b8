// Shared by the two tensor-core tabulation kernels (resident and generated Radon matrix): the index spaces of a stage,
// the rows its tables keep them in, and the tensor maps over those rows.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_tc.cuh"

constexpr int ROW_INVALID = -1;
constexpr int ROW_VERT = 1 << 30;                 // flag: row of the extra ("vertical") class

// One index space of the transform: idx = lo + q*hi, hi in [0, q]; hi == q is the extra class (a = ∞ on the
// type side).  Rows are counted inside one head.
struct RadonSide {
  int32_t count;                   // q*q, or q*q + q with the extra class
  int32_t s_lo, s_hi, s_img;       // regular rows: img*s_img + lo*s_lo + hi*s_hi
  int32_t v0, sv_lo, sv_img;       // extra class : v0 + img*sv_img + lo*sv_lo
  int32_t vert_from;               // images >= vert_from carry the extra class
  int64_t rows_per_head;
};

__device__ __forceinline__ int side_row(const RadonSide& s, int idx, int q) {
  if (idx >= s.count) return ROW_INVALID;
  const int lo = idx % q, hi = idx / q;
  return hi < q ? lo * s.s_lo + hi * s.s_hi : (ROW_VERT | lo * s.sv_lo);
}

namespace tc {
__device__ __forceinline__ void tma_load_5d(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            int c4, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}
}  // namespace tc

typedef CUresult (*RadonEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
inline RadonEncodeFn radon_encode_fn() {
  static const RadonEncodeFn fn = [] {   // initialised once, thread-safe
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      return reinterpret_cast<RadonEncodeFn>(p);
    return static_cast<RadonEncodeFn>(nullptr);
  }();
  return fn;
}

// bf16 map of any rank, fastest dimension first (contiguous), strides of the others in elements; 128-byte swizzle (a box
// is 64 elements wide); out-of-bounds reads give zeros.
inline bool radon_map_elems(CUtensorMap* map, const void* base, int rank, const int64_t* sizes, const int64_t* strides,
                            const int* box) {
  RadonEncodeFn fn = radon_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[5], bytes[4];
  cuuint32_t bx[5], estr[5];
  for (int i = 0; i < rank; ++i) {
    dims[i] = (cuuint64_t)sizes[i];
    bx[i] = (cuuint32_t)box[i];
    estr[i] = 1;
    if (i) bytes[i - 1] = (cuuint64_t)strides[i - 1] * 2;
  }
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, bytes, bx, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 rows of rp entries.  Dimensions (fastest first): entry, then `rank - 1` row indices with the given sizes and
// strides in rows; box = 64 entries x box[] rows.
inline bool radon_map(CUtensorMap* map, const void* base, int64_t rp, int rank, const int64_t* sizes,
                      const int64_t* row_strides, const int* box) {
  int64_t s[5] = {rp}, st[4];
  int b[5] = {64};
  for (int i = 1; i < rank; ++i) { s[i] = sizes[i - 1]; st[i - 1] = row_strides[i - 1] * rp; b[i] = box[i - 1]; }
  return radon_map_elems(map, base, rank, s, st, b);
}

inline RadonSide side(int count, int s_lo, int s_hi, int s_img, int64_t rows_per_head, int v0 = 0, int sv_lo = 0,
                      int sv_img = 0, int vert_from = 1 << 29) {
  RadonSide s;
  s.count = count; s.s_lo = s_lo; s.s_hi = s_hi; s.s_img = s_img; s.v0 = v0; s.sv_lo = sv_lo; s.sv_img = sv_img;
  s.vert_from = vert_from; s.rows_per_head = rows_per_head;
  return s;
}

// One stage as the host states it; src / dst are whole tables [bh][rows_per_head][rp], or the private exchange buffer.
struct StageSpec {
  RadonSide in, out;
  int images;
  const void* src;
  void* dst;
  bool src_private, dst_private;
};

inline StageSpec stage(const RadonSide& in, const RadonSide& out, int images, const void* src, void* dst,
                       bool src_private = false, bool dst_private = false) {
  StageSpec s;
  s.in = in; s.out = out; s.images = images; s.src = src; s.dst = dst; s.src_private = src_private; s.dst_private = dst_private;
  return s;
}

// One stage with the Radon matrix generated beside the image stream (smat_radon_wide.cu); tables only, no exchange buffer.
bool radon_wide_fits(int q, const StageSpec& sp);   // whether a stage's slots, tiles and tables fit (host only)
bool radon_wide_layout_ok(int q, const StageSpec& sp);
cudaError_t launch_radon_wide(int q, int transpose, const StageSpec& sp, int64_t rp, int bh, int* status, cudaStream_t st);

// One stage with the whole matrix in tensor memory as a sparse operand (smat_radon_sparse.cu).
bool radon_sparse_fits(int q);
cudaError_t launch_radon_sparse(int q, int transpose, const StageSpec& sp, int64_t rp, int bh, int* status, cudaStream_t st);
