// Tabulation stages (see smat_radon_tc.cu for the transform) for q = 17, whose 306 or 289 outputs are three MMA tiles: the
// whole matrix R stays in tensor memory as a sparse A operand, so that ONE CTA covers an image.
//
// A row of R has one nonzero per input line, so at most two in every four neighbouring inputs (lines have 17): the
// form tcgen05.mma.sp takes, with half the columns of tensor memory and twice the inputs per cycle.  Only the q rows of the
// extra class on the type side (whole lines) are not; they lie in the last tile, which is kept dense.  Columns:
//   forward    : two sparse tiles 2 x (72 + 24), one dense 144, two accumulators of 64 columns 128    -> 464
//                (input 288, the last, would cost another instruction step in every tile and the columns for it; the
//                epilogue adds it to the 18 rows it meets)
//   transposed : three sparse tiles 3 x (80 + 24), three accumulators 192                             -> 504
// An item is one image restricted to 64 state entries: one TMA box (and one for the extra class of a transposed image) into
// a ring slot, (9 + 9 + 18) instructions of 32 cycles, three tiles read back, rounded and stored.
// Bound by memory: 64 heads of 8192 tokens (1.25 GB) 0.204 ms, transposed 0.206, 0.190 at the HBM rate, where three CTAs
// that shared every image (dense matrix, 102 outputs each) and the generated matrix took 0.257 and 0.270; d = 4, 2 heads of
// 64 K tokens (both stages, 1.35 GB) 0.24 for 0.30.
//   warps 0-15 : epilogue; lane quarter w % 4, column quarter w / 4 (16 columns) of every accumulator; one 32-byte sector
//                per row and tile
//   warp 16    : TMA producer;   warp 17 : MMA issuer (whole warps walk the loops, one lane issues)
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_radon.cuh"
#include "smat_tc.cuh"

namespace {

using namespace tc;

constexpr int ROWS = 128;                 // output indices per tile
constexpr int NE = 64;                    // state entries per item
constexpr int MAX_TILES = 3, MAX_RING = 8, MAX_ACC = 4;
constexpr int EPI = 16, PROD_WARP = EPI, MMA_WARP = EPI + 1;
constexpr int THREADS = 32 * (EPI + 2);

// How the matrix of a direction lies in tensor memory and its images in shared memory, known when it is compiled.
struct SparseShape {
  int q, transpose;
  int count_out, tiles, dense;      // outputs, tiles of them, first dense one (none: tiles)
  int reg_rows;                     // q^2
  int extra_row;                    // slot row of the first extra-class input (none: 0), on an 8-row boundary
  int rows;                         // slot rows up to the last input, the gap before the extra class among them
  int steps, dense_steps;           // sparse steps (32 inputs); a dense tile takes the same rows in steps of 16
  int tail;                         // input that the steps leave out and the epilogue adds (none: -1)
  int meta_cols;                    // columns of positions per sparse tile
  int acc;                          // accumulators of NE columns
  int slot_rows, slot_bytes, ring;
  // First column of a tile's values (a dense tile is the last one); a sparse tile's positions follow them.
  __host__ __device__ constexpr int col(int t) const { return acc * NE + t * (steps * 8 + meta_cols); }
};
__host__ __device__ constexpr SparseShape sparse_shape(int q, int transpose) {
  SparseShape s{};
  const int qq = q * q;
  s.q = q; s.transpose = transpose;
  s.count_out = transpose ? qq : qq + q;
  s.tiles = (s.count_out + ROWS - 1) / ROWS;
  s.dense = transpose ? s.tiles : s.tiles - 1;
  s.reg_rows = qq;
  s.extra_row = transpose ? (qq + 7) / 8 * 8 : 0;
  s.rows = transpose ? s.extra_row + q : qq;
  s.tail = s.rows % 32 == 1 ? s.rows - 1 : -1;   // one input past a whole number of steps costs as much as 31
  const int in_steps = s.tail >= 0 ? s.rows - 1 : s.rows;
  s.steps = (in_steps + 31) / 32;
  s.dense_steps = (in_steps + 15) / 16;
  s.meta_cols = ((s.steps + 1) / 2 * 4 + 7) / 8 * 8;   // a pair of steps takes two of every four columns
  const int cols = s.dense * (s.steps * 8 + s.meta_cols) + (s.tiles - s.dense) * s.dense_steps * 8;
  s.acc = (512 - cols) / NE < MAX_ACC ? (512 - cols) / NE : MAX_ACC;
  s.slot_rows = ((s.steps * 32 > s.rows ? s.steps * 32 : s.rows) + 7) / 8 * 8;
  s.slot_bytes = s.slot_rows * 128;
  const int ring = (227 * 1024 - 2048) / s.slot_bytes;
  s.ring = ring < MAX_RING ? ring : MAX_RING;
  return s;
}
constexpr int sparse_smem(const SparseShape& s) { return 1024 + s.ring * s.slot_bytes + (2 * MAX_RING + 2 * MAX_ACC) * 8 + 16; }
// Boxes and instruction steps stay inside a slot, the extra class starts on a swizzle period behind the regular rows, the
// barriers end inside the allocation; values lie on columns that are multiples of eight, the positions of a pair of steps on
// multiples of four, all behind the accumulators; the rows of the extra class (whole lines) lie in the dense tile.
constexpr bool sparse_layout_ok(const SparseShape& s) {
  for (int t = 0; t < s.tiles; ++t)
    if (s.col(t) % 8 != 0 || (t < s.dense && (s.col(t) + 8 * s.steps) % 4 != 0)) return false;
  const int in_steps = s.tail >= 0 ? s.rows - 1 : s.rows;
  return s.slot_bytes % 1024 == 0 && s.rows <= s.slot_rows && s.steps * 32 <= s.slot_rows && s.dense_steps * 16 <= s.slot_rows &&
         s.steps * 32 >= in_steps && s.dense_steps * 16 >= in_steps &&
         (!s.transpose || (s.extra_row >= s.reg_rows && s.extra_row % 8 == 0)) &&
         s.q >= 16 && s.q <= 64 &&   // three lines at most in 32 inputs (RadonRow::bits); the rows of a box
         s.tiles <= MAX_TILES && s.tiles - s.dense <= 1 && (s.transpose || s.dense * ROWS <= s.reg_rows) && s.acc >= 2 &&
         s.ring >= 3 && s.meta_cols % 8 == 0 && s.meta_cols >= (s.steps + 1) / 2 * 4 - 2 &&
         s.col(s.dense) + (s.tiles - s.dense) * s.dense_steps * 8 <= 512 &&
         1023 + s.ring * s.slot_bytes + (2 * MAX_RING + 2 * MAX_ACC) * 8 + 8 <= sparse_smem(s) && sparse_smem(s) <= 227 * 1024;
}
static_assert(sparse_layout_ok(sparse_shape(17, 0)) && sparse_layout_ok(sparse_shape(17, 1)), "maps of shared and tensor memory");

struct SparseParams {
  int32_t slabs_per_head, images;
  uint32_t slabs, items;            // heads * slabs_per_head; slabs * images
  int32_t src_heads;                // heads of the source table
  int32_t in_vert_from, in_sv_img;
  RadonSide out;
  int64_t rp;
  __nv_bfloat16* dst;
  int* status;
};

// One row of R.
template <int Q, int TRANSPOSE>
struct RadonRow {
  int x, y, step;                   // output x + q y; the nonzero of input line L is (x + step L) mod q
  bool live, line;                  // line: an output of the extra class, the whole line x
  __device__ __forceinline__ explicit RadonRow(int out) {
    y = out / Q; x = out - y * Q;
    live = out < sparse_shape(Q, TRANSPOSE).count_out;
    line = !TRANSPOSE && y >= Q;
    step = TRANSPOSE ? y : (y ? Q - y : 0);   // (x - y L) forward, (x + y L) transposed
  }
  // Its entries at the slot rows [lo, lo + 32): bit k is slot row lo + k.
  __device__ __forceinline__ uint32_t bits(int lo) const {
    if (!live) return 0u;
    if (line) {
      const int a = max(x * Q - lo, 0), b = min(x * Q + Q - lo, 32);
      return b > a ? (0xffffffffu >> (32 - (b - a))) << a : 0u;
    }
    const int first = lo / Q;
    uint32_t w = 0u;
    int at = first * Q - lo, pos = (x + step * first) % Q;
#pragma unroll
    for (int i = 0; i < 3; ++i) {   // 32 inputs touch at most three lines of 17
      const int k = at + pos;
      if (first + i < Q && k >= 0 && k < 32) w |= 1u << k;
      at += Q;
      pos += step;
      if (pos >= Q) pos -= Q;
    }
    if (TRANSPOSE) {                // the extra class meets it at y
      const int k = sparse_shape(Q, TRANSPOSE).extra_row + y - lo;
      if (k >= 0 && k < 32) w |= 1u << k;
    }
    return w;
  }
};

// 32 inputs with at most two nonzeros in every four: the positions, 4 bits to a group, and the two kept values of each
// group, as bit 4 g of v0 and of v1.
__device__ __forceinline__ uint32_t positions(uint32_t w, uint32_t* v0, uint32_t* v1) {
  constexpr uint32_t M = 0x11111111u;
  const uint32_t b1 = w >> 1, b2 = w >> 2, b3 = w >> 3;   // (bit 0 of every nibble counts)
  const uint32_t lo = w | b1, up = b2 | b3;
  // first kept input: 0 or 1 if the lower pair has a nonzero (or the upper has none), else 2; second: 1 if the upper pair
  // has none, else 3, or 2 where both pairs have one and the upper's is input 2
  const uint32_t f0 = ~w & b1 & up, f1 = ~lo & up, s0 = ~up | b3 | ~lo;
  *v0 = (w | f0 | (f1 & b2)) & M;
  *v1 = ((up & (b3 | ~s0)) | (~up & b1)) & M;
  return (f0 & M) | ((f1 & M) << 1) | ((s0 & M) << 2) | ((up & M) << 3);
}

// bf16 pair: 1.0 where the bits are set
__device__ __forceinline__ uint32_t ones(uint32_t lo, uint32_t hi) { return (lo & 1u) * 0x3f80u + (hi & 1u) * 0x3f800000u; }

template <int Q, int TRANSPOSE>
__global__ void __launch_bounds__(THREADS, 1) radon_sparse_kernel(const __grid_constant__ CUtensorMap tm_reg,
                                                                  const __grid_constant__ CUtensorMap tm_vert,
                                                                  const __grid_constant__ SparseParams prm) {
  constexpr SparseShape sh = sparse_shape(Q, TRANSPOSE);
  constexpr int ring = sh.ring, nt = sh.tiles;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + ring * sh.slot_bytes);
  uint64_t* full = bars;                         // [MAX_RING] image landed
  uint64_t* empty = full + MAX_RING;             // [MAX_RING] ... and consumed (tail: one arrival per epilogue warp as well)
  uint64_t* d_full = empty + MAX_RING;           // [MAX_ACC] tile complete
  uint64_t* d_empty = d_full + MAX_ACC;          // [MAX_ACC] ... and read out (one arrival per warp)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(d_empty + MAX_ACC);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{cta_abort, prm.status};
  if (threadIdx.x == 0) {
    *cta_abort = 0;
    for (int s = 0; s < ring; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, sh.tail >= 0 ? 1 + EPI : 1); }
    for (int u = 0; u < sh.acc; ++u) { mbar_init(d_full + u, 1); mbar_init(d_empty + u, EPI); }
    fence_barrier_init();
    prefetch_tmap(&tm_reg);
    prefetch_tmap(&tm_vert);
  }
  if (warp == MMA_WARP) tmem_alloc(tmem_slot, 512);
  {   // slot rows that no box writes meet zeros of R, but must not hold NaN patterns
    constexpr int gap = TRANSPOSE ? sh.extra_row - sh.reg_rows : 0, idle = gap + sh.slot_rows - sh.rows;   // rows per slot
    for (int c = threadIdx.x; c < ring * idle * 8; c += THREADS) {
      const int slot = c / (idle * 8), r = (c >> 3) - slot * idle, row = r < gap ? sh.reg_rows + r : sh.rows + r - gap;
      reinterpret_cast<uint4*>(smem + slot * sh.slot_bytes + row * 128)[c & 7] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  pdl_trigger();   // (after the allocation: a kernel that starts early must not take the tensor memory first)
  const uint32_t tmem_base = *tmem_slot;
  const int qd = warp & 3, part = warp >> 2;
  const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
  if (warp < EPI) {   // R: a warp takes every fourth step of its 32 rows
    for (int t = 0; t < nt; ++t) {
      const RadonRow<Q, TRANSPOSE> row(t * ROWS + qd * 32 + lane);
      const uint32_t col = tmem_base + lane_base + sh.col(t);
      if (t < sh.dense) {
        for (int s = part; s < sh.steps; s += EPI / 4) {
          uint32_t a0, a1, v[8];
          const uint32_t own = positions(row.bits(32 * s), &a0, &a1);
#pragma unroll
          for (int g = 0; g < 8; ++g) v[g] = ones(a0 >> (4 * g), a1 >> (4 * g));
          // the other row of the lane pair takes one half of the positions (see mma_sparse_bf16_ta)
          const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 8);
          tmem_st8(col + 8 * s, v);
          tmem_st1(col + 8 * sh.steps + 2 * s - (s & 1), (lane & 8) ? __byte_perm(other, own, 0x7632) : __byte_perm(own, other, 0x5410));
        }
      } else {
        for (int s = part; s < sh.dense_steps; s += EPI / 4) {
          uint32_t v[8];
          const uint32_t w = row.bits(16 * s);
#pragma unroll
          for (int g = 0; g < 8; ++g) v[g] = ones(w >> (2 * g), w >> (2 * g + 1));
          tmem_st8(col + 8 * s, v);
        }
      }
    }
    tmem_st_wait();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  pdl_wait();

  if (warp == PROD_WARP) {
    const bool leader = elect_one();
    uint32_t slot = 0, par = 1;                                  // par: parity that a fresh `empty` barrier passes
    bool ok = true;
    constexpr uint32_t bytes = (uint32_t)((sh.reg_rows + (TRANSPOSE ? Q : 0)) * 2 * NE);
    for (uint32_t item = blockIdx.x; item < prm.items && ok; item += gridDim.x) {
      const uint32_t img = item / prm.slabs, slab = item - img * prm.slabs, head = slab / (uint32_t)prm.slabs_per_head;
      const int e0 = (int)(slab - head * prm.slabs_per_head) * NE;
      ok = __all_sync(0xffffffffu, mbar_wait(empty + slot, par, wc));
      if (!ok) break;
      if (leader) {
        uint8_t* dst = smem + slot * sh.slot_bytes;
        mbar_expect_tx(full + slot, bytes);
        tma_load_5d(dst, &tm_reg, e0, 0, 0, (int)img, (int)head, full + slot);
        if (TRANSPOSE)   // an image without the extra class reads past the last head: zeros
          tma_load_4d(dst + sh.extra_row * 128, &tm_vert, e0, 0, (int)img * prm.in_sv_img,
                      (int)img >= prm.in_vert_from ? (int)head : prm.src_heads, full + slot);
      }
      if (++slot == (uint32_t)ring) { slot = 0; par ^= 1; }
    }
    if (leader) ring_landed(full, (uint32_t)ring, slot, par, wc);
  } else if (warp == MMA_WARP) {
    // How fast the instructions follow one another, by unrolling.  A sparse one of 64 columns reads shared memory at its full
    // rate; in one burst per item they hold up the boxes that arrive.  64 heads of 8192 tokens, forward / transposed:
    // fully unrolled 0.234 / 0.230 ms, by two 0.204 / 0.230, not at all 0.232 (36 instructions of about 100 cycles are an
    // item's time) / 0.206.  d = 4, 4 heads of 64 K tokens, both stages: 0.51 / 0.51, 0.47 / 0.51, 0.49 / 0.48.
    constexpr int PACE = TRANSPOSE ? 1 : 2;
    constexpr uint32_t id_dense = make_idesc(ROWS, NE, 0, 1);    // R from tensor memory, image rows MN-major
    constexpr uint32_t id_even = make_idesc_sparse(ROWS, NE, 0, 1, 0), id_odd = make_idesc_sparse(ROWS, NE, 0, 1, 1);
    const uint64_t dB0 = make_desc(smem_u32(smem), 0, 1024);
    const bool leader = elect_one();
    uint32_t slot = 0, par = 0, u = 0, up = 1;                   // up: parity that a fresh d_empty barrier passes
    bool ok = true;
    for (uint32_t item = blockIdx.x; item < prm.items && ok; item += gridDim.x) {
      ok = __all_sync(0xffffffffu, mbar_wait(full + slot, par, wc));
      const uint64_t dB = dB0 + (uint64_t)(slot * (uint32_t)(sh.slot_bytes >> 4));
#pragma unroll 1
      for (int t = 0; t < nt; ++t) {
        ok = ok && __all_sync(0xffffffffu, mbar_wait(d_empty + u, up, wc));   // an earlier tile's sums have been read out
        if (!ok) break;
        fence_after_sync();
        if (leader) {
          const uint32_t d = tmem_base + u * NE, a = tmem_base + sh.col(t);
          if (t < sh.dense) {
#pragma unroll (PACE)
            for (int s = 0; s < sh.steps; ++s)
              mma_sparse_bf16_ta(d, a + 8 * s, dB + 256 * s, a + 8 * sh.steps + 4 * (s >> 1), (s & 1) ? id_odd : id_even, s != 0);
          } else {
#pragma unroll (PACE)
            for (int s = 0; s < sh.dense_steps; ++s) mma_bf16_ta(d, a + 8 * s, dB + 128 * s, id_dense, s != 0);
          }
          mma_commit(d_full + u);
          if (t + 1 == nt) mma_commit(empty + slot);
        }
        if (++u == (uint32_t)sh.acc) { u = 0; up ^= 1; }
      }
      if (++slot == (uint32_t)ring) { slot = 0; par ^= 1; }
    }
  } else {
    int rows[nt];
    uint32_t with_tail = 0;
#pragma unroll
    for (int t = 0; t < nt; ++t) {
      const int out = t * ROWS + qd * 32 + lane;
      rows[t] = side_row(prm.out, out, Q);
      if (sh.tail >= 0 && (RadonRow<Q, TRANSPOSE>(out).bits(sh.tail) & 1u)) with_tail |= 1u << t;
    }
    // the tail's 16 columns of this warp: two 16-byte chunks of its swizzled row
    constexpr int tail = sh.tail >= 0 ? sh.tail : 0;
    const uint8_t* tail_row = smem + tail * 128;
    const int c0 = ((2 * part) ^ (tail & 7)) << 4, c1 = ((2 * part + 1) ^ (tail & 7)) << 4;
    uint32_t slot = 0, spar = 0, u = 0, par = 0;
    bool ok = true;
    for (uint32_t item = blockIdx.x; item < prm.items && ok; item += gridDim.x) {
      const uint32_t img = item / prm.slabs, slab = item - img * prm.slabs, head = slab / (uint32_t)prm.slabs_per_head;
      const int e0 = (int)(slab - head * prm.slabs_per_head) * NE;
      __nv_bfloat16* base = prm.dst + (int64_t)head * prm.out.rows_per_head * prm.rp + e0 + part * 16;
      const bool vert = (int)img >= prm.out.vert_from;
      uint4 y[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
      if (sh.tail >= 0) {
        ok = mbar_wait_warp(full + slot, spar, wc);
        if (!ok) break;
        y[0] = *reinterpret_cast<const uint4*>(tail_row + slot * sh.slot_bytes + c0);
        y[1] = *reinterpret_cast<const uint4*>(tail_row + slot * sh.slot_bytes + c1);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + slot);
        if (++slot == (uint32_t)ring) { slot = 0; spar ^= 1; }
      }
#pragma unroll
      for (int t = 0; t < nt; ++t) {
        ok = mbar_wait_warp(d_full + u, par, wc);
        if (!ok) break;
        fence_after_sync();
        uint32_t v[16];
        tmem_ld16(tmem_base + lane_base + u * NE + part * 16, v);
        tmem_ld_wait();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(d_empty + u);
        if (++u == (uint32_t)sh.acc) { u = 0; par ^= 1; }
        const int tv = rows[t];
        if (tv != ROW_INVALID && (!(tv & ROW_VERT) || vert)) {
          const int row = (tv & ROW_VERT) ? prm.out.v0 + (int)img * prm.out.sv_img + (tv & ~ROW_VERT) : (int)img * prm.out.s_img + tv;
          if (sh.tail >= 0 && (with_tail & (1u << t))) {
            const uint32_t yy[8] = {y[0].x, y[0].y, y[0].z, y[0].w, y[1].x, y[1].y, y[1].z, y[1].w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              v[2 * i] = __float_as_uint(__uint_as_float(v[2 * i]) + __uint_as_float(yy[i] << 16));
              v[2 * i + 1] = __float_as_uint(__uint_as_float(v[2 * i + 1]) + __uint_as_float(yy[i] & 0xffff0000u));
            }
          }
          uint32_t o[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i] = pack_bf16(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
          st_global_v8(base + (int64_t)row * prm.rp, o[0], o[1], o[2], o[3], o[4], o[5], o[6], o[7]);
        }
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == MMA_WARP) {
    fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

template <int Q, int TRANSPOSE>
cudaError_t launch(const CUtensorMap& tm_reg, const CUtensorMap& tm_vert, const SparseParams& prm, cudaStream_t st) {
  constexpr int smem = sparse_smem(sparse_shape(Q, TRANSPOSE));
  const auto kernel = radon_sparse_kernel<Q, TRANSPOSE>;
  const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (err != cudaSuccess) return err;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = prm.items < (uint32_t)sms ? prm.items : (unsigned)sms;
  return smat_launch_pdl(kernel, dim3(grid), THREADS, (size_t)smem, st, tm_reg, tm_vert, prm);
}

}  // namespace

bool radon_sparse_fits(int q) { return q == 17; }

cudaError_t launch_radon_sparse(int q, int transpose, const StageSpec& sp, int64_t rp, int bh, int* status, cudaStream_t st) {
  if (!radon_sparse_fits(q) || rp % NE) return cudaErrorInvalidValue;
  const RadonSide& in = sp.in;
  if (sp.out.count != q * q + (transpose ? 0 : q) || in.count != q * q + (transpose ? q : 0)) return cudaErrorInvalidValue;
  SparseParams prm;
  prm.images = sp.images;
  prm.src_heads = bh;
  prm.in_vert_from = in.vert_from;
  prm.in_sv_img = in.sv_img != 0 ? 1 : 0;
  prm.out = sp.out; prm.rp = rp;
  prm.dst = static_cast<__nv_bfloat16*>(sp.dst);
  prm.status = status;
  prm.slabs_per_head = (int)(rp / NE);
  const int64_t items = (int64_t)bh * prm.slabs_per_head * prm.images;
  if (items >= (1LL << 31)) return cudaErrorInvalidValue;
  prm.slabs = (uint32_t)bh * (uint32_t)prm.slabs_per_head;
  prm.items = (uint32_t)items;
  CUtensorMap tm_reg, tm_vert;
  {   // (entry, lo, hi, image, head); a size-one dimension keeps its stride valid
    const int64_t sizes[4] = {q, q, sp.images, bh};
    const int64_t strides[4] = {in.s_lo, in.s_hi, sp.images > 1 ? in.s_img : in.rows_per_head, in.rows_per_head};
    const int box[4] = {q, q, 1, 1};
    if (!radon_map(&tm_reg, sp.src, rp, 5, sizes, strides, box)) return cudaErrorInvalidValue;
  }
  tm_vert = tm_reg;
  if (transpose) {
    const bool per_image = in.sv_img != 0;
    const int64_t sizes[3] = {q, per_image ? sp.images : 1, bh};
    const int64_t strides[3] = {in.sv_lo, per_image ? in.sv_img : in.rows_per_head, in.rows_per_head};
    const int box[3] = {q, 1, 1};
    if (!radon_map(&tm_vert, static_cast<const __nv_bfloat16*>(sp.src) + (int64_t)in.v0 * rp, rp, 4, sizes, strides, box))
      return cudaErrorInvalidValue;
  }
  return transpose ? launch<17, 1>(tm_reg, tm_vert, prm, st) : launch<17, 0>(tm_reg, tm_vert, prm, st);
}
