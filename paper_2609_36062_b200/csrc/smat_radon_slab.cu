// Tabulation U = C F for d = 4 with bf16 tables, both stages of a slab in one CTA and the table between them in shared
// memory (see smat_radon_tc.cu for the two stages and the Radon matrix R).
//
// A slab is 64 state entries of every point of one head.  Stage 1 turns image x2 (q² rows of F) into q² + q rows, which
// belong to q + 1 images of stage 2: W[a3] takes rows (u, x2), G takes rows (x2, x3).  At 64 entries a row is 128 bytes,
// one row of the swizzled MN-major operand, so the stage-1 epilogue writes its rounded sums straight to where the stage-2
// MMAs read them: q + 1 slots of 128 rows (192 KB at q = 11), never written to memory.  The CTA's own U tiles leave from
// the same slots, each dead once the MMAs of its image have read it.
//   warps 0-15   : epilogue, four groups of four that take the items in turn; lane = output index, all 64 entries
//   warp 16      : producer of the F images
//   warp 17, 18  : MMA issuers of stage 1 and stage 2, each with its own ring of accumulators
//   warp 19      : sends the U tiles off by TMA
//   warps 20-23  : the output indices past 128 (q² + q = 132; all of the extra class, sums of one line of the image)
// What it is about is bytes in flight: the slots leave room for a ring of two F images only, and a load takes 2,000 to
// 4,000 cycles.  So most images of the next slab land in stage-2 slots, each as soon as the U tile in it has been read by
// the copy engine, while stage 2 is still at work on the later ones; they are multiplied into accumulators, the first few
// held rounded in the epilogue's registers, and only when all of them have been read may the epilogue write W again.
//
// q = 11, 32 heads of 16,384 entries: 0.515 ms; the tables' bytes take 0.44.  Before, with slabs of 128 entries and W
// through the L2 cache, both ways as TMA tiles: 0.812 (twice the copy engine's work).  With the ring of two alone 0.915;
// images in stage-2 slots 0.774; the roles' loops kept rolled 0.706; four groups 0.612; all lanes of a warp at a barrier
// (one lane polling and a shuffle cost about a hundred cycles more at every wait) 0.515.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_radon.cuh"
#include "smat_tc.cuh"

namespace {

using namespace tc;

constexpr int Q = 11, QQ = Q * Q, NOUT = QQ + Q;
constexpr int NE = 64;                                  // entries per slab
constexpr int SLOT = 128 * 2 * NE;                      // an image (q² rows, padded to 128) or an output tile
constexpr int TILE_BYTES = QQ * 2 * NE;                 // what a box moves
constexpr int NF = 2, NW = Q + 1;                       // slots for F images; for the images of stage 2
constexpr int ACC1 = 5, ACC2 = 2;                       // accumulators of 64 columns
constexpr int LAG = 1;                                  // tile stores in flight
constexpr int PRE = 7;                                  // images of a slab that land in stage-2 slots
constexpr int EPI = 16, GROUP = 4, GROUPS = 4;          // epilogue warps; a group of four reads an accumulator
constexpr int PROD_WARP = EPI, MMA1_WARP = EPI + 1, MMA2_WARP = EPI + 2, STORE_WARP = EPI + 3, ALU_WARP = EPI + 4;
constexpr int STEPS = 8;                                // K-steps of 16 rows per image
constexpr int R_COLS = 64;                              // columns of R: 128 operand rows, two bf16 a column
constexpr int ALU_ROWS = NOUT - 128;                    // output indices summed on the ALUs, a warp for each
constexpr int THREADS = 32 * (ALU_WARP + ALU_ROWS);
constexpr int OFF_F = 0, OFF_W = NF * SLOT, OFF_MINI = OFF_W + NW * SLOT, OFF_BARS = OFF_MINI + ((Q * 128 + 63) & ~63);
constexpr int NBARS = 2 * NF + 2 * PRE + 2 * ACC1 + GROUPS + ACC2 + 3 + NW;
constexpr int SMEM = 1024 + OFF_BARS + NBARS * 8 + 16;
static_assert(SMEM <= 227 * 1024, "the slots must fit shared memory");
static_assert(R_COLS + 64 * (ACC1 + ACC2) <= 512, "R and the accumulators must fit tensor memory");
// Stage 1 takes the images in this order: those in the ring's slots first (they land while stage 1 of the slab before is at
// work), then those in stage-2 slots, then the rest through the ring.
__device__ constexpr int image_at(int t) { return t < NF ? PRE + t : (t < NF + PRE ? t - NF : t); }
__device__ __forceinline__ bool in_ring(int t) { return t < NF || t >= NF + PRE; }
constexpr int EARLY = NF + PRE;                         // items multiplied before W may be written
static_assert(EARLY <= ACC1 + GROUPS, "they wait in accumulators and, rounded, in the groups' registers");
static_assert(PRE + LAG <= NW, "the store loop tells of every such slot");
static_assert(PRE + NF <= Q, "the ring takes at least as many images as it has slots");
static_assert(NW % GROUPS == 0, "stage 2: a group has the same images of every slab");
static_assert(QQ <= 128 && ALU_ROWS > 0 && ALU_ROWS <= 8, "the leftover indices");

struct SlabParams {
  uint32_t slabs;            // heads * slabs_per_head
  uint32_t slabs_per_head;
  int* status;
};

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* smem_src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(map), "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}

// A ring position and the parity its "full" barrier shows; the "empty" barrier is waited for with the other one, which
// a fresh barrier passes.
template <int N>
struct Ring {
  uint32_t at = 0, par = 0;
  __device__ __forceinline__ void next() {
    if (++at == N) { at = 0; par ^= 1; }
  }
};

// Byte offset of a 16-byte chunk of a row in a swizzled slot.
__device__ __forceinline__ int chunk_at(int row, int chunk) { return row * 128 + ((chunk ^ (row & 7)) << 4); }

// Byte offset of entries 2 pair and 2 pair + 1 of a row; and the sum over q rows at given offsets, rounded.
__device__ __forceinline__ int pair_at(int row, int pair) { return chunk_at(row, pair >> 2) + (pair & 3) * 4; }
__device__ __forceinline__ uint32_t rows_sum(const uint8_t* slot, const int (&at)[Q]) {
  uint32_t w[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) w[i] = *reinterpret_cast<const uint32_t*>(slot + at[i]);
  float a[2] = {0.f, 0.f}, b[2] = {0.f, 0.f};
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    a[i & 1] += __uint_as_float(w[i] << 16);
    b[i & 1] += __uint_as_float(w[i] & 0xffff0000u);
  }
  return pack_bf16(a[0] + a[1], b[0] + b[1]);
}

__global__ void __launch_bounds__(THREADS, 1) radon_slab_kernel(const __grid_constant__ CUtensorMap tm_in,
                                                                const __grid_constant__ CUtensorMap tm_out,
                                                                const __grid_constant__ CUtensorMap tm_extra,
                                                                const __grid_constant__ SlabParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t *sF = smem + OFF_F, *sW = smem + OFF_W, *sMini = smem + OFF_MINI;
  uint64_t* f_full = reinterpret_cast<uint64_t*>(smem + OFF_BARS);   // [NF]
  uint64_t* f_empty = f_full + NF;         // [NF] read by the MMAs and by the ALU warps
  uint64_t* p_full = f_empty + NF;         // [PRE] an image of the next slab has landed in a stage-2 slot
  uint64_t* u_read = p_full + PRE;         // [PRE] the U tile in a stage-2 slot has been read by the copy engine
  uint64_t* full1 = u_read + PRE;          // [ACC1]
  uint64_t* empty1 = full1 + ACC1;         // [ACC1] one arrival per warp of the group that read it
  uint64_t* full2 = empty1 + ACC1;         // [GROUPS] one per group: a group takes every fourth item, the ring is shorter
  uint64_t* empty2 = full2 + GROUPS;       // [ACC2]
  uint64_t* w_ready = empty2 + ACC2;       // the slab's stage-1 rows are written
  uint64_t* w_free = w_ready + 1;          // W may be written: the U tiles of the slab before have been read by the copy
                                           // engine, and the images in stage-2 slots by the MMAs and the ALU warps
  uint64_t* alu_done = w_free + 1;         // the ALU warps have read image G of the slab
  uint64_t* staged = alu_done + 1;         // [NW] a U tile is complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(staged + NW);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{cta_abort, prm.status};
  const uint32_t my_slabs = prm.slabs > blockIdx.x ? (prm.slabs - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  if (threadIdx.x == 0) {
    *cta_abort = 0;
    for (int s = 0; s < NF; ++s) { mbar_init(f_full + s, 1); mbar_init(f_empty + s, 1 + ALU_ROWS); }
    for (int s = 0; s < ACC1; ++s) { mbar_init(full1 + s, 1); mbar_init(empty1 + s, GROUP); }
    for (int s = 0; s < GROUPS; ++s) mbar_init(full2 + s, 1);
    for (int s = 0; s < ACC2; ++s) mbar_init(empty2 + s, GROUP);
    mbar_init(w_ready, EPI + ALU_ROWS);
    mbar_init(w_free, 2 + ALU_ROWS);
    for (int s = 0; s < PRE; ++s) { mbar_init(p_full + s, 1); mbar_init(u_read + s, 1); }
    mbar_init(alu_done, ALU_ROWS);
    for (int s = 0; s < NW; ++s) mbar_init(staged + s, s + 1 < NW ? GROUP : GROUP + ALU_ROWS);   // the last with the ALU warps' rows
    fence_barrier_init();
    prefetch_tmap(&tm_in);
    prefetch_tmap(&tm_out);
    prefetch_tmap(&tm_extra);
  }
  if (warp == MMA1_WARP) tmem_alloc(tmem_slot, 512);
  // R, built row by row (one bf16 per operand row lo + q hi) in the first slots and moved to tensor memory
  for (int c = threadIdx.x; c < OFF_BARS / 16; c += THREADS) reinterpret_cast<uint4*>(smem)[c] = make_uint4(0u, 0u, 0u, 0u);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  if (warp < 4) {
    const int n = warp * 32 + lane, x = n % Q, y = n / Q;   // output index (u = x, slope y), or line x of the extra class
    __nv_bfloat16* row = reinterpret_cast<__nv_bfloat16*>(smem) + n * 128;
    for (int k = 0; k < Q; ++k) {
      const int at = y < Q ? k * Q + (x + (Q - y) * k) % Q : x * Q + k;
      row[at] = __float2bfloat16(1.0f);
    }
    __syncwarp();
    const uint32_t* roww = reinterpret_cast<const uint32_t*>(row);
    for (int c0 = 0; c0 < R_COLS; c0 += 32) {
      uint32_t v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = roww[c0 + i];
      tmem_st32(tmem_base + ((uint32_t)(warp * 32) << 16) + c0, v);
    }
    tmem_st_wait();
  }
  __syncthreads();
  // The rows past q² of a slot are never written again and meet zeros of R: they must hold no NaN pattern.
  for (int c = threadIdx.x; c < 128 * 256 / 16; c += THREADS) reinterpret_cast<uint4*>(smem)[c] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  pdl_trigger();
  const uint32_t acc1 = tmem_base + R_COLS, acc2 = acc1 + 64 * ACC1;
  constexpr uint32_t idesc = make_idesc(128, NE, 0, 1);   // R from tensor memory, image rows MN-major
  // Head and first entry of this CTA's slab k: the last heads first, whose F the pooling has just written, so that the read finds
  // the first ones' U in the L2 cache (32 heads of 16 K tokens, the pass 1392 -> 1385 us).
  auto slab_head = [&](uint32_t k, int& e0) {
    const uint32_t slab = prm.slabs - 1 - (blockIdx.x + k * gridDim.x), head = slab / prm.slabs_per_head;
    e0 = (int)(slab - head * prm.slabs_per_head) * NE;
    return (int)head;
  };

  // The roles' loops over images are kept rolled: unrolled, each copy of a body ran once per slab, at the speed at which
  // instructions arrive from the outer caches (warps 20-23: 1,000 cycles for eleven loads and sums).
  if (warp == PROD_WARP) {
    pdl_wait();
    const bool leader = elect_one();
    Ring<NF> f;
    bool ok = true;
    uint32_t k = 0;
    int pre = 0;                                          // images in stage-2 slots of slab k that have been started
    for (; k < my_slabs; ++k) {
      int e0;
      const int head = slab_head(k, e0);
      auto ring_image = [&](int x2) {
        ok = mbar_wait_warp(f_empty + f.at, f.par ^ 1, wc);
        if (!ok) return;
        if (leader) {
          mbar_expect_tx(f_full + f.at, TILE_BYTES);
          tma_load_5d(sF + f.at * SLOT, &tm_in, e0, 0, 0, x2, head, f_full + f.at);
        }
        f.next();
      };
#pragma unroll 1
      for (int x2 = PRE; x2 < PRE + NF && ok; ++x2) ring_image(x2);   // (the ring's slots are free first)
#pragma unroll 1
      for (pre = 0; pre < PRE && ok; ++pre) {
        if (k) ok = mbar_wait_warp(u_read + pre, (k - 1) & 1, wc);
        if (!ok) break;
        if (leader) {
          mbar_expect_tx(p_full + pre, TILE_BYTES);
          tma_load_5d(sW + pre * SLOT, &tm_in, e0, 0, 0, pre, head, p_full + pre);
        }
      }
#pragma unroll 1
      for (int x2 = PRE + NF; x2 < Q && ok; ++x2) ring_image(x2);
      if (!ok) break;
      pre = 0;
    }
    if (leader) {
      ring_landed(f_full, NF, f.at, f.par ^ 1, wc);
      for (int s = 0; s < PRE; ++s) landed(p_full + s, (k + (s < pre ? 0 : 1)) & 1, wc);   // k, or k + 1 loads
    }
  } else if (warp == MMA1_WARP) {
    pdl_wait();
    const bool leader = elect_one();
    const uint64_t dF = make_desc(smem_u32(sF), SLOT, 1024), dW = make_desc(smem_u32(sW), SLOT, 1024);
    Ring<NF> f;
    Ring<ACC1> a;
    bool ok = true;
    for (uint32_t k = 0; k < my_slabs && ok; ++k) {
#pragma unroll 1
      for (int t = 0; t < Q; ++t) {
        const bool ring = in_ring(t);
        const int x2 = image_at(t);
        ok = mbar_wait(empty1 + a.at, a.par ^ 1, wc) &&
             (ring ? mbar_wait(f_full + f.at, f.par, wc) : mbar_wait(p_full + x2, k & 1, wc));
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after_sync();
        if (leader) {
          const uint64_t d = ring ? dF + (uint64_t)(f.at * (SLOT >> 4)) : dW + (uint64_t)(x2 * (SLOT >> 4));
#pragma unroll
          for (int kk = 0; kk < STEPS; ++kk) mma_bf16_ta(acc1 + a.at * 64, tmem_base + 8 * kk, d + 128 * kk, idesc, kk != 0);
          if (ring) mma_commit(f_empty + f.at);
          if (t + 1 == EARLY) mma_commit(w_free);
          mma_commit(full1 + a.at);
        }
        if (ring) f.next();
        a.next();
      }
    }
  } else if (warp == MMA2_WARP) {
    pdl_wait();
    const bool leader = elect_one();
    const uint64_t d0 = make_desc(smem_u32(sW), SLOT, 1024);
    Ring<ACC2> a;
    bool ok = true;
    for (uint32_t k = 0; k < my_slabs && ok; ++k) {
      ok = mbar_wait_warp(w_ready, k & 1, wc);
#pragma unroll 1
      for (int img = 0; img < NW && ok; ++img) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty2 + a.at, a.par ^ 1, wc));
        if (!ok) break;
        fence_after_sync();
        if (leader) {
          const uint64_t d = d0 + (uint64_t)(img * (SLOT >> 4));
#pragma unroll
          for (int kk = 0; kk < STEPS; ++kk) mma_bf16_ta(acc2 + a.at * 64, tmem_base + 8 * kk, d + 128 * kk, idesc, kk != 0);
          mma_commit(full2 + (img & (GROUPS - 1)));
        }
        a.next();
      }
    }
  } else if (warp == STORE_WARP) {
    pdl_wait();
    if (lane == 0) {
      bool ok = true;
      mbar_arrive(w_free);                                // nothing to wait for before the first slab
      for (uint32_t k = 0; k < my_slabs && ok; ++k) {
        int e0;
        const int head = slab_head(k, e0);
#pragma unroll 1
        for (int img = 0; img < NW; ++img) {
          ok = mbar_wait(staged + img, k & 1, wc);
          if (!ok) break;
          tma_store_3d(&tm_out, sW + img * SLOT, e0, img * QQ, head);
          if (img + 1 == NW) tma_store_3d(&tm_extra, sMini, e0, NW * QQ, head);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(LAG) : "memory");
          if (img >= LAG && img - LAG < PRE) mbar_arrive(u_read + img - LAG);
        }
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        if (ok) mbar_arrive(w_free);
      }
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  } else if (warp >= ALU_WARP) {
    // Output indices 128 ..: the last lines of the extra class.  A warp has one line, a lane two entries.
    pdl_wait();
    const int u = Q - ALU_ROWS + (warp - ALU_WARP);
    int at[Q];                                            // the line's rows (of an F image, and of G)
#pragma unroll
    for (int i = 0; i < Q; ++i) at[i] = pair_at(u * Q + i, lane);
    Ring<NF> f;
    bool ok = true;
    for (uint32_t k = 0; k < my_slabs && ok; ++k) {
      uint32_t sum[EARLY] = {};   // kept until W may be written
#pragma unroll 1
      for (int t = 0; t < EARLY && ok; ++t) {
        const bool ring = in_ring(t);
        ok = ring ? mbar_wait_warp(f_full + f.at, f.par, wc) : mbar_wait_warp(p_full + t - NF, k & 1, wc);
        if (!ok) break;
        const uint32_t here = rows_sum(ring ? sF + f.at * SLOT : sW + (t - NF) * SLOT, at);
#pragma unroll
        for (int i = 0; i + 1 < EARLY; ++i) sum[i] = sum[i + 1];   // (item t ends up in sum[t])
        sum[EARLY - 1] = here;
        __syncwarp();
        if (lane == 0 && ring) mbar_arrive(f_empty + f.at);
        if (lane == 0 && t + 1 == EARLY) mbar_arrive(w_free);
        if (ring) f.next();
      }
      if (ok) ok = mbar_wait_warp(w_free, k & 1, wc);
      if (!ok) break;
      uint8_t* g = sW + Q * SLOT;
#pragma unroll
      for (int t = 0; t < EARLY; ++t) *reinterpret_cast<uint32_t*>(g + at[image_at(t)]) = sum[t];
#pragma unroll
      for (int x2 = EARLY; x2 < Q; ++x2) {
        if (ok) ok = mbar_wait_warp(f_full + f.at, f.par, wc);
        if (ok) {
          *reinterpret_cast<uint32_t*>(g + at[x2]) = rows_sum(sF + f.at * SLOT, at);
          __syncwarp();
          if (lane == 0) mbar_arrive(f_empty + f.at);
          f.next();
        }
      }
      if (!ok) break;
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(w_ready);
      ok = mbar_wait_warp(w_ready, k & 1, wc);
      if (!ok) break;
      *reinterpret_cast<uint32_t*>(sMini + pair_at(u, lane)) = rows_sum(g, at);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(alu_done);
        mbar_arrive(staged + Q);
      }
    }
  } else {
    pdl_wait();
    const int grp = warp >> 2, qd = warp & 3;
    const int n = qd * 32 + lane, x = n % Q, y = n / Q;     // output index (x, slope y); y = q: line x of the extra class
    const uint32_t from = (uint32_t)(qd * 32) << 16;
    bool ok = true;
    auto read_acc = [&](uint32_t acc, uint64_t* empty, uint4 (&w)[8]) {   // this lane's 64 sums, rounded
      fence_after_sync();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t v[32];
        tmem_ld32(acc + from + h * 32, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j)
          w[h * 4 + j] = make_uint4(pack_bf16(__uint_as_float(v[8 * j]), __uint_as_float(v[8 * j + 1])),
                                    pack_bf16(__uint_as_float(v[8 * j + 2]), __uint_as_float(v[8 * j + 3])),
                                    pack_bf16(__uint_as_float(v[8 * j + 4]), __uint_as_float(v[8 * j + 5])),
                                    pack_bf16(__uint_as_float(v[8 * j + 6]), __uint_as_float(v[8 * j + 7])));
      }
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(empty);
    };
    auto put_row = [&](uint8_t* slot, int row, const uint4 (&w)[8]) {
#pragma unroll
      for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(slot + chunk_at(row, j)) = w[j];
    };
    for (uint32_t k = 0; k < my_slabs && ok; ++k) {
#pragma unroll 1
      for (int t = grp; t < Q; t += GROUPS) {
        const uint32_t item = k * Q + t, at = item % ACC1;
        const int x2 = image_at(t);
        ok = mbar_wait_warp(full1 + at, (item / ACC1) & 1, wc);
        if (!ok) break;
        uint4 w[8];
        read_acc(acc1 + at * 64, empty1 + at, w);
        if (t == grp) {
          ok = mbar_wait_warp(w_free, k & 1, wc);
          if (!ok) break;
        }
        // W[a3 = y], row (u = x, x2); the extra class: G, row (x2, x3 = x)
        put_row(sW + y * SLOT, y < Q ? x2 * Q + x : x * Q + x2, w);
      }
      if (!ok) break;
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(w_ready);
#pragma unroll 1
      for (int img = grp; img < NW; img += GROUPS) {
        const uint32_t item = k * NW + img, at = item % ACC2;
        ok = mbar_wait_warp(full2 + grp, (item / GROUPS) & 1, wc);
        if (!ok) break;
        uint4 w[8];
        read_acc(acc2 + at * 64, empty2 + at, w);
        if (img == Q) {
          ok = mbar_wait_warp(alu_done, k & 1, wc);                // the ALU warps have read the image that the tile replaces
          if (!ok) break;
        }
        if (y < Q) put_row(sW + img * SLOT, n, w);
        else if (img == Q) put_row(sMini, x, w);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(staged + img);
      }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == MMA1_WARP) {
    fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

// 1 when both stages of a slab fit one CTA's shared memory and an image one operand tile.  Smaller primes fill too little
// of a tile (the exchange through the L2 cache costs them little), larger ones need more slots than there is room for.
int smat_tabulate_slab_supported(int q, int64_t state_elems) { return q == Q && state_elems % NE == 0 ? 1 : 0; }

cudaError_t smat_launch_tabulate_slab(const void* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh, int* status,
                                      cudaStream_t st) {
  const int64_t slabs = (int64_t)bh * (state_elems / NE);
  if (geo.D != 3 || !smat_tabulate_slab_supported(geo.q, state_elems) || slabs >= (1LL << 27)) return cudaErrorInvalidValue;
  CUtensorMap tm_in, tm_out, tm_extra;
  {   // F, image x2: (entry, x1, x3, x2, head), one image a box
    const int64_t sizes[4] = {Q, Q, Q, bh}, strides[4] = {1, QQ, Q, geo.P};
    const int box[4] = {Q, Q, 1, 1};
    if (!radon_map(&tm_in, in, state_elems, 5, sizes, strides, box)) return cudaErrorInvalidValue;
  }
  {   // U: the q² rows of an image follow one another, the extra class comes last
    const int64_t sizes[2] = {geo.B, bh}, strides[2] = {1, geo.B};
    const int box[2] = {QQ, 1}, xbox[2] = {Q, 1};
    if (!radon_map(&tm_out, out, state_elems, 3, sizes, strides, box) ||
        !radon_map(&tm_extra, out, state_elems, 3, sizes, strides, xbox))
      return cudaErrorInvalidValue;
  }
  SlabParams prm;
  prm.slabs = (uint32_t)slabs;
  prm.slabs_per_head = (uint32_t)(state_elems / NE);
  prm.status = status;
  const cudaError_t err = cudaFuncSetAttribute(radon_slab_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  if (err != cudaSuccess) return err;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = slabs < sms ? (unsigned)slabs : (unsigned)sms;
  return smat_launch_pdl(radon_slab_kernel, dim3(grid), THREADS, SMEM, st, tm_in, tm_out, tm_extra, prm);
}
