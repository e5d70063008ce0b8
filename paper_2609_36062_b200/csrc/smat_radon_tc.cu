// Tabulation U = C F (Algorithm 2) and its transpose F̄ = Cᵀ Ū on the tensor cores, for d = 3 and d = 4 with
// bf16 tables.
//
// The incidence matrix factors through the two-dimensional finite Radon transform over F_q x F_q,
//     (R f)(a, u) = Σ_{lo + a hi ≡ u} f(lo, hi)  for slopes a in F_q,      (R f)(∞, u) = Σ_lo f(lo, u),
// a 0/1 matrix with q^2 + q rows and q^2 columns:
//   d = 3 : U = R F, one image per state entry.
//   d = 4 : stage 1, one image per x2 :  W[a3][x2][u] = Σ_{x3} F[u - a3 x3, x2, x3],  G[x3][x2] = Σ_{x1} F[x1, x2, x3]
//           stage 2, one image per a3 :  U[(1, a2, a3), b] = Σ_{x2} W[a3][x2][b - a2 x2];
//                    the image G gives the directions (0, 1, a3) and (0, 0, 1).
// These are the sums of Algorithm 2 taken one coordinate pair at a time (same real numbers, different order).
// The transposes run the same stages backwards with Rᵀ.  R is small (q <= 23) and fixed, the images are
// independent across the r p state entries, so each stage is a product of a resident 0/1 matrix with a stream
// of images: dense enough for the tensor cores (q of every q^2 entries of a row are nonzero, and the
// 5th-generation tensor cores multiply-add about 60 times faster than the fp32 pipes add), bound by the image
// traffic.
//
// radon_tc_kernel, persistent, one CTA per SM.  An item is one image restricted to 128 consecutive state entries;
// R has up to 128 output indices (and for q = 11 four more, below), so one CTA covers an image:
//   warps 0-3      : build R once and move it to tensor memory (lane = output index, one column
//                    per two operand rows), where the MMAs read it as their A operand
//   warp 16 lane 0 : TMA producer; a ring slot holds `sps` lines (fixed hi, all lo) of the image x 128 state entries
//                    (MN-major B operand, two boxes of 64 entries); the extra class travels in a slot of its own
//   warps 17, 18 (lane 0) : MMA issuers, alternating items: D[128 outputs, 128 entries] += R_slot * B_slot; up to
//                    four accumulators in flight
//   warps 0-15     : epilogue, one output index (TMEM lane) per thread and one 32-entry column chunk per warp:
//                    round to bf16 and store 64 contiguous bytes of the output row as two 32-byte sectors
//   warps 19, 20   : q = 11 only.  q^2 + q = 132 output indices are one tile of 128 and 4 left over, all of the extra
//                    class (the sum of one line's q rows): these warps add them up from the ring slot itself, so
//                    that one CTA covers an image
// d = 4 with q <= 11 (forward with q = 11: smat_radon_slab.cu instead): both stages in ONE launch, slab by slab.  Stage 2
// of a slab needs stage 1 of every image of the same slab and nothing else, so a CTA keeps the slab's W rows in a private exchange buffer (q^3 + q^2 rows of 128
// entries, rewritten for every slab, stored and loaded with the L2 evict-last priority while F and U stream with
// evict-first) and the full-size W table is never built.  The storing warps make the slab's rows visible (memory
// fence, proxy fence) and arrive on a barrier the producer waits on before the first stage-2 load.
// That stage (d = 3, q = 11, forward) also sends its output tiles off by TMA: the epilogue writes the rounded tile into the
// item's own ring slot (as large as a tile, and dead once the MMAs have read it) in the box layout, and lane 0 of warp 18
// issues the tile stores and frees the slot; the bulk of the stores bypasses the LSU.
// The kernel exists twice: radon_tc_kernel<false> for one stage per launch with every index through the MMAs and direct
// stores (small primes), without cache hints or phase tables; radon_tc_kernel<true> with them.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_radon.cuh"
#include "smat_tc.cuh"

namespace {

using namespace tc;
using tc::tma_load_4d;
using tc::tma_load_5d;

constexpr int TILE_ROWS = 128;                    // output indices per tile (MMA M)
constexpr int EPI_WARPS = 16;
constexpr int PROD_WARP = EPI_WARPS;
constexpr int MMA_WARP = EPI_WARPS + 1;
constexpr int MMA_WARPS = 2;                      // issuing threads; they take the items alternately
constexpr int ALU_WARP = MMA_WARP + MMA_WARPS;    // first of the warps that sum the leftover extra-class rows
constexpr int ALU_WARPS = 2;
constexpr int ALU_MAX_ROWS = 8;
constexpr int RADON_THREADS = 32 * (ALU_WARP + ALU_WARPS);
constexpr int MAX_ACC = 4;                        // accumulators in flight: what the R columns leave of 512, at most 4
constexpr int RADON_EXCHANGE_CTAS = 148;          // CTAs of a one-launch two-stage tabulation (one exchange slab each)

// One stage: input and output index spaces, and where the rows live.  A "private" table is the exchange buffer of the
// two-stage kernel: [CTA][rows_per_head][128 entries], one slab per CTA, rewritten for every slab so that it stays in L2.
struct RadonPhase {
  RadonSide in, out;
  int32_t images;
  int32_t src_private, dst_private;
  int32_t src_heads;               // extent of the source maps' last coordinate: one past it reads zeros
  int64_t dst_pitch;               // entries per row of dst
  __nv_bfloat16* dst;
};

struct RadonParams {
  int32_t q, transpose;
  int32_t sps, sr;                 // lines (hi values) per ring slot; rows of a slot = sps*q rounded up to 16
  int32_t nreg, nslots;            // slots of regular lines per image; plus one when the input has the extra class
  int32_t rows_mma;                // output indices of the MMA tile (<= 128)
  int32_t alu_rows;                // output indices rows_mma .. (all of the extra class) summed on the ALUs, straight from
                                   // the ring slot; the tile then leaves through that slot and TMA stores.  0: every index
                                   // goes through the MMAs, direct stores
  int32_t ring;                    // ring slots
  int32_t mini_bytes;              // alu_rows: per slot, room for the extra-class rows of the tile (two halves)
  int32_t nph;                     // 1, or 2: both stages of the d = 4 tabulation, slab by slab
  int32_t slabs_per_head;          // rp / 128
  int64_t slabs;                   // heads * slabs_per_head
  RadonPhase ph[2];
  int* status;
};

// The items of one CTA, in the order every role walks them.  One phase: item = (slab, image) with the slab index
// fastest over the whole grid.  Two phases: slab by slab, the images of phase 0 and then those of phase 1, whose input
// is what phase 0 wrote for the same slab.
struct ItemIter {
  uint32_t slab, img, ph, left;    // the current item, and the items left including it
  uint32_t step, slabs, nph, im0, im1;
  __device__ __forceinline__ ItemIter(const RadonParams& p, uint32_t first, uint32_t step_, uint32_t nph_) {
    step = step_; slabs = (uint32_t)p.slabs; nph = nph_;
    im0 = (uint32_t)p.ph[0].images; im1 = nph > 1 ? (uint32_t)p.ph[1].images : 0u;
    ph = 0;
    if (nph == 1) {
      const uint32_t total = slabs * im0;                       // < 2^31 (checked by the launcher)
      left = first < total ? (total - 1 - first) / step + 1 : 0;
      img = first / slabs; slab = first - img * slabs;
    } else {
      left = first < slabs ? ((slabs - 1 - first) / step + 1) * (im0 + im1) : 0;
      img = 0; slab = first;
    }
  }
  __device__ __forceinline__ void next() {
    --left;
    if (nph == 1) {
      slab += step;
      while (slab >= slabs) { slab -= slabs; ++img; }
    } else if (++img == (ph ? im1 : im0)) {
      img = 0;
      if (ph == 0) ph = 1; else { ph = 0; slab += step; }
    }
  }
  // last item of phase 0 of a slab: phase 1 may start once its output is visible
  __device__ __forceinline__ bool closes_phase0() const { return nph > 1 && ph == 0 && img + 1 == im0; }
};

// Row of the streamed operand that holds input index (lo, line): slot line / sps, then the line's q rows.
__device__ __forceinline__ int operand_row(const RadonParams& p, int line, int lo) {
  if (line >= p.q) return p.nreg * p.sr + lo;                 // extra class: a slot of its own
  const int slot = line / p.sps;
  return slot * p.sr + (line - slot * p.sps) * p.q + lo;
}

// Marks in `row` (one bf16 per operand row, zeroed by the caller) the input indices incident with output index n.
// Forward: n = (u, a); a < q meets every line hi in lo = u - a hi, a = q (extra class) meets the whole line u.
// Transposed: n = point (lo, hi); it lies on one offset u = lo + a hi of every slope a, and on offset hi of the extra class.
__device__ __forceinline__ void mark_incident(const RadonParams& p, int n, __nv_bfloat16* row) {
  const int q = p.q, x = n % q, y = n / q;
  const __nv_bfloat16 one = __float2bfloat16(1.0f);
  if (!p.transpose) {
    if (y < q) {
      int lo = x;                                               // u - a*hi for hi = 0, 1, ...
      for (int hi = 0; hi < q; ++hi) {
        row[operand_row(p, hi, lo)] = one;
        lo -= y; if (lo < 0) lo += q;
      }
    } else {
      for (int lo = 0; lo < q; ++lo) row[operand_row(p, x, lo)] = one;
    }
  } else {
    int u = x;                                                  // lo + a*hi for a = 0, 1, ...
    for (int a = 0; a < q; ++a) {
      row[operand_row(p, a, u)] = one;
      u += y; if (u >= q) u -= q;
    }
    if (p.ph[0].in.count > q * q) row[operand_row(p, q, y)] = one;
  }
}

// box of 64 state entries x q rows x sps lines (regular map) or 64 x q rows (extra-class map)
__device__ __forceinline__ void tma_load_5d(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            int c4, uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
      ::"r"(smem_u32(smem_dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}

// L2 eviction policies: the exchange rows of the two-stage kernel should stay in the cache (they are rewritten for
// every slab, and written back to memory only when evicted), the tables streaming past them should leave it first.
enum { POLICY_NORMAL = 0, POLICY_FIRST = 1, POLICY_LAST = 2 };
__device__ __forceinline__ uint64_t l2_policy(int kind) {
  uint64_t p;
  if (kind == POLICY_FIRST) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  else if (kind == POLICY_LAST) asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void st_global_v8_hint(void* dst, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                                  uint32_t w4, uint32_t w5, uint32_t w6, uint32_t w7, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8}, %9;" ::"l"(dst), "r"(w0),
               "r"(w1), "r"(w2), "r"(w3), "r"(w4), "r"(w5), "r"(w6), "r"(w7), "l"(pol)
               : "memory");
}
// Tile stores: shared memory (box layout, 128-byte swizzle) -> global, as one bulk group per item.
__device__ __forceinline__ void tma_store_5d(const CUtensorMap* map, const void* smem_src, int c0, int c1, int c2, int c3,
                                             int c4, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3, %4, %5, %6}], [%1], %7;"
      ::"l"(map), "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, const void* smem_src, int c0, int c1, int c2, int c3,
                                             uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group.L2::cache_hint [%0, {%2, %3, %4, %5}], [%1], %6;"
      ::"l"(map), "r"(smem_u32(smem_src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// The MMAs of one ring slot: STEPS K-steps of 16 operand rows.  Fully unrolled so that the lone issuing thread spends
// a handful of instructions per MMA.  A K-step reads 8 columns of R (two bf16 per column) and 16 rows of the slot.
template <int STEPS>
__device__ __forceinline__ void issue_slot(uint32_t tmem_d, uint32_t tmem_a, uint64_t dB, uint32_t idesc, bool first) {
#pragma unroll
  for (int kk = 0; kk < STEPS; ++kk)
    mma_bf16_ta(tmem_d, tmem_a + kk * 8, dB + (uint64_t)(kk * 128), idesc, !(first && kk == 0));
}
__device__ __forceinline__ void issue_slot_steps(int steps, uint32_t tmem_d, uint32_t tmem_a, uint64_t dB, uint32_t idesc,
                                                 bool first) {
  switch (steps) {
    case 1: issue_slot<1>(tmem_d, tmem_a, dB, idesc, first); break;
    case 2: issue_slot<2>(tmem_d, tmem_a, dB, idesc, first); break;
    case 3: issue_slot<3>(tmem_d, tmem_a, dB, idesc, first); break;
    case 4: issue_slot<4>(tmem_d, tmem_a, dB, idesc, first); break;
    case 5: issue_slot<5>(tmem_d, tmem_a, dB, idesc, first); break;
    case 6: issue_slot<6>(tmem_d, tmem_a, dB, idesc, first); break;
    case 7: issue_slot<7>(tmem_d, tmem_a, dB, idesc, first); break;
    default: issue_slot<8>(tmem_d, tmem_a, dB, idesc, first); break;
  }
}

// FEAT = false is the plain instantiation (one stage per launch, every index through the MMAs, direct stores, no cache
// hints): the single-thread roles pay for every instruction, and the prime-specific paths would cost the others time.
template <bool FEAT>
__global__ void __launch_bounds__(RADON_THREADS, 1) radon_tc_kernel(const __grid_constant__ CUtensorMap tm_reg0,
                                                                    const __grid_constant__ CUtensorMap tm_vert0,
                                                                    const __grid_constant__ CUtensorMap tm_reg1,
                                                                    const __grid_constant__ CUtensorMap tm_vert1,
                                                                    const __grid_constant__ CUtensorMap tm_oreg0,
                                                                    const __grid_constant__ CUtensorMap tm_overt0,
                                                                    const RadonParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int q = prm.q;
  const int slot_bytes = prm.sr * 256;                          // two 64-entry blocks of sr rows x 128 bytes
  const int kt = prm.nslots * prm.sr;                           // operand rows per image
  uint8_t* sRing = smem;
  uint8_t* sMini = sRing + prm.ring * slot_bytes;                                  // [ring] extra-class rows (tma_out)
  int32_t* out_tab = reinterpret_cast<int32_t*>(sMini + prm.ring * prm.mini_bytes);  // [2][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(out_tab + 2 * TILE_ROWS);
  uint64_t* full = bars;                    // [ring] slot filled (TMA bytes)
  uint64_t* empty = bars + prm.ring;        // [ring] slot consumed by the MMAs (arrival from the epilogue, once the item is complete)
  uint64_t* acc_full = empty + prm.ring;    // [MAX_ACC] accumulator complete
  uint64_t* acc_empty = acc_full + MAX_ACC; // [MAX_ACC] accumulator read out (one arrival per epilogue warp)
  uint64_t* w_ready = acc_empty + MAX_ACC;  // phase 0 of the current slab written out (one arrival per storing warp)
  uint64_t* staged = w_ready + 1;           // [ring] tma_out: the item's tile is complete in its slot (one arrival per
                                            // epilogue warp)
  uint64_t* alu_done = staged + prm.ring;   // [ring] tma_out: the ALU warps have read the slot and written their rows
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(alu_done + prm.ring);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{cta_abort, prm.status};
  const bool tma_out = FEAT && prm.alu_rows > 0;
  const uint32_t nph = FEAT ? (uint32_t)prm.nph : 1u;

  if (threadIdx.x == 0) {
    *cta_abort = 0;
    for (int s = 0; s < prm.ring; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);   // (tma_out: the storing thread frees the slot)
      mbar_init(alu_done + s, ALU_WARPS);
      mbar_init(staged + s, EPI_WARPS);
    }
    for (int b = 0; b < MAX_ACC; ++b) { mbar_init(acc_full + b, 1); mbar_init(acc_empty + b, EPI_WARPS); }
    mbar_init(w_ready, EPI_WARPS);
    fence_barrier_init();
    prefetch_tmap(&tm_reg0);
    prefetch_tmap(&tm_vert0);
    if (nph > 1) { prefetch_tmap(&tm_reg1); prefetch_tmap(&tm_vert1); }
  }
  if (warp == MMA_WARP) tmem_alloc(tmem_slot, 512);
  // R, built row by row in the (still unused) ring and moved to tensor memory: lane = output
  // index, one column per two operand rows.  The launcher guarantees ring * slot_bytes >= 128 * kt * 2.
  __nv_bfloat16* scratch = reinterpret_cast<__nv_bfloat16*>(sRing);
  for (int c = threadIdx.x; c < prm.ring * (slot_bytes + prm.mini_bytes) / 16; c += blockDim.x)
    reinterpret_cast<uint4*>(sRing)[c] = make_uint4(0u, 0u, 0u, 0u);
  for (int n = threadIdx.x; n < TILE_ROWS; n += blockDim.x)
    for (int h = 0; h < (int)nph; ++h)
      out_tab[h * TILE_ROWS + n] = n < prm.rows_mma ? side_row(prm.ph[h].out, n, q) : ROW_INVALID;
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t r_cols = (uint32_t)((kt / 2 + 31) & ~31);       // columns taken by R
  const uint32_t nacc = min(MAX_ACC, (int)((512 - r_cols) / 128));
  if (warp < 4) {
    const int n = warp * 32 + lane;
    __nv_bfloat16* row = scratch + (size_t)n * kt;
    if (n < prm.rows_mma && n < prm.ph[0].out.count) mark_incident(prm, n, row);
    __syncwarp();
    const uint32_t* roww = reinterpret_cast<const uint32_t*>(row);
    for (int c0 = 0; c0 < (int)r_cols; c0 += 32) {
      uint32_t v[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = (c0 + i) * 2 < kt ? roww[c0 + i] : 0u;
      tmem_st32(tmem_base + ((uint32_t)(warp * 32) << 16) + c0, v);
    }
    tmem_st_wait();
  }
  __syncthreads();
  // rows no box writes must never hold NaN patterns: the ones just written are 0 or 1, which is fine
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  pdl_trigger();
  const uint32_t tmem_acc = tmem_base + r_cols;

  // per phase: streaming tables, or the exchange rows (two-stage kernel only)
  const uint64_t pol_src0 = l2_policy(nph > 1 ? (prm.ph[0].src_private ? POLICY_LAST : POLICY_FIRST) : POLICY_NORMAL);
  const uint64_t pol_src1 = l2_policy(nph > 1 ? (prm.ph[1].src_private ? POLICY_LAST : POLICY_FIRST) : POLICY_NORMAL);
  const uint64_t pol_dst0 = l2_policy(nph > 1 ? (prm.ph[0].dst_private ? POLICY_LAST : POLICY_FIRST) : POLICY_NORMAL);
  const uint64_t pol_dst1 = l2_policy(nph > 1 ? (prm.ph[1].dst_private ? POLICY_LAST : POLICY_FIRST) : POLICY_NORMAL);
  const uint32_t first = blockIdx.x, step = gridDim.x;
  const uint32_t sph = (uint32_t)prm.slabs_per_head;

  // ---- storing thread (tma_out: one stage, one slot per item): one bulk group of tile stores per item; the slot, which holds
  // the tile, goes back to the producer when the stores have read it.  Lane 0 of the second MMA warp, which has no items then.
  auto store_role = [&]() {
    pdl_wait();
    const RadonPhase& ph = prm.ph[0];
    const uint32_t ring = (uint32_t)prm.ring;
    uint32_t slot = 0, prev_slot = 0, par = 0;                  // par: what a slot's "staged" barrier shows
    bool have_prev = false;
    for (ItemIter it(prm, first, step, nph); it.left; it.next()) {
      const uint32_t head = it.slab / sph;
      const int e0 = (int)(it.slab - head * sph) * 128;
      if (!mbar_wait(staged + slot, par, wc)) break;
      const uint8_t *tile = sRing + slot * slot_bytes, *mini = sMini + slot * prm.mini_bytes;
      tma_store_5d(&tm_oreg0, tile, e0, 0, 0, (int)it.img, (int)head, pol_dst0);
      tma_store_5d(&tm_oreg0, tile + prm.sr * 128, e0 + 64, 0, 0, (int)it.img, (int)head, pol_dst0);
      if ((int)it.img >= ph.out.vert_from) {
        const int ci = ph.out.sv_img != 0 ? (int)it.img : 0;   // the map's image stride is sv_img rows
        tma_store_4d(&tm_overt0, mini, e0, 0, ci, (int)head, pol_dst0);
        tma_store_4d(&tm_overt0, mini + prm.mini_bytes / 2, e0 + 64, 0, ci, (int)head, pol_dst0);
      }
      bulk_commit();
      if (have_prev) {
        bulk_wait_read<1>();
        mbar_arrive(empty + prev_slot);
      }
      prev_slot = slot;
      have_prev = true;
      if (++slot == ring) { slot = 0; par ^= 1; }
    }
    if (have_prev) { bulk_wait_read<0>(); mbar_arrive(empty + prev_slot); }
    bulk_wait_all();
  };

  if (warp == PROD_WARP && lane == 0) {
    // ---- TMA producer -----------------------------------------------------------------------------------------
    pdl_wait();
    // The two single-thread roles keep running slot / parity counters: a lone thread pays the full latency of every
    // instruction, so divisions by the ring size inside the loop would show in the kernel time.
    uint32_t slot = 0, par = 0;                               // ring position; parity of the empty barrier's phase to wait for
    uint32_t wpar = 0;                                        // parity of w_ready for the current slab
    bool first_lap = true, ok = true;
    const uint32_t reg_bytes = 2u * 128u * (uint32_t)(q * prm.sps), vert_bytes = 2u * 128u * (uint32_t)q;
    for (ItemIter it(prm, first, step, nph); it.left && ok; it.next()) {
      const RadonPhase& ph = FEAT ? prm.ph[it.ph] : prm.ph[0];
      const CUtensorMap* tm_reg = FEAT && it.ph ? &tm_reg1 : &tm_reg0;
      const CUtensorMap* tm_vert = FEAT && it.ph ? &tm_vert1 : &tm_vert0;
      const uint32_t head = it.slab / sph;
      const int e0 = ph.src_private ? 0 : (int)(it.slab - head * sph) * 128;
      const int hc = ph.src_private ? (int)blockIdx.x : (int)head;
      const uint64_t pol = it.ph ? pol_src1 : pol_src0;
      if (it.ph == 1 && it.img == 0) {   // this slab's phase 0 output is complete and visible to the copy engine
        ok = mbar_wait(w_ready, wpar, wc);
        wpar ^= 1;
        fence_proxy_async_all();
        if (!ok) break;
      }
      for (int g = 0; g < prm.nslots; ++g) {
        if (!first_lap) ok = mbar_wait(empty + slot, par, wc);
        if (!ok) break;
        uint8_t* dst = sRing + slot * slot_bytes;
        if (g < prm.nreg) {   // lines hi = g*sps ..; lines past q - 1 are out of bounds and arrive as zeros
          mbar_expect_tx(full + slot, reg_bytes);
          if (FEAT) {
            tma_load_5d(dst, tm_reg, e0, 0, g * prm.sps, (int)it.img, hc, full + slot, pol);
            tma_load_5d(dst + prm.sr * 128, tm_reg, e0 + 64, 0, g * prm.sps, (int)it.img, hc, full + slot, pol);
          } else {
            tma_load_5d(dst, tm_reg, e0, 0, g * prm.sps, (int)it.img, hc, full + slot);
            tma_load_5d(dst + prm.sr * 128, tm_reg, e0 + 64, 0, g * prm.sps, (int)it.img, hc, full + slot);
          }
        } else {              // extra class; an image without it reads past the last head: zeros
          const int h = (int)it.img >= ph.in.vert_from ? hc : ph.src_heads;
          const int ci = (int)it.img * ph.in.sv_img;   // 0 when every image shares the rows
          mbar_expect_tx(full + slot, vert_bytes);
          if (FEAT) {
            tma_load_4d(dst, tm_vert, e0, 0, ci, h, full + slot, pol);
            tma_load_4d(dst + prm.sr * 128, tm_vert, e0 + 64, 0, ci, h, full + slot, pol);
          } else {
            tma_load_4d(dst, tm_vert, e0, 0, ci, h, full + slot);
            tma_load_4d(dst + prm.sr * 128, tm_vert, e0 + 64, 0, ci, h, full + slot);
          }
        }
        if (++slot == (uint32_t)prm.ring) {
          slot = 0;
          if (first_lap) { first_lap = false; par = 0; } else par ^= 1;
        }
      }
    }
    ring_landed(full, (uint32_t)prm.ring, slot, first_lap ? 1u : par, wc);
  } else if (warp >= MMA_WARP && warp < ALU_WARP && lane == 0) {
    // ---- MMA issuers: the two threads take the items alternately, so that the issue latency of one item (waits,
    // MMAs, commits: more than the tensor pipe needs for it) overlaps with the other thread's item.  Both phases
    // share R and the slot layout, so the issuers only count items. ---------------------------------------------
    pdl_wait();
    const uint32_t me = (uint32_t)(warp - MMA_WARP);
    if (tma_out && me == 1) store_role();
    constexpr uint32_t idesc = make_idesc(TILE_ROWS, 128, 0, 1);   // A from tensor memory (R), B MN-major (image rows)
    const uint64_t dB0 = make_desc(smem_u32(sRing), prm.sr * 128, 1024);
    const uint32_t slot16 = (uint32_t)slot_bytes >> 4;            // descriptor address units are 16 bytes
    const uint32_t slot_cols = (uint32_t)prm.sr / 2;              // columns of R per slot
    const int steps = prm.sr / 16, nslots = prm.nslots;
    const int steps_last = ((q - (prm.nreg - 1) * prm.sps) * q + 15) / 16, steps_extra = (q + 15) / 16;
    const uint32_t ring = (uint32_t)prm.ring;
    const uint32_t items = ItemIter(prm, first, step, nph).left;
    uint32_t slot = 0, par = 0;                                   // ring position and the parity its full barrier shows
    uint32_t buf = 0, apar = 0;                                   // accumulator; parity of its empty barrier's phase to wait for
    bool ok = true;
    if (nslots == 1) {
      // One slot per item (q <= 11): a single thread, and the leanest loop: every instruction here is on the
      // critical path of the stage.
      for (uint32_t n_item = 0; me == 0 && n_item < items && ok; ++n_item) {
        if (n_item >= nacc) ok = mbar_wait(acc_empty + buf, apar, wc);
        if (!ok) break;
        ok = mbar_wait(full + slot, par, wc);
        if (!ok) break;
        fence_after_sync();
        issue_slot_steps(steps, tmem_acc + buf * 128, tmem_base, dB0 + (uint64_t)(slot * slot16), idesc, true);
        if (!tma_out) mma_commit(empty + slot);   // tma_out: the storing thread frees the slot once the tile has left it
        mma_commit(acc_full + buf);
        if (++slot == ring) { slot = 0; par ^= 1; }
        if (++buf == nacc) { buf = 0; if (n_item >= nacc) apar ^= 1; }
      }
    } else {
      uint32_t turn = 0;
      for (uint32_t n_item = 0; n_item < items && ok; ++n_item) {
        const bool mine = turn == me;
        if (++turn == MMA_WARPS) turn = 0;
        if (!mine) {   // the other thread's item: step the counters over it
          for (int g = 0; g < nslots; ++g)
            if (++slot == ring) { slot = 0; par ^= 1; }
          if (++buf == nacc) { buf = 0; if (n_item >= nacc) apar ^= 1; }
          continue;
        }
        if (n_item >= nacc) ok = mbar_wait(acc_empty + buf, apar, wc);
        if (!ok) break;
        fence_after_sync();
        const uint32_t tmem_d = tmem_acc + buf * 128;
        uint32_t tmem_a = tmem_base;
        for (int g = 0; g < nslots && ok; ++g, tmem_a += slot_cols) {
          ok = mbar_wait(full + slot, par, wc);
          if (!ok) break;
          fence_after_sync();
          // the last slot of regular lines and the slot of the extra class hold fewer rows than a full slot: R has
          // only zeros for the rest, so their K-steps are left out
          const int st = g + 1 < prm.nreg ? steps : (g < prm.nreg ? steps_last : steps_extra);
          issue_slot_steps(st, tmem_d, tmem_a, dB0 + (uint64_t)(slot * slot16), idesc, g == 0);
          if (++slot == ring) { slot = 0; par ^= 1; }
        }
        if (ok) mma_commit(acc_full + buf);   // the only commit of the item: the epilogue frees its slots when it sees it
        if (++buf == nacc) { buf = 0; if (n_item >= nacc) apar ^= 1; }
      }
    }
  } else if (FEAT && warp >= ALU_WARP) {
    // ---- leftover rows on the ALUs ----------------------------------------------------------------------------
    // q*q + q output indices rarely fill whole tiles of 128.  When only a few are left over, and they belong to the
    // extra class (index q*q + u = the sum of line u's q rows), these warps add the rows up from the slot itself
    // instead of a second, nearly empty tile paying for every MMA again.  A task is one leftover index and 8 state
    // entries (one 16-byte chunk of the swizzled slot).
    if (tma_out) {
      pdl_wait();
      const int tid_a = (warp - ALU_WARP) * 32 + lane, tasks = prm.alu_rows * 16;
      const uint32_t ring = (uint32_t)prm.ring;
      uint32_t slot = 0, par = 0;
      for (ItemIter it(prm, first, step, nph); it.left; it.next()) {
        if (!mbar_wait_warp(full + slot, par, wc)) break;
        if ((int)it.img >= prm.ph[0].out.vert_from) {
          const uint8_t* sl = sRing + slot * slot_bytes;
          for (int task = tid_a; task < tasks; task += 32 * ALU_WARPS) {
            const int u = prm.rows_mma + (task >> 4) - q * q, ch = task & 15;
            const uint8_t* blk = sl + (ch >> 3) * prm.sr * 128;
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.f;
            for (int lo = 0; lo < q; ++lo) {
              const int r = u * q + lo;                           // operand row of (line u, lo): one slot holds every line
              const uint4 w = *reinterpret_cast<const uint4*>(blk + r * 128 + (((ch & 7) ^ (r & 7)) << 4));
              acc[0] += __uint_as_float(w.x << 16); acc[1] += __uint_as_float(w.x & 0xffff0000u);
              acc[2] += __uint_as_float(w.y << 16); acc[3] += __uint_as_float(w.y & 0xffff0000u);
              acc[4] += __uint_as_float(w.z << 16); acc[5] += __uint_as_float(w.z & 0xffff0000u);
              acc[6] += __uint_as_float(w.w << 16); acc[7] += __uint_as_float(w.w & 0xffff0000u);
            }
            // into the slot's extra-class rows, from where the storing thread sends them with the tile
            uint8_t* mrow = sMini + slot * prm.mini_bytes + (ch >> 3) * (prm.mini_bytes / 2) + u * 128;
            *reinterpret_cast<uint4*>(mrow + (((ch & 7) ^ (u & 7)) << 4)) =
                make_uint4(pack_bf16(acc[0], acc[1]), pack_bf16(acc[2], acc[3]), pack_bf16(acc[4], acc[5]),
                           pack_bf16(acc[6], acc[7]));
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(alu_done + slot);
        if (++slot == ring) { slot = 0; par ^= 1; }
      }
    }
  } else if (warp < EPI_WARPS) {
    // ---- epilogue ---------------------------------------------------------------------------------------------
    pdl_wait();
    // Warp w reads lane quarter w % 4 (32 output indices) and the 32-entry column chunk w / 4 of every item.
    const int qd = warp & 3, cb = warp >> 2;
    const int orow = qd * 32 + lane;                            // output index of this CTA = TMEM lane
    const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
    const int tv0 = out_tab[orow], tv1 = nph > 1 ? out_tab[TILE_ROWS + orow] : ROW_INVALID;
    const bool active = qd * 32 < prm.rows_mma;                 // warp-uniform: some output index in these lanes
    uint32_t buf = 0, apar = 0, eslot = 0, epar = 0;
    // tma_out: where this thread's 64 bytes go inside the slot (or inside the slot's extra rows)
    const bool st_mini = orow >= q * q;
    const int st_idx = st_mini ? orow - q * q : orow;
    const int st_off = (cb >> 1) * (st_mini ? prm.mini_bytes / 2 : prm.sr * 128) + st_idx * 128;
    for (ItemIter it(prm, first, step, nph); it.left; it.next()) {
      const RadonPhase& ph = FEAT ? prm.ph[it.ph] : prm.ph[0];
      const uint32_t head = it.slab / sph;
      const int e0 = ph.dst_private ? 0 : (int)(it.slab - head * sph) * 128;
      const int64_t hrow = (int64_t)(ph.dst_private ? blockIdx.x : head) * ph.out.rows_per_head;
      const int tv = it.ph ? tv1 : tv0;
      if (!mbar_wait_warp(acc_full + buf, apar, wc)) break;
      fence_after_sync();
      if (tma_out) {
        // The tile leaves through the item's own slot (the MMAs are done with it): every thread writes its 64 bytes
        // in the box layout of a TMA tile — regular indices into the slot (row = index), extra-class indices into
        // the slot's extra rows — and the storing thread sends the tile off.  The LSU sees 4 wavefronts per warp
        // store instead of 32, and the bulk of the traffic bypasses it.
        uint32_t v[32];
        tmem_ld32(tmem_acc + lane_base + buf * 128 + cb * 32, v);
        tmem_ld_wait();
        fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + buf);             // the accumulator is in registers
        if (!mbar_wait_warp(alu_done + eslot, epar, wc)) break;   // the ALU warps have read the image
        if (tv != ROW_INVALID) {
          const int idx = st_idx;
          uint8_t* trow = (st_mini ? sMini + eslot * prm.mini_bytes : sRing + eslot * slot_bytes) + st_off;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4*>(trow + ((((cb & 1) * 4 + j) ^ (idx & 7)) << 4)) =
                make_uint4(pack_bf16(__uint_as_float(v[8 * j]), __uint_as_float(v[8 * j + 1])),
                           pack_bf16(__uint_as_float(v[8 * j + 2]), __uint_as_float(v[8 * j + 3])),
                           pack_bf16(__uint_as_float(v[8 * j + 4]), __uint_as_float(v[8 * j + 5])),
                           pack_bf16(__uint_as_float(v[8 * j + 6]), __uint_as_float(v[8 * j + 7])));
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(staged + eslot);
        if (++eslot == (uint32_t)prm.ring) { eslot = 0; epar ^= 1; }
        if (++buf == nacc) { buf = 0; apar ^= 1; }
        continue;
      }
      if (warp == 0 && prm.nslots > 1) {   // every MMA of the item has completed: its ring slots are free (a commit per slot would cost the
                         // issuing thread more than the MMAs of the slot)
        for (int g = 0; g < prm.nslots; ++g) {
          if (lane == 0) mbar_arrive(empty + eslot);
          if (++eslot == (uint32_t)prm.ring) eslot = 0;
        }
      }
      if (active) {
        uint32_t v[32];
        tmem_ld32(tmem_acc + lane_base + buf * 128 + cb * 32, v);
        tmem_ld_wait();
        const bool vert = (int)it.img >= ph.out.vert_from;
        if (tv != ROW_INVALID && (!(tv & ROW_VERT) || vert)) {
          const int row = (tv & ROW_VERT) ? ph.out.v0 + (int)it.img * ph.out.sv_img + (tv & ~ROW_VERT)
                                          : (int)it.img * ph.out.s_img + tv;
          __nv_bfloat16* dst = ph.dst + (hrow + row) * ph.dst_pitch + e0 + cb * 32;
#pragma unroll
          for (int h8 = 0; h8 < 2; ++h8) {   // two whole 32-byte sectors per thread
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              w[i] = pack_bf16(__uint_as_float(v[16 * h8 + 2 * i]), __uint_as_float(v[16 * h8 + 2 * i + 1]));
            if (FEAT)
              st_global_v8_hint(dst + 16 * h8, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7], it.ph ? pol_dst1 : pol_dst0);
            else
              st_global_v8(dst + 16 * h8, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
          }
        }
      }
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty + buf);
      if (it.closes_phase0()) {   // the slab's phase 0 rows before the copy engine reads them
        __threadfence();
        fence_proxy_async_all();
        __syncwarp();
        if (lane == 0) mbar_arrive(w_ready);
      }
      if (++buf == nacc) { buf = 0; apar ^= 1; }
    }
  }
  fence_before_sync();
  __syncthreads();
  if (warp == MMA_WARP) {
    fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

struct RadonShape {
  int sps, sr, nreg, nslots, rows_mma, alu_rows, ring, mini_bytes, smem;
};

// Ring slots of `sps` lines (sps*q rows, rounded up to 16), chosen for the least MMA work.  R (128 lanes x one column per two
// operand rows) and at least two accumulators of 128 columns must fit the 512 columns of tensor memory, and the ring must be
// able to hold the scratch copy of R while it is built.  Returns false when q is too large for this kernel.
bool radon_shape(int q, int transpose, int in_has_extra, int count_out, RadonShape* s) {
  const int budget = 227 * 1024 - 1024 - 512 - TILE_ROWS * 8;
  if (q < 2 || q > 64) return false;
  // A few indices past a full tile, all of the extra class, with every line in one slot, are left to the ALUs (q = 11:
  // 132 = 128 + 4 indices).
  const int left = count_out > TILE_ROWS ? count_out - TILE_ROWS : 0;
  if (left > 0 && (left > ALU_MAX_ROWS || transpose || in_has_extra || TILE_ROWS < q * q)) return false;
  int best = 1 << 30;
  for (int sps = 1; sps <= q; ++sps) {
    const int sr = (sps * q + 15) & ~15;
    if (sr > 128) break;
    const int nreg = (q + sps - 1) / sps, nslots = nreg + (in_has_extra ? 1 : 0);
    const int r_cols = (nslots * sr / 2 + 31) & ~31;
    if (r_cols + 2 * 128 > 512) continue;
    const int slot_bytes = sr * 256;
    int ring = budget / slot_bytes;
    if (ring > 8) ring = 8;
    if (ring < 3 || ring < nslots || (nslots > 1 && ring < 2 * nslots)) continue;   // several slots per item are freed
                                                                                    // together: room for two items
    const int cost = nslots * (sr + 48);   // operand rows per image, plus a charge per slot for its hand-over
    if (cost < best) {
      best = cost;
      s->sps = sps; s->sr = sr; s->nreg = nreg; s->nslots = nslots;
      s->rows_mma = count_out - left; s->alu_rows = left; s->ring = ring; s->mini_bytes = 0;
      s->smem = ring * slot_bytes + TILE_ROWS * 8 + 512 + 1024;
    }
  }
  if (best == (1 << 30)) return false;
  if (left == 0) return true;
  // The tile is stored by TMA from the item's own slot, which is as large; every slot gets room for the q extra-class rows of
  // its tile (two 64-entry halves).
  if (s->nslots != 1 || s->sps < q || s->sr != TILE_ROWS) return false;
  s->mini_bytes = 2 * ((q + 7) & ~7) * 128;
  const int slot_bytes = s->sr * 256 + s->mini_bytes, ring = budget / slot_bytes;
  if (ring < s->ring) s->ring = ring;
  s->smem = s->ring * slot_bytes + TILE_ROWS * 8 + 512 + 1024;
  return s->ring >= 4;
}

// The shared-memory map of radon_tc_kernel for a shape, checked on the host before every launch: ring slots, the
// per-slot extra-class rows (tile stores only), the output-row table and the barrier words must be disjoint and inside
// the allocation; nothing the copy engine or a thread writes for a slot may leave the slot.
//   [0, ring * slot)                      ring slots, slot = 2 halves of sr rows x 128 bytes (1024-byte aligned: sr % 16 == 0)
//   [.., + ring * mini)                   extra-class rows per slot (two halves of mini / 2)
//   [.., + 2 * 128 * 4)                   output-row table
//   [.., + (4 ring + 2 MAX_ACC + 1) * 8 + 8)   barriers, the tensor-memory slot word, the abort flag
bool radon_layout_ok(int q, const RadonShape& sh, int in_has_extra) {
  const int slot = sh.sr * 256, half = sh.sr * 128;
  const int bars = (4 * sh.ring + 2 * MAX_ACC + 1) * 8 + 8;
  bool ok = sh.sr % 16 == 0 && sh.sr <= TILE_ROWS && sh.ring >= sh.nslots;        // the scratch copy of R: 128 rows x kt bf16
  ok = ok && sh.nslots == sh.nreg + (in_has_extra ? 1 : 0) && sh.nreg * sh.sps >= q;
  ok = ok && q * sh.sps * 128 <= half && q * 128 <= half;                         // a load box (lines or extra class) per half
  ok = ok && ((sh.nslots * sh.sr / 2 + 31) & ~31) + 2 * 128 <= 512;               // R columns and two accumulators
  ok = ok && sh.rows_mma <= TILE_ROWS;
  if (sh.alu_rows)   // the tile is written into the item's slot: one 128-byte row per regular output index, the others behind
    ok = ok && sh.nslots == 1 && q * q <= sh.sr && sh.rows_mma >= q * q && sh.mini_bytes % 2048 == 0 && sh.mini_bytes / 2 >= q * 128;
  ok = ok && 1023 + sh.ring * (slot + sh.mini_bytes) + 2 * TILE_ROWS * 4 + bars <= sh.smem && sh.smem <= 227 * 1024;
  return ok;
}

// nph = 1: one stage over the whole tables.  nph = 2: both stages in one launch, which must share R (the same
// direction, the same index counts) and exchange their rows through the private buffer.
cudaError_t launch_radon(int q, int transpose, int nph, const StageSpec* sp, int64_t rp, int bh, int* status,
                         cudaStream_t st) {
  RadonShape sh;
  const int in_has_extra = sp[0].in.count > q * q;
  int max_images = sp[0].images;
  if (nph == 2 && sp[1].images > max_images) max_images = sp[1].images;
  if (!radon_shape(q, transpose, in_has_extra, sp[0].out.count, &sh) || rp % 128 ||
      (int64_t)bh * (rp / 128) * max_images * 2 >= (1LL << 31))
    return cudaErrorInvalidValue;
  if (nph == 2 && (sp[1].in.count != sp[0].in.count || sp[1].out.count != sp[0].out.count || sh.alu_rows > 0))
    return cudaErrorInvalidValue;
  RadonParams prm;
  prm.q = q; prm.transpose = transpose; prm.sps = sh.sps; prm.sr = sh.sr; prm.nreg = sh.nreg; prm.nslots = sh.nslots;
  prm.rows_mma = sh.rows_mma; prm.alu_rows = sh.alu_rows;
  prm.ring = sh.ring; prm.nph = nph; prm.slabs_per_head = (int)(rp / 128); prm.slabs = (int64_t)bh * (rp / 128);
  prm.status = status;
  prm.mini_bytes = sh.mini_bytes;
  if (!radon_layout_ok(q, sh, in_has_extra)) return cudaErrorInvalidConfiguration;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (nph == 2 && sms > RADON_EXCHANGE_CTAS) sms = RADON_EXCHANGE_CTAS;  // one private exchange slab per CTA was sized for
  int64_t ctas = sms;
  const int64_t items = nph == 1 ? prm.slabs * sp[0].images : prm.slabs;
  if (items < ctas) ctas = items;
  CUtensorMap tm_reg[2], tm_vert[2];
  for (int i = 0; i < nph; ++i) {
    RadonPhase& ph = prm.ph[i];
    const RadonSide& in = sp[i].in;
    const int images = sp[i].images;
    const int64_t src_rp = sp[i].src_private ? 128 : rp, src_heads = sp[i].src_private ? ctas : bh;
    ph.in = in; ph.out = sp[i].out; ph.images = images;
    ph.src_private = sp[i].src_private; ph.dst_private = sp[i].dst_private;
    ph.src_heads = (int)src_heads;
    ph.dst_pitch = sp[i].dst_private ? 128 : rp;
    ph.dst = static_cast<__nv_bfloat16*>(sp[i].dst);
    {   // regular lines: (entry, lo, hi, image, head); a size-one dimension keeps its stride valid
      const int64_t sizes[4] = {q, q, images, src_heads};
      const int64_t strides[4] = {in.s_lo, in.s_hi, images > 1 ? in.s_img : in.rows_per_head, in.rows_per_head};
      const int box[4] = {q, sh.sps, 1, 1};
      if (!radon_map(&tm_reg[i], sp[i].src, src_rp, 5, sizes, strides, box)) return cudaErrorInvalidValue;
    }
    if (in_has_extra) {   // extra class: (entry, lo, image, head), rows v0 + image*sv_img + lo*sv_lo
      const bool per_image = in.sv_img != 0;
      const int64_t sizes[3] = {q, per_image ? images : 1, src_heads};
      const int64_t strides[3] = {in.sv_lo, per_image ? in.sv_img : in.rows_per_head, in.rows_per_head};
      const int box[3] = {q, 1, 1};
      if (!radon_map(&tm_vert[i], static_cast<const __nv_bfloat16*>(sp[i].src) + (int64_t)in.v0 * src_rp, src_rp, 4, sizes,
                     strides, box))
        return cudaErrorInvalidValue;
      ph.in.sv_img = per_image ? 1 : 0;   // the kernel passes image * sv_img as the coordinate
    } else {
      tm_vert[i] = tm_reg[i];
    }
  }
  CUtensorMap tm_oreg = tm_reg[0], tm_overt = tm_reg[0];
  if (prm.alu_rows > 0) {   // the same two shapes over the output rows: boxes of q lines, and of the extra class
    const RadonSide& out = sp[0].out;
    const int images = sp[0].images;
    const bool per_image = out.sv_img != 0;
    const int64_t sizes[4] = {q, q, images, bh}, vsizes[3] = {q, per_image ? images : 1, bh};
    const int64_t strides[4] = {out.s_lo, out.s_hi, images > 1 ? out.s_img : out.rows_per_head, out.rows_per_head};
    const int64_t vstrides[3] = {out.sv_lo, per_image ? out.sv_img : out.rows_per_head, out.rows_per_head};
    const int box[4] = {q, q, 1, 1}, vbox[3] = {q, 1, 1};
    if (!radon_map(&tm_oreg, sp[0].dst, rp, 5, sizes, strides, box) ||
        !radon_map(&tm_overt, static_cast<__nv_bfloat16*>(sp[0].dst) + (int64_t)out.v0 * rp, rp, 4, vsizes, vstrides, vbox))
      return cudaErrorInvalidValue;
  }
  if (nph == 1) {
    prm.ph[1] = prm.ph[0]; tm_reg[1] = tm_reg[0]; tm_vert[1] = tm_vert[0];
  }
  const bool feat = nph > 1 || prm.alu_rows > 0;
  // the plain instantiation has no use for the two ALU warps
  const unsigned threads = feat ? RADON_THREADS : 32 * ALU_WARP;
  auto kernel = feat ? radon_tc_kernel<true> : radon_tc_kernel<false>;
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem);
  if (err != cudaSuccess) return err;
  return smat_launch_pdl(kernel, dim3((unsigned)ctas), threads, sh.smem, st, tm_reg[0], tm_vert[0], tm_reg[1], tm_vert[1], tm_oreg,
                         tm_overt, prm);
}

// The two stages of d = 4 run as one launch when a CTA's exchange rows (q^3 + q^2 rows of 128 entries), times the
// CTAs of the grid, stay well inside the L2 cache, and one CTA covers every output index of an image.
bool radon_two_stage_fits(int q, int transpose) {
  RadonShape sh;
  const int qq = q * q;
  if (!radon_shape(q, transpose, transpose ? 1 : 0, transpose ? qq : qq + q, &sh)) return false;
  return ((int64_t)qq * q + qq) * 256 * RADON_EXCHANGE_CTAS <= (64LL << 20);
}

}  // namespace

// Which kernel runs a stage: q = 17 the one with the sparse form of the matrix in tensor memory (smat_radon_sparse.cu), q = 13
// (and d = 3 beyond) the one that generates it, smaller primes, whose outputs are one tile, the kernel above.  Measured (ms):
// q = 17, 64 heads of 8192 tokens, d = 3, three CTAs of the kernel above sharing every image 0.257, sparse 0.204; transposed,
// generated 0.270, sparse 0.206; d = 4, 2 heads of 64 K tokens, three CTAs 0.302, sparse 0.241.  q = 13, d = 3, 32 heads of 4096
// tokens, generated 0.071, sparse 0.071; d = 4, 4 heads of 40960 tokens 0.211, sparse 0.220.
static bool sparse_matrix(int q) { return radon_sparse_fits(q); }
static bool generates_matrix(int q) { return q == 13; }

// The stages of a tabulation of prime q, D = 2 or 3, without their tables.  fused: those of D = 3 run as one launch with
// the table between them in the private exchange buffer.
static int radon_stages(int q, int D, int transpose, bool fused, StageSpec (&sp)[2]) {
  const int qq = q * q, qqq = qq * q;
  if (D == 2) {
    const RadonSide pts = side(qq, 1, q, 0, qq);
    const RadonSide typ = side(qq + q, 1, q, 0, qq + q, qq, 1, 0, 0);
    sp[0] = transpose ? stage(typ, pts, 1, nullptr, nullptr) : stage(pts, typ, 1, nullptr, nullptr);
    return 1;
  }
  const int64_t wrows = qqq + qq;
  const RadonSide f_side = side(qq, 1, qq, q, qqq);                         // image x2, points (x1, x3)
  const RadonSide w1_side = side(qq + q, 1, qq, q, wrows, qqq, q, 1, 0);    // (u, a3) -> W[a3][x2][u]; extra class -> G[x3][x2]
  const RadonSide w2_side = side(qq, 1, q, qq, wrows);                      // image a3 (image q: G), points (u, x2)
  const RadonSide u_side = side(qq + q, 1, q, qq, wrows + q, qqq + qq, 1, 0, q);
  if (!transpose) {
    sp[0] = stage(f_side, w1_side, q, nullptr, nullptr, false, fused);
    sp[1] = stage(w2_side, u_side, q + 1, nullptr, nullptr, fused, false);
  } else {
    sp[0] = stage(u_side, w2_side, q + 1, nullptr, nullptr, false, fused);
    sp[1] = stage(w1_side, f_side, q, nullptr, nullptr, fused, false);
  }
  return 2;
}

// 1 when the tensor-core tabulation covers this geometry (d = 3 or 4): every stage of both directions fits the kernel that
// would run it.
int smat_tabulate_tc_supported(const SmatGeo& geo, int64_t state_elems) {
  if ((geo.D != 2 && geo.D != 3) || state_elems % 128) return 0;
  const int q = geo.q;
  for (int transpose = 0; transpose < 2; ++transpose) {
    StageSpec sp[2];
    const int stages = radon_stages(q, geo.D, transpose, false, sp);
    for (int i = 0; i < stages; ++i) {
      RadonShape sh;
      if (!(sparse_matrix(q) || (generates_matrix(q) && radon_wide_fits(q, sp[i])) || radon_shape(q, transpose, sp[i].in.count > q * q, sp[i].out.count, &sh)))
        return 0;
    }
  }
  return 1;
}

// Rows (of state_elems bf16 each, per head) of the intermediate table the d = 4 stages exchange.
int64_t smat_tabulate_tc_scratch_rows(const SmatGeo& geo) {
  return geo.D == 3 ? (int64_t)geo.q * geo.q * geo.q + (int64_t)geo.q * geo.q : 0;
}

// bf16 elements of the scratch table smat_launch_tabulate_tc needs: the whole intermediate table W, or, when both
// directions run their two stages in one launch, one slab of it (128 entries per row) per CTA.
int64_t smat_tabulate_tc_scratch_elems(const SmatGeo& geo, int64_t state_elems, int bh) {
  const int64_t rows = smat_tabulate_tc_scratch_rows(geo);
  if (rows == 0) return 0;
  if (radon_two_stage_fits(geo.q, 0) && radon_two_stage_fits(geo.q, 1)) {
    int64_t ctas = (int64_t)bh * (state_elems / 128);
    if (ctas > RADON_EXCHANGE_CTAS) ctas = RADON_EXCHANGE_CTAS;
    return ctas * rows * 128;
  }
  return (int64_t)bh * rows * state_elems;
}

// Host-only: 1 when every stage of a tabulation of prime q has a kernel whose shared-memory map holds: the resident matrix
// (with its tile stores at q = 11), the generated one, or, for d = 3 alone, its forward
// stage.  (The both-stages kernel of smat_radon_slab.cu has one map, asserted where it is compiled.)
int smat_tabulate_tc_layout_ok(int q) {
  StageSpec sp[2];
  if (q >= 19) {
    radon_stages(q, 2, 0, false, sp);
    return radon_wide_layout_ok(q, sp[0]) ? 1 : 0;
  }
  for (int D = 2; D <= 3; ++D)
    for (int transpose = 0; transpose < 2; ++transpose) {
      const int stages = radon_stages(q, D, transpose, false, sp);
      for (int i = 0; i < stages; ++i) {
        if (sparse_matrix(q)) continue;   // (its maps are asserted where it is compiled)
        if (generates_matrix(q)) {
          if (!radon_wide_layout_ok(q, sp[i])) return 0;
          continue;
        }
        const int extra = sp[i].in.count > q * q;
        RadonShape sh;
        if (!radon_shape(q, transpose, extra, sp[i].out.count, &sh)) return 0;
        if (!radon_layout_ok(q, sh, extra)) return 0;
      }
    }
  return 1;
}

// transpose = 0: in = F [bh][P][rp] bf16, out = U [bh][B][rp] bf16.  transpose = 1: in = Ū [bh][B][rp], out = F̄ [bh][P][rp].
// scratch: smat_tabulate_tc_scratch_elems bf16 (d = 4 only).  One launch for d = 3; one or two for d = 4.
cudaError_t smat_launch_tabulate_tc(const void* in, void* out, void* scratch, const SmatGeo& geo, int64_t state_elems,
                                    int bh, int transpose, int* status, cudaStream_t st, int* launches) {
  const int q = geo.q;
  *launches = 0;
  if (geo.D != 2 && geo.D != 3) return cudaErrorInvalidValue;
  if (geo.D == 3 && !transpose && smat_tabulate_slab_supported(q, state_elems)) {
    *launches = 1;
    return smat_launch_tabulate_slab(in, out, geo, state_elems, bh, status, st);
  }
  const bool fused = geo.D == 3 && radon_two_stage_fits(q, transpose);
  StageSpec sp[2];
  const int stages = radon_stages(q, geo.D, transpose, fused, sp);
  sp[0].src = in;
  sp[stages - 1].dst = out;
  if (stages == 2) { sp[0].dst = scratch; sp[1].src = scratch; }
  if (fused) {
    *launches = 1;
    return launch_radon(q, transpose, 2, sp, state_elems, bh, status, st);
  }
  *launches = stages;
  for (int i = 0; i < stages; ++i) {
    const cudaError_t err = sparse_matrix(q)      ? launch_radon_sparse(q, transpose, sp[i], state_elems, bh, status, st)
                            : generates_matrix(q) ? launch_radon_wide(q, transpose, sp[i], state_elems, bh, status, st)
                                                  : launch_radon(q, transpose, 1, &sp[i], state_elems, bh, status, st);
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

int smat_tabulate_d3_wide_supported(const SmatGeo& geo, int64_t state_elems) {
  if (geo.D != 2 || geo.q < 19 || state_elems % 128) return 0;
  StageSpec sp[2];
  radon_stages(geo.q, 2, 0, false, sp);
  return radon_wide_fits(geo.q, sp[0]) ? 1 : 0;
}

cudaError_t smat_launch_tabulate_d3_wide(const void* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                         int* status, cudaStream_t st) {
  StageSpec sp[2];
  radon_stages(geo.q, 2, 0, false, sp);
  sp[0].src = in; sp[0].dst = out;
  return launch_radon_wide(geo.q, 0, sp[0], state_elems, bh, status, st);
}
