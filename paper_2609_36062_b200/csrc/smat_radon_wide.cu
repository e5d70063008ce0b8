// Tabulation stages (see smat_radon_tc.cu for the transform) for primes whose Radon matrix fills more than one MMA tile
// of 128 output indices: q = 13 (182 indices) and, for d = 3, 19 to 53 (380 to 2862).  (q = 17: smat_radon_sparse.cu.)
//
// radon_wide_kernel, persistent, one CTA per SM.  An item is one image restricted to 128 consecutive state entries and
// up to three tiles of outputs, each with an accumulator of 128 columns in tensor memory; the image streams through a
// ring of 64-row slots (MN-major B operand) and every slot is applied to all the tiles before it is released.  So an
// image of q <= 19 is loaded by one CTA once, where the kernel with the matrix resident in tensor memory splits the
// outputs over two or three CTAs that all load it.  The matrix is neither loaded nor kept (3 x 128 x 368 bf16 at q = 19
// would not fit beside anything else): a row of R has one nonzero per input line, (u - a hi) mod q or (lo + a hi) mod q,
// which a bit mask of 64 inputs per row and slot holds (worked out once per launch: 1 KB per tile and slot); a thread per
// output index spreads the mask over 32 columns of the ring of four A tiles that the remaining 128 columns of tensor
// memory hold.  The nonzeros are 2.0, whose bf16 pattern is a single bit (one shift and one mask per register), and the
// sums are halved when they are rounded: both exact.  More than three tiles (q >= 23): the CTAs are shared out over the
// groups of tiles, in proportion to their tiles, and every group walks the images in the same order.
// Bound: q = 13 and 19 by the image and table rows (32 heads of 4096 tokens, 368 MB: 0.069 ms, 0.056 at the HBM rate; 32
// heads of 12288 tokens at q = 19: 0.170 ms, where the sums on the fp32 ALUs took 0.446); q >= 23 by the tensor pipe (75 % active
// at q = 37, whose images the groups read from memory once, 731 MB for a table of 718; two tiles per item and eight A tiles in
// flight instead of three and four: 0.98 ms instead of 0.69): 16 heads, sums on the ALUs / here: q = 23 0.321 / 0.172 ms,
// 29 0.540 / 0.321, 31 0.708 / 0.404, 37 1.053 / 0.690.
//   warps 0-15  : epilogue; lane quarter w % 4, column quarter w / 4 of every accumulator: round to bf16, whole sectors
//   warps 16-27 : generators of R, three groups of four warps that take the (slot, tile) pairs in turn
//   warp 28     : TMA producer;   warps 29-31 : MMA issuers, one per tile
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
constexpr int NE = 128;                   // state entries per item
constexpr int SLOT = 64;                  // operand rows per ring slot = columns of R per A tile
constexpr int B_SLOT = NE * SLOT * 2;     // bytes
constexpr int MAX_BBUF = 12;              // ring slots at most
constexpr int MT = 3;                     // tiles per item at most, and accumulators
constexpr int A_RING = 4;                 // A tiles in tensor memory, 32 columns each
constexpr uint32_t A_COL = MT * NE;       // first column of the A ring
// Barriers of the A tiles.  Pair n of the (slot, tile) sequence lies in ring position n % A_RING, but three issuers and
// three generator groups that go their own pace look at it: a parity wait is only safe for a thread that cannot be a
// whole phase off, so the barriers repeat after A_BARS pairs, more than the image ring (MAX_BBUF slots of MT tiles) lets
// any two of them be apart.
constexpr int A_BARS = 64;
static_assert(A_BARS >= (MAX_BBUF + 1) * MT + 2 * A_RING, "barrier reuse distance");
constexpr int EPI = 16, GEN_GROUPS = 3;   // warps, groups of four warps
constexpr int GEN_WARP = EPI, PROD_WARP = EPI + 4 * GEN_GROUPS, MMA_WARP = PROD_WARP + 1;
constexpr int THREADS = 32 * (MMA_WARP + MT);

struct WideParams {
  int32_t q, transpose;
  uint32_t inv_q;                 // floor(2^32 / q) + 1: x / q = umulhi(x, inv_q) for x < 2^16
  int32_t n_reg;                  // input indices in the regular slots: q*q, or all of them where the extra class follows
  int32_t n_in;                   // all input indices
  int32_t span, nreg, nslots;     // indices per regular slot, regular slots, slots (one more for a separate extra class)
  int32_t flat;                   // slots are 64 consecutive rows; else whole lines
  int32_t tiles, groups;          // output tiles, and the groups of at most MT tiles the CTAs are shared out over
  int32_t bbuf;                   // ring slots
  int32_t slabs_per_head, images;
  uint32_t slabs, items;          // heads * slabs_per_head; slabs * images
  int32_t src_heads;
  int32_t in_vert_from, in_sv_img;
  RadonSide out;
  int64_t rp;
  __nv_bfloat16* dst;
  int* status;
};

// One image's slab.
struct WideItem {
  uint32_t slab, img;
  __device__ __forceinline__ WideItem(const WideParams& p, uint32_t item) {
    img = item / p.slabs;
    slab = p.slabs - 1 - (item - img * p.slabs);   // the last heads first: the kernel before has just written them
  }
};

__device__ __forceinline__ int group_tile(const WideParams& p, int g) { return g * p.tiles / p.groups; }
// The groups' shares of the CTAs: a slot costs about half a tile besides its tiles.
__device__ __forceinline__ int first_cta(const WideParams& p, int g) {
  return (int)gridDim.x * (2 * group_tile(p, g) + g) / (2 * p.tiles + p.groups);
}

// Row `out` of R restricted to the inputs [lo, hi) (at most 64), as two words of 32 inputs: input 32 w + k sits at bit
// (k >> 1) + 16 (k & 1) of word w, so that the bf16 pair of tensor-memory column 16 w + c is bits c and 16 + c.
__device__ __forceinline__ void row_mask(const WideParams& p, int out, int lo, int hi, uint32_t (&w)[2]) {
  const int q = p.q;
  w[0] = w[1] = 0u;
  if (out >= p.out.count) return;
  const int y = (int)__umulhi((uint32_t)out, p.inv_q), x = out - y * q;
  if (!p.transpose && y >= q) {   // extra class: the whole line x
    const int a = max(x * q - lo, 0), b = min(x * q + q, hi) - lo;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int c = min(max(a - 32 * i, 0), 32), d = min(max(b - 32 * i, 0), 32);
      if (d > c) {
        const uint32_t even = ((1u << ((d + 1) >> 1)) - 1) & ~((1u << ((c + 1) >> 1)) - 1);
        const uint32_t odd = ((1u << (d >> 1)) - 1) & ~((1u << (c >> 1)) - 1);
        w[i] = even | (odd << 16);
      }
    }
    return;
  }
  // input line L meets the row at (x - y L) mod q (forward) or (x + y L) mod q (transposed); the extra class of the
  // transposed side (line q) at y
  const int step = p.transpose ? y : (y ? q - y : 0);
  int line = (int)__umulhi((uint32_t)lo, p.inv_q);
  const uint32_t m = (uint32_t)(x + step * line);
  int pos = (int)(m - __umulhi(m, p.inv_q) * (uint32_t)q);
#pragma unroll
  for (int i = 0; i < 6; ++i) {   // 64 inputs touch at most six lines of 13
    const int k = line * q + (line < q ? pos : y) - lo;
    if (k >= 0 && k < hi - lo) {
      const uint32_t bit = 1u << (((k & 31) >> 1) + ((k & 1) << 4));
      if (k < 32) w[0] |= bit; else w[1] |= bit;
    }
    ++line;
    pos += step;
    if (pos >= q) pos -= q;
  }
}

__global__ void __launch_bounds__(THREADS, 1) radon_wide_kernel(const __grid_constant__ CUtensorMap tm_reg,
                                                                const __grid_constant__ CUtensorMap tm_vert,
                                                                const __grid_constant__ WideParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int bbuf = prm.bbuf, nslots = prm.nslots;
  uint8_t* sB = smem;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + bbuf * B_SLOT);
  uint64_t* b_full = bars;                       // [MAX_BBUF]
  uint64_t* b_empty = b_full + MAX_BBUF;         // [MAX_BBUF] one arrival per tile
  uint64_t* a_full = b_empty + MAX_BBUF;         // [A_BARS]
  uint64_t* a_empty = a_full + A_BARS;           // [A_BARS] the pair's MMAs have finished
  uint64_t* d_full = a_empty + A_BARS;           // [MT]
  uint64_t* d_empty = d_full + MT;               // [MT]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(d_empty + MT);
  volatile int* cta_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int32_t* out_tab = reinterpret_cast<int32_t*>(tmem_slot + 2);                  // [MT * 128]
  uint2* masks = reinterpret_cast<uint2*>(out_tab + MT * ROWS);                  // [nslots][nt][128]
  // this CTA's group of tiles, and its share of the items
  int group = 0;
  while (group + 1 < prm.groups && (int)blockIdx.x >= first_cta(prm, group + 1)) ++group;
  const int tile0 = group_tile(prm, group), nt = group_tile(prm, group + 1) - tile0;
  const uint32_t item0 = blockIdx.x - first_cta(prm, group), step = first_cta(prm, group + 1) - first_cta(prm, group);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WaitCtx wc{cta_abort, prm.status};
  if (threadIdx.x == 0) {
    *cta_abort = 0;
    for (int s = 0; s < bbuf; ++s) { mbar_init(b_full + s, 1); mbar_init(b_empty + s, nt); }
    for (int s = 0; s < A_BARS; ++s) { mbar_init(a_full + s, 4); mbar_init(a_empty + s, 1); }
    for (int u = 0; u < MT; ++u) { mbar_init(d_full + u, 1); mbar_init(d_empty + u, EPI); }
    fence_barrier_init();
    prefetch_tmap(&tm_reg);
    prefetch_tmap(&tm_vert);
  }
  if (warp == MMA_WARP) tmem_alloc(tmem_slot, 512);
  if (!prm.flat)   // operand rows no box writes meet zeros of R, but must not hold NaN patterns
    for (int c = threadIdx.x; c < bbuf * B_SLOT / 16; c += THREADS) reinterpret_cast<uint4*>(smem)[c] = make_uint4(0u, 0u, 0u, 0u);
  auto slot_lo = [&](int s) { return s < prm.nreg ? s * prm.span : prm.n_reg; };
  auto slot_hi = [&](int s) { return s < prm.nreg ? min((s + 1) * prm.span, prm.n_reg) : prm.n_in; };
  for (int o = threadIdx.x; o < nt * ROWS; o += THREADS) out_tab[o] = side_row(prm.out, tile0 * ROWS + o, prm.q);
  for (int k = threadIdx.x; k < nslots * nt * ROWS; k += THREADS) {
    const int s = k / (nt * ROWS), o = k - s * nt * ROWS;
    uint32_t w[2];
    row_mask(prm, tile0 * ROWS + o, slot_lo(s), slot_hi(s), w);
    masks[k] = make_uint2(w[0], w[1]);
  }
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  pdl_trigger();   // (after the allocation: a kernel that starts early must not take the tensor memory first)
  const uint32_t tmem_base = *tmem_slot;

  if (warp >= GEN_WARP && warp < PROD_WARP) {
    // ---- generators of R: lane = output index of the tile -----------------------------------------------------------
    const int mine = (warp - GEN_WARP) >> 2, qd = warp & 3;
    const uint32_t my_items = item0 < prm.items ? (prm.items - item0 + step - 1) / step : 0;
    const uint32_t pairs = (uint32_t)(nslots * nt);              // of one item, in the order (slot, tile)
    const uint32_t total = my_items * pairs;
    const uint2* mrow = masks + qd * 32 + lane;
    uint32_t k = mine;                                           // pair inside its item
    while (k >= pairs) k -= pairs;
    for (uint32_t n = mine; n < total; n += GEN_GROUPS) {
      const uint2 w = mrow[k * ROWS];
      k += GEN_GROUPS;
      while (k >= pairs) k -= pairs;
      uint32_t v[32];
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        v[c] = (c <= 14 ? w.x << (14 - c) : w.x >> 1) & 0x40004000u;
        v[16 + c] = (c <= 14 ? w.y << (14 - c) : w.y >> 1) & 0x40004000u;
      }
      const uint32_t was = n - A_RING;
      if (n >= A_RING) {   // (the first tiles of R are made while the kernel before runs on)
        if (n < A_RING + GEN_GROUPS) pdl_wait();
        if (!mbar_wait_warp(a_empty + (was & (A_BARS - 1)), (was / A_BARS) & 1, wc)) break;
      }
      fence_after_sync();
      tmem_st32(tmem_base + ((uint32_t)(qd * 32) << 16) + A_COL + (n & (A_RING - 1)) * 32, v);
      tmem_st_wait();
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full + (n & (A_BARS - 1)));
    }
  } else if (warp == PROD_WARP) {
    // ---- TMA producer (the whole warp walks the loop, one lane issues: as for the MMAs below) -------------------------
    pdl_wait();
    const bool leader = elect_one();
    uint32_t slot = 0, par = 1;                                  // par: parity that a fresh b_empty barrier passes
    bool ok = true;
    const uint32_t reg_bytes = (uint32_t)((prm.flat ? SLOT : prm.span) * 2 * NE), vert_bytes = (uint32_t)(prm.q * 2 * NE);
    const int lines = prm.span / prm.q;
    for (uint32_t item = item0; item < prm.items && ok; item += step) {
      const WideItem it(prm, item);
      const uint32_t head = it.slab / (uint32_t)prm.slabs_per_head;
      const int eb = (int)(it.slab - head * prm.slabs_per_head) * (NE / 64);   // first 64-entry block
      const int vhead = (int)it.img >= prm.in_vert_from ? (int)head : prm.src_heads;
      for (int s = 0; s < nslots; ++s) {
        if (!mbar_try_wait(b_empty + slot, par)) ok = mbar_wait(b_empty + slot, par, wc);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (leader) {
          uint8_t* dst = sB + slot * B_SLOT;
          uint64_t* bar = b_full + slot;
          if (prm.flat) {         // both 64-entry halves in one box; rows past the image's end arrive as zeros
            mbar_expect_tx(bar, reg_bytes);
            tma_load_5d(dst, &tm_reg, 0, s * SLOT, eb, (int)it.img, (int)head, bar);
          } else if (s < prm.nreg) {
            mbar_expect_tx(bar, reg_bytes);
            tma_load_5d(dst, &tm_reg, eb * 64, 0, s * lines, (int)it.img, (int)head, bar);
            tma_load_5d(dst + SLOT * 128, &tm_reg, eb * 64 + 64, 0, s * lines, (int)it.img, (int)head, bar);
          } else {                // extra class; an image without it reads past the last head: zeros
            mbar_expect_tx(bar, vert_bytes);
            tma_load_4d(dst, &tm_vert, eb * 64, 0, (int)it.img * prm.in_sv_img, vhead, bar);
            tma_load_4d(dst + SLOT * 128, &tm_vert, eb * 64 + 64, 0, (int)it.img * prm.in_sv_img, vhead, bar);
          }
        }
        if (++slot == (uint32_t)bbuf) { slot = 0; par ^= 1; }
      }
    }
    if (leader) ring_landed(b_full, (uint32_t)bbuf, slot, par, wc);
  } else if (warp >= MMA_WARP) {
    // ---- MMA issuers: one warp per tile of the group (its waits, MMAs and commits take longer than the tensor pipe
    // needs for a tile's share of a slot, so one thread for all three tiles would hold the pipe up).  The whole warp
    // walks the loop, so that addresses and descriptors stay in uniform registers; one elected lane issues. ------------
    pdl_wait();
    const int t = warp - MMA_WARP;
    if (t < nt) {
      constexpr uint32_t idesc = make_idesc(ROWS, NE, 0, 1);    // R from tensor memory, image rows MN-major
      const uint64_t dB0 = make_desc(smem_u32(sB), SLOT * 128, 1024);
      const int last_steps = (slot_hi(nslots - 1) - slot_lo(nslots - 1) + 15) >> 4;
      const int reg_steps = (prm.span + 15) >> 4, end_steps = (prm.n_reg - (prm.nreg - 1) * prm.span + 15) >> 4;
      const bool leader = elect_one();
      uint32_t slot = 0, par = 0, n = t;
      uint32_t u = t, up = 1;                                    // up: parity that a fresh d_empty barrier passes
      bool ok = true;
      for (uint32_t item = item0; item < prm.items && ok; item += step) {
        const uint32_t d = tmem_base + u * NE;
        ok = __all_sync(0xffffffffu, mbar_wait(d_empty + u, up, wc));   // an earlier item's sums have been read out
        for (int s = 0; s < nslots && ok; ++s, n += (uint32_t)nt) {
          const uint32_t bar = n & (A_BARS - 1), apar = (n / A_BARS) & 1;
          bool rb = mbar_try_wait(b_full + slot, par), ra = mbar_try_wait(a_full + bar, apar);
          if (!__all_sync(0xffffffffu, rb && ra)) {
            rb = mbar_wait(b_full + slot, par, wc) && mbar_wait(a_full + bar, apar, wc);
            ok = __all_sync(0xffffffffu, rb);
            if (!ok) break;
          }
          fence_after_sync();
          const uint64_t dB = dB0 + (uint64_t)(slot * (B_SLOT >> 4));
          const uint32_t a = tmem_base + A_COL + (n & (A_RING - 1)) * 32;
          const int steps = s + 1 == nslots ? last_steps : (s + 1 == prm.nreg ? end_steps : reg_steps);
          if (leader) {
            if (steps == 4) {
              mma_bf16_ta(d, a, dB, idesc, s != 0);
#pragma unroll
              for (int kk = 1; kk < 4; ++kk) mma_bf16_ta(d, a + 8 * kk, dB + 128 * kk, idesc, 1);
            } else {
              for (int kk = 0; kk < steps; ++kk) mma_bf16_ta(d, a + 8 * kk, dB + 128 * kk, idesc, (s | kk) != 0);
            }
            mma_commit(a_empty + bar);
            mma_commit(b_empty + slot);
            if (s + 1 == nslots) mma_commit(d_full + u);
          }
          if (++slot == (uint32_t)bbuf) { slot = 0; par ^= 1; }
        }
        u += (uint32_t)nt;
        if (u >= MT) { u -= MT; up ^= 1; }
      }
    }
  } else if (warp < EPI) {
    // ---- epilogue -------------------------------------------------------------------------------------------------
    pdl_wait();
    const int qd = warp & 3, cb = warp >> 2;
    const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
    uint32_t unit = 0, par = 0;
    bool ok = true;
    for (uint32_t item = item0; item < prm.items && ok; item += step) {
      const WideItem it(prm, item);
      const uint32_t head = it.slab / (uint32_t)prm.slabs_per_head;
      const int e0 = (int)(it.slab - head * prm.slabs_per_head) * NE;
      __nv_bfloat16* base = prm.dst + (int64_t)head * prm.out.rows_per_head * prm.rp + e0 + cb * 32;
      const bool vert = (int)it.img >= prm.out.vert_from;
      for (int t = 0; t < nt; ++t) {
        const int tv = out_tab[t * ROWS + qd * 32 + lane];
        ok = mbar_wait_warp(d_full + unit, par, wc);
        if (!ok) break;
        fence_after_sync();
        if ((tile0 + t) * ROWS + qd * 32 < prm.out.count) {   // warp-uniform: some output index in these lanes
          const int row = (tv & ROW_VERT) ? prm.out.v0 + (int)it.img * prm.out.sv_img + (tv & ~ROW_VERT)
                                          : (int)it.img * prm.out.s_img + tv;
          uint32_t v[32];
          tmem_ld32(tmem_base + lane_base + unit * NE + cb * 32, v);
          tmem_ld_wait();
          fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(d_empty + unit);            // the accumulator is in registers
          if (tv != ROW_INVALID && (!(tv & ROW_VERT) || vert)) {
            __nv_bfloat16* dst = base + (int64_t)row * prm.rp;
#pragma unroll
            for (int h8 = 0; h8 < 2; ++h8) {                     // whole 32-byte sectors; R's nonzeros were 2
              uint32_t o[8];
#pragma unroll
              for (int i = 0; i < 8; ++i)
                o[i] = pack_bf16(0.5f * __uint_as_float(v[16 * h8 + 2 * i]), 0.5f * __uint_as_float(v[16 * h8 + 2 * i + 1]));
              st_global_v8(dst + 16 * h8, o[0], o[1], o[2], o[3], o[4], o[5], o[6], o[7]);
            }
          }
        } else if (lane == 0) {
          mbar_arrive(d_empty + unit);
        }
        if (++unit == MT) { unit = 0; par ^= 1; }
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

}  // namespace

// Shared memory besides the image ring.
static int wide_fixed_smem(int nslots, int tiles) {
  const int groups = (tiles + MT - 1) / MT, widest = (tiles + groups - 1) / groups;
  return 1024 + MT * ROWS * 4 + (2 * MAX_BBUF + 2 * A_BARS + 2 * MT) * 8 + 16 + nslots * widest * ROWS * 8;
}
static int wide_ring(int nslots, int tiles) {
  const int ring = (227 * 1024 - wide_fixed_smem(nslots, tiles)) / B_SLOT;
  return ring > MAX_BBUF ? MAX_BBUF : ring;
}

namespace {

// How a stage's image is cut into ring slots and its outputs into tiles.
struct WideShape {
  bool flat;                      // slots of 64 consecutive rows; else whole lines
  int lines, span, n_reg;         // lines and indices per regular slot, input indices in regular slots
  int nreg, nslots, tiles, groups, ring, smem;
};

bool wide_shape(int q, const StageSpec& sp, WideShape* w) {
  const RadonSide& in = sp.in;
  const int qq = q * q;
  if (q < 13) return false;
  const bool extra = in.count > qq;
  const bool merged = extra && in.v0 == qq && in.sv_lo == 1 && in.vert_from == 0 && sp.images == 1;   // rows follow on
  w->flat = in.s_lo == 1 && in.s_hi == q && (!extra || merged);
  if (!w->flat && q > SLOT) return false;
  w->lines = w->flat ? 1 : SLOT / q;
  w->n_reg = w->flat ? in.count : qq;
  w->span = w->flat ? SLOT : w->lines * q;
  w->nreg = (w->n_reg + w->span - 1) / w->span;
  w->nslots = w->nreg + (in.count > w->n_reg ? 1 : 0);
  w->tiles = (sp.out.count + ROWS - 1) / ROWS;
  w->groups = (w->tiles + MT - 1) / MT;
  w->ring = wide_ring(w->nslots, w->tiles);
  w->smem = wide_fixed_smem(w->nslots, w->tiles) + w->ring * B_SLOT;
  return w->ring >= 4;
}

// The shared-memory map of radon_wide_kernel for a shape, checked on the host before every launch: what follows the ring
// must end inside the allocation, no box may write past its slot, and a slot's inputs must fit the masks.
//   [0, ring * B_SLOT)                                      ring slots: two halves of SLOT rows x 128 bytes
//   [.., + (2 MAX_BBUF + 2 A_BARS + 2 MT) * 8 + 8)          barriers, the tensor-memory slot word, the abort flag
//   [.., + MT * ROWS * 4)                                   output-row table
//   [.., + nslots * widest * ROWS * 8)                      masks of the widest group's tiles
bool wide_layout_ok(int q, const StageSpec& sp, const WideShape& w) {
  const int widest = (w.tiles + w.groups - 1) / w.groups, qq = q * q;
  bool ok = widest <= MT && w.ring >= 1 && w.ring <= MAX_BBUF && B_SLOT == 2 * SLOT * 128 && B_SLOT % 1024 == 0;
  ok = ok && w.span <= SLOT && w.nreg * w.span >= w.n_reg && (w.flat || (w.lines * q == w.span && w.n_reg == qq));
  ok = ok && (w.nslots == w.nreg || (w.nslots == w.nreg + 1 && sp.in.count == qq + q && q <= SLOT));   // the extra class
  ok = ok && (SLOT + q - 2) / q + 1 <= 6;                                                // lines a slot touches (row_mask)
  ok = ok && w.tiles * ROWS >= sp.out.count && qq + q < (1 << 16);                       // index arithmetic by umulhi
  const int end = w.ring * B_SLOT + (2 * MAX_BBUF + 2 * A_BARS + 2 * MT) * 8 + 8 + MT * ROWS * 4 + w.nslots * widest * ROWS * 8;
  return ok && 1023 + end <= w.smem && w.smem <= 227 * 1024;
}

}  // namespace

bool radon_wide_layout_ok(int q, const StageSpec& sp) {
  WideShape w;
  return wide_shape(q, sp, &w) && wide_layout_ok(q, sp, w);
}

bool radon_wide_fits(int q, const StageSpec& sp) {
  WideShape w;
  return wide_shape(q, sp, &w);
}

cudaError_t launch_radon_wide(int q, int transpose, const StageSpec& sp, int64_t rp, int bh, int* status, cudaStream_t st) {
  const RadonSide& in = sp.in;
  WideShape w;
  if (!wide_shape(q, sp, &w) || rp % NE) return cudaErrorInvalidValue;
  if (!wide_layout_ok(q, sp, w)) return cudaErrorInvalidConfiguration;
  WideParams prm;
  prm.q = q; prm.transpose = transpose;
  prm.inv_q = (uint32_t)((1ULL << 32) / (uint32_t)q) + 1;
  prm.n_in = in.count;
  prm.flat = w.flat; prm.n_reg = w.n_reg; prm.span = w.span; prm.nreg = w.nreg; prm.nslots = w.nslots;
  prm.tiles = w.tiles; prm.groups = w.groups; prm.bbuf = w.ring;
  prm.images = sp.images;
  prm.src_heads = bh;
  prm.in_vert_from = in.vert_from;
  prm.in_sv_img = in.sv_img != 0 ? 1 : 0;
  prm.out = sp.out; prm.rp = rp;
  prm.dst = static_cast<__nv_bfloat16*>(sp.dst);
  prm.status = status;
  prm.slabs_per_head = (int)(rp / NE);
  prm.slabs = (uint32_t)bh * (uint32_t)prm.slabs_per_head;
  const int64_t items = (int64_t)prm.slabs * prm.images;
  if (items * prm.nslots * MT >= (1LL << 31)) return cudaErrorInvalidValue;   // pairs are counted in 32 bits
  prm.items = (uint32_t)items;
  CUtensorMap tm_reg, tm_vert;
  const int64_t s_img = sp.images > 1 ? in.s_img : in.rows_per_head;   // a size-one dimension keeps its stride valid
  if (prm.flat) {   // (entry of a 64-entry block, row, block, image, head)
    const int64_t sizes[5] = {64, prm.n_reg, rp / 64, sp.images, bh};
    const int64_t strides[4] = {rp, 64, s_img * rp, in.rows_per_head * rp};
    const int box[5] = {64, SLOT, NE / 64, 1, 1};
    if (!radon_map_elems(&tm_reg, sp.src, 5, sizes, strides, box)) return cudaErrorInvalidValue;
  } else {          // (entry, lo, hi, image, head)
    const int64_t sizes[4] = {q, q, sp.images, bh};
    const int64_t strides[4] = {in.s_lo, in.s_hi, s_img, in.rows_per_head};
    const int box[4] = {q, w.lines, 1, 1};
    if (!radon_map(&tm_reg, sp.src, rp, 5, sizes, strides, box)) return cudaErrorInvalidValue;
  }
  tm_vert = tm_reg;
  if (prm.n_in > prm.n_reg) {
    const bool per_image = in.sv_img != 0;
    const int64_t sizes[3] = {q, per_image ? sp.images : 1, bh};
    const int64_t strides[3] = {in.sv_lo, per_image ? in.sv_img : in.rows_per_head, in.rows_per_head};
    const int box[3] = {q, 1, 1};
    if (!radon_map(&tm_vert, static_cast<const __nv_bfloat16*>(sp.src) + (int64_t)in.v0 * rp, rp, 4, sizes, strides, box))
      return cudaErrorInvalidValue;
  }
  cudaError_t err = cudaFuncSetAttribute(radon_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, w.smem);
  if (err != cudaSuccess) return err;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t grid = items * prm.groups < sms ? items * prm.groups : sms;
  // Every group of tiles needs a CTA (see first_cta); none waits for another, so that a device with fewer SMs, a slice of
  // one among them, runs them one after the other.
  if (grid < 2 * prm.tiles + prm.groups) grid = 2 * prm.tiles + prm.groups;
  return smat_launch_pdl(radon_wide_kernel, dim3((unsigned)grid), THREADS, w.smem, st, tm_reg, tm_vert, prm);
}
