// Long-range rows without tables.  What a routed read takes from the type table is
//     x_t · U_h = x_t · Σ_{s in the cells of hyperplane h} y_s z_sᵀ = Σ_s (x_t · y_s) z_s,
// and where a type's tokens are few and the keys that they see are few as well, the right-hand side moves less than the tables
// do: a warp gathers the rows of one type's tokens (X) and, 16 at a time, those of the tokens of its cells (Y, Z), forms the
// 16 x 16 scores and multiplies them into the outputs.  The same with the roles exchanged gives dK and dV: the rows of a cell's
// tokens against the tokens of all types through the cell, both products from one gather (DUAL).  The rows come from the L2
// cache, which holds a head's K and V many times over, and nothing but the outputs goes back to memory.
//
// Scores are rounded to bf16 once, as the causal tiles' are; tables are rounded once for F and once or three times for U.  In the
// ungated forward and dQ of d = 2 (one table, rounded once) they enter as a leading part and a remainder, 16 bits, and where
// the plan's tables would be fp32 (partial tiles, forward only) in three parts, which hold all 24 bits.  The rows' error against fp64 there, in the
// 2-norm: 1.1e-7 from fp32 tables, 3e-7 to 1.2e-6 with three parts (the matrix instructions' sums), 2.5e-6 with two; of the
// outputs, rounded to bf16, 1.660e-3 each way.
//
// The matrix instructions are those of a warp (m16n8k16): from d = 3 on a type has 3 to 31 rows, which fill a tile or two of 16
// and would leave most of a 128-row one of tcgen05 empty, and at 545 TFLOP/s measured they are not what the kernel waits for.  (At d = 2
// a type has 17 to 128 rows and would fill such a tile; there the same kernel takes them in blocks of 32, each of which gathers
// the keys again, and the rule below counts that.)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_tc.cuh"

namespace {

using namespace tc;

constexpr int LN_STEP = 16;                                  // gathered rows per step
constexpr int LN_STAGES = 2, LN_STAGE = 2 * LN_STEP * 256;   // stages of the ring (line_products_kernel counts on two), their bytes

struct LineParams {
  const __nv_bfloat16 *x1, *x2, *y, *z;   // [bh][T][128]
  void *out1, *out2;                      // rows like X, bf16 or fp32
  __nv_bfloat16* copy;                    // the distant rows, for the tables' export: K then V of a token (null: not wanted)
  int64_t copy_head;                      // tokens between heads there
  int copy_swap;                          // Y holds V and Z holds K
  int* mark;                              // word that says what the workspace holds (null: not wanted)
  int mark_value;
  int* clear;                             // status word of a pass that begins with this launch, which waits for nothing that could fail
  const float* lam;                       // gated: prefix sums of the log-gates [bh][T]
  int64_t T;
  uint32_t n, m, P, B, q, D;
  uint32_t key_first, key_count, key_period;   // the gathered block: its first token, its tokens, the period of its groups
  uint32_t qpow[SMAT_MAX_DIM + 1], dir_start[SMAT_MAX_DIM];
  uint32_t q_inv, lines_inv, per_inv;     // of q, lines, groups x blocks:             
                                          // ceil(2^32 / .): quotients by umulhi, exact while dividend x divisor < 2^32
  uint32_t groups, blocks, lines, slots, steps;   // row groups of a head, row blocks of a group, gathered groups of a group
  uint32_t full_steps;                            // steps before the first that has a slot without a token
  uint32_t items;
  int rows_are_types, out_f32, ones;
};

__device__ __forceinline__ uint32_t div_q(const LineParams& p, uint32_t v) { return __umulhi(v, p.q_inv); }
__device__ __forceinline__ uint32_t mod_q(const LineParams& p, uint32_t v) { return v - __umulhi(v, p.q_inv) * p.q; }

// Direction number `dir`: its coordinates after the leading one, as a little-endian number; lead: where the leading one stands.
__device__ __forceinline__ uint32_t direction(const LineParams& p, uint32_t dir, int& lead) {
  lead = 0;
  while (lead + 1 < (int)p.D && dir >= p.dir_start[lead + 1]) ++lead;
  return dir - p.dir_start[lead];
}
// The gathered groups of a row group, for D <= 2: the i-th one is ((c0 + c1 i) mod q) m0 + i m1, but where i == odd one out of
// the pattern.  Cells of hyperplane (1, a | b): x2 = i, x1 = b - a i; of (0, 1 | b): x2 = b, x1 = i.  Types through cell (x1, x2):
// i q + (x1 + i x2), and the last direction's q q + x2.
struct LineOf {
  uint32_t g, c0, c1, m0, m1;
};
__device__ __forceinline__ LineOf line_of(const LineParams& p, uint32_t g) {
  LineOf l;
  l.g = g;
  const uint32_t hi = div_q(p, g), lo = g - hi * p.q;
  l.c0 = lo; l.c1 = 0; l.m0 = 1; l.m1 = p.q;
  if (p.D == 2) {
    if (!p.rows_are_types) {
      l.c1 = hi;
    } else if (hi < p.q) {
      l.c1 = hi ? p.q - hi : 0;
    } else {
      l.m0 = p.q;
      l.m1 = 1;
    }
  }
  return l;
}
// Slot e of row group l.g.  Slots go over the gathered groups first, then over their tokens; one that has none is given the
// first token of its group (every group has one) and is not `there`.
struct Slot {
  uint32_t t;
  bool there;
};
__device__ __forceinline__ Slot slot_token(const LineParams& p, const LineOf& l, uint32_t e) {
  const uint32_t j = p.lines == 1 ? e : __umulhi(e, p.lines_inv);
  uint32_t i = e - j * p.lines, first;
  if (p.D <= 2) {
    uint32_t x = mod_q(p, l.c0 + l.c1 * i);
    if (p.rows_are_types) {
      first = x * l.m0 + i * l.m1;
    } else {
      if (i == p.q) x = l.c1;
      const uint32_t h = i * p.q + x;
      first = (h ? h : p.B) - 1;
    }
  } else if (p.rows_are_types) {   // cell i of hyperplane g: its coordinates but one are free
    int lead;
    const uint32_t dir = div_q(p, l.g), b = l.g - dir * p.q;
    uint32_t tail = direction(p, dir, lead), acc = 0, cell = 0;
    for (int k = 0; k < (int)p.D; ++k) {
      if (k == lead) continue;
      const uint32_t hi = div_q(p, i), x = i - hi * p.q;
      i = hi;
      cell += x * p.qpow[k];
      if (k > lead) {
        const uint32_t th = div_q(p, tail);
        acc = mod_q(p, acc + (tail - th * p.q) * x);
        tail = th;
      }
    }
    first = cell + (b >= acc ? b - acc : b + p.q - acc) * p.qpow[lead];
  } else {   // type of direction i through cell g
    int lead;
    uint32_t tail = direction(p, i, lead), acc = 0, v = l.g;
    for (int k = 0; k < (int)p.D; ++k) {
      const uint32_t hi = div_q(p, v), x = v - hi * p.q;
      v = hi;
      if (k == lead) acc += x;
      if (k > lead) {
        const uint32_t th = div_q(p, tail);
        acc = mod_q(p, acc + (tail - th * p.q) * x);
        tail = th;
      }
    }
    const uint32_t h = i * p.q + mod_q(p, acc);
    first = (h ? h : p.B) - 1;
  }
  const uint32_t at = first + j * p.key_period;
  Slot s;
  s.there = e < p.slots && at < p.key_count;
  s.t = p.key_first + (s.there ? at : first);
  return s;
}
// Row r of row group g: the token, or -1.
__device__ __forceinline__ int row_token(const LineParams& p, uint32_t g, uint32_t r) {
  if (p.rows_are_types) {
    const uint32_t at = (g ? g : p.B) - 1 + r * p.B;
    return at < p.m ? (int)(p.n + at) : -1;
  }
  const uint32_t t = g + r * p.P;
  return t < p.n ? (int)t : -1;
}

__device__ __forceinline__ void lds16(uint32_t addr, uint32_t* w) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_trans(uint32_t addr, uint32_t (&w)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma16816_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// 16-byte piece c of row r in a tile of 256-byte rows: pieces 2 q of rows 2 k and 2 k + 1 lie in different bank groups, and so do
// piece c of rows 0 to 7.  (Rows 272 bytes apart need no exclusive or, but a sector then lands across two: 70 us where this takes 60.)
__device__ __forceinline__ uint32_t piece(uint32_t r, uint32_t c) { return r * 256 + ((c ^ (r & 7)) << 4); }

template <int RT, bool DUAL>
struct LineSmem {
  static constexpr bool x_regs = RT * (1 + DUAL) == 1;
  static constexpr int warps_per_sm = x_regs ? 12 : 8;
  static constexpr int x_bytes = x_regs ? 0 : RT * (1 + DUAL) * 4096, bytes = LN_STAGES * LN_STAGE + x_bytes;
};

// A CTA is one warp (what is the same for all of it stays in uniform registers; with two to a CTA 3 to 5 % more) and takes an item (16 RT
// rows of a row group) from beginning to end, with a ring of its own in shared memory: no barriers.
// Stages of the ring: X of an item, then 16 gathered rows of Y and Z after the other.  Lane (g, q) = (lane / 4, lane % 4) of the
// matrix instructions:
//   scores   its words of a row are bytes 32 q to 32 q + 31 of either half: the order of the contracted index is free, as
//            long as X and Y have the same
//   outputs  the rows of Z transposed on the way from shared memory (ldmatrix)
// Bound by the instructions that a warp issues for a stage, about 290 one after the other at 12 warps to an SM (8 where a thread's
// accumulators are 128), not by the gather: 7 to 12 TB/s, where row loads alone reach 16.  Three tables' kernels / this one, us:
// d = 3, 32 heads of 2048 tokens 137 / 33, of 4096 163 / 57, 128 heads of 8192 917 / 410, 16 heads of 16 K 312 / 147, of 24 K
// 529 / 255; d = 4, 32 heads of 4096 552 / 190; fp32 tables (scores in three parts: about 370 instructions, with two 89 and 36 us): d = 3,
// 32 heads of 5056 503 / 105; d = 2, 32 of 4160 238 / 38.
// The first form, four warps to an item with the scores exchanged through shared memory, took 156 where this takes 57; with a
// test for every kind of stage in front of each and all of Z in registers (spills) it was 77.
template <int RT, bool DUAL, bool GATED, int PARTS>
__global__ void __launch_bounds__(32, LineSmem<RT, DUAL>::warps_per_sm)
line_products_kernel(const __grid_constant__ LineParams p) {
  using L = LineSmem<RT, DUAL>;
  constexpr int NX = 1 + DUAL;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t lane = threadIdx.x, g = lane >> 2, q = lane & 3;
  const uint32_t ring = smem_u32(smem), xs = ring + LN_STAGES * LN_STAGE + lane * 16;
  const uint32_t crow = lane >> 4, cpiece = lane & 15;   // pieces that a lane copies: rows crow + 2 i

  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (p.mark) *p.mark = p.mark_value;
    if (p.clear) *p.clear = 0;
  }
  uint32_t it = blockIdx.x;

  struct Item {
    uint32_t g, rb, bh;
  };
  auto item_at = [&](uint32_t i) {
    Item a;
    a.bh = __umulhi(i, p.per_inv);
    const uint32_t in = i - a.bh * p.groups * p.blocks;
    a.g = p.blocks == 1 ? in : in / p.blocks;
    a.rb = in - a.g * p.blocks;
    return a;
  };
  auto factor = [&](uint32_t bh, int t) -> float {   // decay between a token and the block boundary
    const float* l = p.lam + (int64_t)bh * p.T;
    const float edge = l[p.n - 1];
    return t < (int)p.n ? expf(edge - l[t]) : expf(l[t] - edge);
  };

  // The loads, two stages ahead of the products: of item `la`, X or a step's 16 slots, into slot lslot of the ring.
  uint32_t lslot = 0;
  Item la = item_at(it);
  LineOf line = line_of(p, la.g);
  bool more = true;       // there is such an item
  Slot ntok{0, false};    // the lane's slot of the 32 that are being loaded
  float nfac = 0.f;
  uint32_t to[4];         // where the pieces of rows crow + 2 i go, i mod 4
#pragma unroll
  for (int i = 0; i < 4; ++i) to[i] = ring + piece(crow + 2 * i, cpiece);
  int64_t head = (int64_t)la.bh * p.T * 128 + cpiece * 8;
  const __nv_bfloat16 *ly = p.y + head, *lz = p.z + head;
  auto load_rows = [&]() {
    if (more) {
      const __nv_bfloat16 *lx = p.x1 + head, *lx2 = DUAL ? p.x2 + head : nullptr;
      int mine = row_token(p, la.g, la.rb * (RT * 16) + lane);
      if (mine < 0) mine = row_token(p, la.g, 0);   // (what comes of it is not stored)
#pragma unroll
      for (int i = 0; i < RT * 8; ++i) {
        const uint32_t t = __shfl_sync(0xffffffffu, mine, crow + 2 * i), dst = to[i & 3] + lslot * LN_STAGE + (i >> 2) * 2048;
        cp_async16(dst, lx + (uint64_t)t * 128);
        if (DUAL) cp_async16(dst + 4096, lx2 + (uint64_t)t * 128);
      }
    }
    cp_async_commit();
    lslot ^= 1;
  };
  auto load_keys = [&](uint32_t step) {
    if (!(step & 1)) {
      ntok = slot_token(p, line, step * LN_STEP + lane);
      if (GATED) nfac = ntok.there ? factor(la.bh, (int)ntok.t) : 0.f;
    }
    const uint32_t from = crow + (step & 1) * 16, stage = lslot * LN_STAGE;
#pragma unroll
    for (int i = 0; i < LN_STEP / 2; ++i) {
      const uint32_t t = __shfl_sync(0xffffffffu, ntok.t, from + 2 * i), dst = to[i & 3] + stage + (i >> 2) * 2048;
      cp_async16(dst, ly + (uint64_t)t * 128);
      cp_async16(dst + 4096, lz + (uint64_t)t * 128);
    }
    cp_async_commit();
    lslot ^= 1;
  };
  // The stage behind step `step` of an item of p.steps: a step of the same one, X of the next one, or that one's first step.
  auto load_behind = [&](uint32_t step) {
    if (step < p.steps) {
      load_keys(step);
    } else if (step == p.steps) {
      const uint32_t i = p.groups * p.blocks * la.bh + la.g * p.blocks + la.rb + gridDim.x;
      more = i < p.items;
      if (more) {
        la = item_at(i);
        line = line_of(p, la.g);
        head = (int64_t)la.bh * p.T * 128 + cpiece * 8;
        ly = p.y + head;
        lz = p.z + head;
      }
      load_rows();
    } else if (more) {
      load_keys(0);
    } else {
      cp_async_commit();
      lslot ^= 1;
    }
  };
  load_rows();
  load_keys(0);

  uint32_t slot = 0;
  // this lane's words for the scores of row g (two pieces in either half), and its row of the transposed tiles
  const uint32_t s_at[2] = {ring + piece(g, 2 * q), ring + piece(g, 2 * q + 1)}, o_at = ring + piece(lane & 15, lane >> 4);
  auto lds_scores = [&](uint32_t off, uint32_t i, uint32_t (&w)[4]) {   // 16-byte group i of the row at off
    lds16(s_at[i & 1] + off + (i >> 1) * 128, w);
  };
  while (true) {
    const Item cur = la;
    uint32_t xf[L::x_regs ? 2 : 1][16];
    cp_async_wait<LN_STAGES - 1>();
    __syncwarp();
    {
      const uint32_t tile = slot * LN_STAGE;
#pragma unroll
      for (int o = 0; o < NX * RT; ++o)   // 16 rows
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t w[4];
            lds_scores(tile + o * 4096 + hf * 2048, i, w);
            if (L::x_regs) {
#pragma unroll
              for (int k = 0; k < 4; ++k) xf[L::x_regs ? hf : 0][4 * i + k] = w[k];
            } else {
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(xs + ((o * 2 + hf) * 4 + i) * 512), "r"(w[0]), "r"(w[1]),
                           "r"(w[2]), "r"(w[3]) : "memory");
            }
          }
      __syncwarp();
      load_behind(1);
      slot ^= 1;
    }
    float acc[NX][RT][16][4];
#pragma unroll
    for (int o = 0; o < NX; ++o)
#pragma unroll
      for (int rt = 0; rt < RT; ++rt)
#pragma unroll
        for (int nt = 0; nt < 16; ++nt)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[o][rt][nt][v] = 0.f;
    Slot tok{0, false};
    float fac = 0.f;
    const bool copies = p.copy && cur.g < p.q && cur.rb == 0;   // the q hyperplanes of one direction hold every distant token once
#pragma unroll 1
    for (uint32_t s = 0; s < p.steps; ++s) {
      const uint32_t tile = slot * LN_STAGE, half = (s & 1) * 16;
      if (!(s & 1)) { tok = ntok; fac = nfac; }
      cp_async_wait<LN_STAGES - 1>();
      __syncwarp();
      uint32_t pp[PARTS][NX][RT][4];   // the scores, in bf16 parts
#pragma unroll
      for (int o = 0; o < NX; ++o) {
        float sc[RT][2][4], sd[RT][2][4];   // two sums each: a chain of products is as long as their latencies
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t y[2][4];
#pragma unroll
          for (int nt = 0; nt < 2; ++nt) lds_scores(tile + o * 4096 + nt * 2048, i, y[nt]);
#pragma unroll
          for (int rt = 0; rt < RT; ++rt) {
            uint32_t lo[4], hi[4];
            if (L::x_regs) {
#pragma unroll
              for (int k = 0; k < 4; ++k) { lo[k] = xf[0][4 * i + k]; hi[k] = xf[L::x_regs ? 1 : 0][4 * i + k]; }
            } else {
              lds16(xs + (((o * RT + rt) * 2) * 4 + i) * 512, lo);
              lds16(xs + (((o * RT + rt) * 2 + 1) * 4 + i) * 512, hi);
            }
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
              if (i == 0) {
                mma16816_first(sc[rt][nt], lo[0], hi[0], lo[1], hi[1], y[nt][0], y[nt][1]);
                mma16816_first(sd[rt][nt], lo[2], hi[2], lo[3], hi[3], y[nt][2], y[nt][3]);
              } else {
                mma16816(sc[rt][nt], lo[0], hi[0], lo[1], hi[1], y[nt][0], y[nt][1]);
                mma16816(sd[rt][nt], lo[2], hi[2], lo[3], hi[3], y[nt][2], y[nt][3]);
              }
            }
          }
        }
        if (!GATED && s >= p.full_steps) {   // slots without a token
          const unsigned there = __ballot_sync(0xffffffffu, tok.there) >> (half + 2 * q);
#pragma unroll
          for (int v = 0; v < 8; ++v)   // n-tile v / 4, register v % 4
            if (!(there >> ((v >> 2) * 8 + (v & 1)) & 1))
#pragma unroll
              for (int rt = 0; rt < RT; ++rt) sc[rt][v >> 2][v & 3] = sd[rt][v >> 2][v & 3] = 0.f;
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          float f0 = 1.f, f1 = 1.f;
          if (GATED) {
            f0 = __shfl_sync(0xffffffffu, fac, half + nt * 8 + 2 * q);
            f1 = __shfl_sync(0xffffffffu, fac, half + nt * 8 + 2 * q + 1);
          }
#pragma unroll
          for (int rt = 0; rt < RT; ++rt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              float v0 = sc[rt][nt][2 * hf] + sd[rt][nt][2 * hf], v1 = sc[rt][nt][2 * hf + 1] + sd[rt][nt][2 * hf + 1];
              if (GATED) { v0 *= f0; v1 *= f1; }
#pragma unroll
              for (int part = 0; part < PARTS; ++part) {   // (a remainder is exact)
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(v0, v1);
                pp[part][o][rt][2 * nt + hf] = *reinterpret_cast<const uint32_t*>(&h2);
                if (part + 1 < PARTS) {
                  const float2 h = __bfloat1622float2(h2);
                  v0 -= h.x;
                  v1 -= h.y;
                }
              }
            }
        }
      }
      if (copies) {
#pragma unroll 1
        for (int i = 0; i < LN_STEP / 2; ++i) {
          const uint32_t r = crow + 2 * i;
          const uint32_t t = __shfl_sync(0xffffffffu, tok.t, half + r);
          if (__shfl_sync(0xffffffffu, (int)tok.there, half + r)) {   // (the halves of the warp copy different rows)
            uint32_t w[4];
            uint4* dst = reinterpret_cast<uint4*>(p.copy + ((int64_t)cur.bh * p.copy_head + t) * 256) + cpiece;
            lds16(ring + tile + piece(r, cpiece), w);
            dst[p.copy_swap ? 16 : 0] = make_uint4(w[0], w[1], w[2], w[3]);
            lds16(ring + tile + 4096 + piece(r, cpiece), w);
            if (p.ones && cpiece == 15) w[3] = __byte_perm(w[3], 0x3f800000u, 0x7610);
            dst[p.copy_swap ? 0 : 16] = make_uint4(w[0], w[1], w[2], w[3]);
          }
          __syncwarp();   // the products behind are instructions of the whole warp
        }
      }
#pragma unroll
      for (int o = 0; o < NX; ++o) {
#pragma unroll
        for (int j = 0; j < 8; j += 4) {   // (half of the columns at a time: all of Z at once would spill)
          uint32_t b[4][4];
#pragma unroll
          for (int c = 0; c < 4; ++c) ldsm4_trans((o_at + tile + (1 - o) * 4096) ^ ((j + c) << 5), b[c]);
          if (!DUAL && !GATED && j == 4 && p.ones && g == 7) b[3][2] = b[3][3] = 0x3f803f80u;   // column 127 of both keys of a register
          if (o + 1 == NX && j == 4) {
            __syncwarp();   // every lane has what it needs of the slot
            load_behind(s + 2);
            slot ^= 1;
          }
#pragma unroll
          for (int part = 0; part < PARTS; ++part)
#pragma unroll
            for (int rt = 0; rt < RT; ++rt)
#pragma unroll
              for (int c = 0; c < 8; ++c)
                mma16816(acc[o][rt][2 * j + c], pp[part][o][rt][0], pp[part][o][rt][1], pp[part][o][rt][2], pp[part][o][rt][3],
                         b[c / 2][2 * (c & 1)], b[c / 2][2 * (c & 1) + 1]);
        }
      }
    }
#pragma unroll
    for (int rt = 0; rt < RT; ++rt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int t = row_token(p, cur.g, cur.rb * (RT * 16) + rt * 16 + hf * 8 + g);
        float f = 1.f;
        if (GATED && t >= 0) f = factor(cur.bh, t);
        const int64_t at = ((int64_t)cur.bh * p.T + t) * 128;
#pragma unroll
        for (int o = 0; o < NX; ++o) {
          void* out = o ? p.out2 : p.out1;
          if (p.out_f32) {   // n-tile nt of a row: eight columns, two to a lane
            if (t >= 0)
#pragma unroll
              for (int nt = 0; nt < 16; ++nt)
                *reinterpret_cast<float2*>(static_cast<float*>(out) + at + nt * 8 + 2 * q) =
                    make_float2(acc[o][rt][nt][2 * hf] * f, acc[o][rt][nt][2 * hf + 1] * f);
          } else if (t >= 0) {
#pragma unroll
            for (int nt = 0; nt < 16; ++nt)
              *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(out) + at + nt * 8 + 2 * q) =
                  pack_bf16(acc[o][rt][nt][2 * hf] * f, acc[o][rt][nt][2 * hf + 1] * f);
          }
        }
      }
    it += gridDim.x;
    if (it >= p.items) break;
  }
}

template <int RT, bool DUAL, bool GATED, int PARTS>
cudaError_t launch_lines(const LineParams& p, cudaStream_t st) {
  using L = LineSmem<RT, DUAL>;
  static_assert(L::warps_per_sm * (L::bytes + 1024) <= 228 * 1024, "the rings of an SM");
  auto* kernel = line_products_kernel<RT, DUAL, GATED, PARTS>;
  const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, L::bytes);
  if (err != cudaSuccess) return err;
  const uint32_t most = (uint32_t)smat_sm_count() * L::warps_per_sm;
  return smat_launch_pdl(kernel, dim3(p.items < most ? p.items : most), 32, (size_t)L::bytes, st, p);
}

struct LineShape {
  uint32_t rt, groups, blocks, lines, slots;   // 16-row tiles of a row block; see LineParams
  uint64_t items;
};
LineShape line_shape(const SmatGeo& g, int bh, int rows_are_types, bool dual = false) {
  const int64_t rows = rows_are_types ? (g.m + g.B - 1) / g.B : (g.n + g.P - 1) / g.P;
  const int64_t layers = rows_are_types ? (g.n + g.P - 1) / g.P : (g.m + g.B - 1) / g.B;
  LineShape s;
  s.rt = rows <= 16 || dual ? 1 : 2;   // (both products of 32 rows are more than a thread's registers)
  s.groups = (uint32_t)(rows_are_types ? g.B : g.P);
  s.lines = (uint32_t)(rows_are_types ? g.qpow[g.D - 1] : g.A);
  s.blocks = (uint32_t)((rows + s.rt * 16 - 1) / (s.rt * 16));
  s.slots = (uint32_t)(s.lines * layers);
  s.items = (uint64_t)bh * s.groups * s.blocks;
  return s;
}

}  // namespace

bool smat_lines_supported(const SmatGeo& geo, int bh) {
  if (geo.dense_G || geo.T >= ((int64_t)1 << 30) || geo.n < geo.P || geo.m < geo.B || (uint64_t)geo.B * geo.q >= (1ull << 31))
    return false;
  // Quotients by umulhi: items by items of a head, slots by lines.  The two-product launch has the most row blocks (d = 2 with a
  // prime given by the caller, one head of 1.1 M tokens, q = 32771: 65,542 items a head where the single products have 32,771).
  for (int launch = 0; launch < 3; ++launch) {
    const int types = launch == 0;
    const LineShape s = line_shape(geo, bh, types, launch == 2);
    const int64_t layers = (types ? geo.n / geo.P : geo.m / geo.B) + 1;
    if (s.items * s.groups * s.blocks >= (1ull << 32) || (uint64_t)s.lines * layers * s.lines >= (1ull << 31)) return false;
  }
  return true;
}

// The line lies where the gathered bytes (from the L2 cache) pass the tables' (to and from memory) by a limit; the pass in us, with
// tables / without.  Forward 2.3: d = 3, q = 29, 16 heads, ratio 1.7 (24 K tokens) 648 / 387, 2.1 (28 K) 673 / 607, 2.3 (32 K) 696 / 677, 2.9
// (40 K) 765 / 850; d = 4, q = 11, 16 heads, 2.0 (10,240) 608 / 536, 2.5 (12,288) 615 / 643; with fp32 tables d = 2, 16 heads, 2.0
// (34,880) 1097 / 392; d = 3, 8 heads, 1.4 (41,024) 1159 / 637.  d = 4 with fp32 tables (scores in three parts, staged sums) 1.85: 8
// heads, 1.7 (16,448) 717 / 671, 2.0 (19,520) 733 / 769, 2.2 (22,592) 748 / 867; not beyond, where tables are summed by Algorithm 2: d = 5,
// 8 heads of 3136 62 ms / 185 us.  Plans made for training steps 1.75, since dK
// and dV take two products of a gather: d = 4, 8 heads, 1.5 (7168) 845 / 751, 2.0 (8192) 851 / 876, gated 974 / 1019.  d = 2 with a bf16
// table 0.75: there is one, and its pooling and read are near the memory rate; 32 heads, 0.7 (4096) 85 / 83 and the training step
// 250 / 237, 16 heads, 0.8 (6144), the training step 210.7 / 214.5.  Types of less than two tokens leave the row tile empty: 16
// heads of 5376, d = 4 (1.8) 587 / 580.
// Items, a warp each: one to an SM (plans are made without a device: the chip's count), but with bf16 tables half of the warps that
// the chip runs.  That line is not where the speed turns (2 heads of 4096 tokens, d = 3, 45 with tables, 39 without): below it
// positional arrays give the same bits as positions, for routed calls form tables on every plan.
bool smat_lines_pay(const SmatGeo& geo, int bh, int table_bytes, bool trains) {
  constexpr uint64_t SMS = 148;
  if (!smat_lines_supported(geo, bh) || 2 * geo.B > geo.m) return false;
  const LineShape s = line_shape(geo, bh, 1);
  const double gathered = (double)s.groups * s.blocks * s.slots * 512;
  const double tables = 2.0 * (double)(geo.P + (geo.D == 1 ? 0 : geo.B)) * 16384 * table_bytes;
  const double limit = geo.D == 1 && table_bytes == 2 ? 0.75 : trains ? 1.75 : geo.D == 3 && table_bytes == 4 ? 1.85 : 2.3;
  return s.items >= (table_bytes == 2 ? 6 * SMS : SMS) && gathered <= limit * tables;
}

namespace {
LineParams line_geometry(const SmatGeo& geo, const LineShape& sh, int rows_are_types) {
  LineParams p{};
  p.T = geo.T; p.n = (uint32_t)geo.n; p.m = (uint32_t)geo.m; p.P = (uint32_t)geo.P; p.B = (uint32_t)geo.B;
  p.q = (uint32_t)geo.q; p.D = (uint32_t)geo.D;
  for (int k = 0; k < geo.D; ++k) { p.qpow[k] = (uint32_t)geo.qpow[k]; p.dir_start[k] = (uint32_t)geo.dir_group_start[k]; }
  p.rows_are_types = rows_are_types;
  p.key_first = rows_are_types ? 0 : p.n; p.key_count = rows_are_types ? p.n : p.m; p.key_period = rows_are_types ? p.P : p.B;
  p.groups = sh.groups; p.lines = sh.lines; p.slots = sh.slots; p.blocks = sh.blocks; p.items = (uint32_t)sh.items;
  p.steps = (p.slots + LN_STEP - 1) / LN_STEP;
  p.q_inv = (uint32_t)(((1ull << 32) + geo.q - 1) / geo.q);
  p.lines_inv = (uint32_t)(((1ull << 32) + p.lines - 1) / p.lines);
  const uint32_t per = p.groups * p.blocks;
  p.per_inv = (uint32_t)(((1ull << 32) + per - 1) / per);
  p.full_steps = p.lines * (p.key_count / p.key_period) / LN_STEP;
  return p;
}

// One state of the tables as the pass's kernels would leave it, widened to fp32 (verification export): where *mark says that
// the workspace holds K and V in the tables' place, from these with the roundings of the tables, else from the table.
__global__ void __launch_bounds__(256) line_tables_kernel(const __grid_constant__ LineParams p, const int* mark,
                                                          const __nv_bfloat16* beside, const __nv_bfloat16* behind, const void* table,
                                                          int table_bf16, int profile_bf16, int types, float* dst) {
  const uint32_t grp = blockIdx.x, bh = blockIdx.y, j = threadIdx.x & 127, i0 = threadIdx.x >> 7;
  const int64_t at = ((int64_t)bh * gridDim.x + grp) * 16384 + threadIdx.x;
  pdl_wait();
  const int where = *mark;
  if (where == 0) {
    for (int k = 0; k < 64; ++k)
      dst[at + k * 256] = table_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(table)[at + k * 256])
                                     : static_cast<const float*>(table)[at + k * 256];
    return;
  }
  const __nv_bfloat16* src = where == 1 ? beside + (int64_t)bh * p.T * 256 : behind + (int64_t)bh * p.n * 256;
  float sum[64];
  for (int k = 0; k < 64; ++k) sum[k] = 0.f;
  const LineOf line = line_of(p, types ? grp : 0);
  const uint32_t layers = p.slots / p.lines, cells = types ? p.lines : 1;
  for (uint32_t c = 0; c < cells; ++c) {
    float f[64];
    for (int k = 0; k < 64; ++k) f[k] = 0.f;
    for (uint32_t l = 0; l < layers; ++l) {
      Slot e{grp + l * p.P, grp + l * p.P < p.n};
      if (types) e = slot_token(p, line, l * p.lines + c);
      if (!e.there) continue;
      const uint32_t t = e.t;
      const __nv_bfloat16* kv = src + (int64_t)t * 256;
      const float v = __bfloat162float(kv[128 + j]);
#pragma unroll
      for (int k = 0; k < 64; ++k) f[k] += __bfloat162float(kv[2 * k + i0]) * v;
    }
#pragma unroll
    for (int k = 0; k < 64; ++k) sum[k] += profile_bf16 ? __bfloat162float(__float2bfloat16_rn(f[k])) : f[k];
  }
#pragma unroll
  for (int k = 0; k < 64; ++k) dst[at + k * 256] = table_bf16 ? __bfloat162float(__float2bfloat16_rn(sum[k])) : sum[k];
}
}  // namespace

cudaError_t smat_launch_line_tables(const SmatGeo& geo, int bh, const int* mark, const void* beside, const void* behind,
                                    const void* table, int table_bf16, int profile_bf16, int types, float* dst, cudaStream_t st) {
  const LineParams p = line_geometry(geo, line_shape(geo, bh, 1), 1);
  using B16 = const __nv_bfloat16;
  return smat_launch_pdl(line_tables_kernel, dim3((unsigned)(types ? geo.B : geo.P), (unsigned)bh), 256, 0, st, p, mark,
                         static_cast<B16*>(beside), static_cast<B16*>(behind), table, table_bf16, profile_bf16, types, dst);
}

cudaError_t smat_launch_line_products(const SmatLineArgs& a, const SmatGeo& geo, int bh, cudaStream_t st) {
  // (score parts and the ones column: of one ungated product)
  if (a.parts < 1 || a.parts > 3 || ((a.parts > 1 || a.ones) && (a.out2 || a.lam))) return cudaErrorInvalidValue;
  LineParams p = line_geometry(geo, line_shape(geo, bh, a.rows_are_types, a.out2 != nullptr), a.rows_are_types);
  using B16 = const __nv_bfloat16;
  p.x1 = static_cast<B16*>(a.x1); p.x2 = static_cast<B16*>(a.x2); p.y = static_cast<B16*>(a.y); p.z = static_cast<B16*>(a.z);
  p.out1 = a.out1; p.out2 = a.out2; p.out_f32 = a.out_f32; p.ones = a.ones;
  p.copy = static_cast<__nv_bfloat16*>(a.copy); p.copy_head = a.copy_head; p.copy_swap = a.copy_swap; p.mark = a.mark; p.mark_value = a.mark_value;
  p.clear = a.clear;
  p.lam = a.lam;
  if (a.out2) return a.lam ? launch_lines<1, true, true, 1>(p, st) : launch_lines<1, true, false, 1>(p, st);
  if (line_shape(geo, bh, a.rows_are_types).rt == 1) {
    if (a.lam) return launch_lines<1, false, true, 1>(p, st);
    return a.parts == 3   ? launch_lines<1, false, false, 3>(p, st)
           : a.parts == 2 ? launch_lines<1, false, false, 2>(p, st)
                          : launch_lines<1, false, false, 1>(p, st);
  }
  if (a.lam) return launch_lines<2, false, true, 1>(p, st);
  return a.parts == 3   ? launch_lines<2, false, false, 3>(p, st)
         : a.parts == 2 ? launch_lines<2, false, false, 2>(p, st)
                        : launch_lines<2, false, false, 1>(p, st);
}
