// Internal declarations shared by the translation units of libsmat (not part of the C boundary).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "smat_geometry.h"

// ---- token groups -----------------------------------------------------------------------------
// A "group" is a set of tokens t0, t0+ts, t0+2ts, ... that one state belongs to:
//   CHUNK   g = chunk index        tokens g*c .. g*c+c-1                          (Sec. 3.1, causal branch)
//   PROFILE g = packed profile x   distant tokens t ≡ x (mod P), t < n            (Eq. "schedule", F_x)
//   TYPE    g = type h             recent tokens with (t-n+1) ≡ h (mod B), t < T  (Eq. "schedule", U_h)
enum SmatGroupMode { SMAT_GM_NONE = 0, SMAT_GM_CHUNK = 1, SMAT_GM_PROFILE = 2, SMAT_GM_TYPE = 3 };

// A listed group may hold any number of tokens: what it has behind its first SMAT_HEAVY_TOKENS is cut into parts of at most
// as many, for kernels that hand these out to several CTAs (where groups hold fewer than SMAT_LISTED_SMALL on average).
constexpr int SMAT_HEAVY_TOKENS = 128, SMAT_LISTED_SMALL = 16;
struct SmatHeavyPart {
  uint16_t bh, group, number;   // (at most 65535 heads, 27000 groups of a routed call, 65535 * 128 tokens); the first part is 1
};
struct SmatGroupSpec {
  int mode;
  int64_t n, T, c, period;  // period = P (PROFILE) or B (TYPE)
  int64_t base, rem;        // the block's tokens = base * period + rem: a group has base or base + 1 of them
  // User-supplied routing (content-based assignment, Sec. 3): when `list` is non-null the tokens of PROFILE / TYPE
  // group g of head bh are list[bh * list_stride + offs[bh * offs_stride + g] ...  offs[... + g + 1]) (token positions
  // in [0, T), ascending inside a group) instead of the positional strides.
  const int32_t* list;
  const int32_t* offs;
  int64_t list_stride, offs_stride;
  const SmatHeavyPart* heavy;   // the parts of all heads, *heavy_count of them in any order (null: not made)
  const int32_t* heavy_count;
};

// a / b of non-negative numbers; a 64-bit division takes the device several hundred cycles, and every role of a persistent
// kernel makes one per item.
SMAT_HD int64_t smat_div(int64_t a, int64_t b) {
  return ((uint64_t)(a | b) >> 32) == 0 ? (int64_t)((uint32_t)a / (uint32_t)b) : a / b;
}

// The tokens of one group: position of the k-th one is at(k).
struct SmatTokens {
  int64_t t0, ts, cnt;
  const int32_t* lst;
  SMAT_HD int64_t at(int64_t k) const { return lst ? (int64_t)lst[k] : t0 + k * ts; }
};

SMAT_HD SmatTokens smat_group_tokens(const SmatGroupSpec& s, int64_t bh, int64_t g) {
  SmatTokens r;
  r.lst = nullptr; r.t0 = 0; r.ts = 1; r.cnt = 0;
  if (s.mode != SMAT_GM_CHUNK && s.list) {
    const int32_t* o = s.offs + bh * s.offs_stride + g;
    r.lst = s.list + bh * s.list_stride + o[0];
    r.cnt = o[1] - o[0];
    return r;
  }
  switch (s.mode) {
    case SMAT_GM_CHUNK:
      r.t0 = g * s.c; r.ts = 1; r.cnt = s.c;
      break;
    case SMAT_GM_PROFILE:
      r.t0 = g; r.ts = s.period; r.cnt = s.base + (g < s.rem);
      break;
    case SMAT_GM_TYPE: {
      int64_t i0 = g ? g : s.period;  // paper's 1-based recent index of the first token of this type
      r.t0 = s.n + i0 - 1; r.ts = s.period; r.cnt = s.base + (i0 <= s.rem);
      break;
    }
    default:
      break;
  }
  return r;
}

// Whether two arrays share memory.
inline bool smat_overlap(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return x < y + b_bytes && y < x + a_bytes;
}

// ---- within-chunk tiles on the fp32 ALUs ------------------------------------------------------------
// Out[i] = Σ_j X_ij P3_j + P4_i · St (+ acc[i] for rows acc_lo <= t < acc_hi), X_ij = P1_i · P2_j for j <= i (upper:
// j >= i) of the same chunk.  P1, P2, P4 have score_dim columns, P3, acc and Out out_dim; the states are
// [bh][NC][score_dim][out_dim], or [..][out_dim][score_dim] with st_trans.
struct SmatTileJob {
  const void *p1, *p2, *p3, *p4;   // [bh][T][.] rows in the plan's dtype
  const float* st;
  const float* acc;                // [bh][T][out_dim] fp32
  int64_t acc_lo, acc_hi;
  void* out;
  int upper, st_trans;
};
struct SmatTileArgs {
  SmatTileJob job[3];
  int jobs;
  int64_t T;
  int c, NC;
  const float* lam;                // gated variant: prefix sums of the log-gates [bh][T]; X_ij is multiplied by the decay
  int together;                    // set by the launcher: an output shares memory with its job's P2 or P3
};
// The output of a job may be the array of one of that job's operands (row for row).
cudaError_t smat_launch_tile_rows(const SmatTileArgs& a, int bf16, int score_dim, int out_dim, int bh, cudaStream_t st);

// Exclusive scans of per-chunk states [bh][NC][state] in place, over up to two independent chunk ranges each;
// reverse = suffix scan.
struct SmatScanJob {
  float* S;
  int64_t lo0, hi0, lo1, hi1;
  int reverse;
};
struct SmatScanArgs {
  SmatScanJob job[2];
  int jobs;
};
cudaError_t smat_launch_scan(const SmatScanArgs& a, int64_t state_elems, int64_t NC, int bh, cudaStream_t st);

// Algorithm 2 (direct form) and its transpose, one slab of state entries per CTA held in shared memory.
// transpose = 0: out[h] = Σ_{x ∈ H_h} in[x]  (in: P states, out: B states)
// transpose = 1: out[x] = Σ_{h ∋ x} in[h]   (in: B states, out: P states)
cudaError_t smat_launch_tabulate_alg2(const float* in, float* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                      int transpose, cudaStream_t st);
// Largest slab (entries) the direct tabulation can hold in shared memory; 0 if none fits.
int smat_tabulate_alg2_slab(int64_t rows_in, int64_t state_elems);

cudaError_t smat_launch_mask(uint8_t* mask, const SmatGeo& geo, cudaStream_t st);

// Pooling of outer products into one fp32 state per group: state[bh][g] = Σ_{tokens of g} a_tᵀ b_t (a: r columns,
// b: p columns), for up to four sets of groups in one launch.
struct SmatPoolJob {
  const void *a, *b;               // [bh][T][.] rows in the plan's dtype
  float* state;
  SmatGroupSpec grp;
  int64_t groups;                  // states per head
};
struct SmatPoolArgs {
  SmatPoolJob job[4];
  int jobs;
};
int smat_sm_count();   // SMs of the device
// Shared memory to ask for in a launch of `ctas` CTAs that need `bytes` each: while every CTA can have an SM to itself, more
// than half of what an SM has.  A launch that is set up while the one before drains is placed on the SMs that are free then,
// two CTAs to one where both fit, although others will be free by the time it begins.  fp32, d = 1, forward and backward:
// 2 heads of 512 tokens, 64 wide, 41.1 -> 28.9 us, one head of 1024 42.3 -> 30.5, 128 wide 72.5 -> 56.2.
inline int smat_smem_alone(int64_t ctas, int bytes) {
  constexpr int more_than_half = 116 * 1024;
  return ctas <= smat_sm_count() && bytes < more_than_half ? more_than_half : bytes;
}
// clear (or null): status word that the launch sets to zero.
cudaError_t smat_launch_pool(const SmatPoolArgs& a, int bf16, int64_t Tlen, int bh, int r, int p, int* clear, cudaStream_t st);

// Routed reads of per-group fp32 states [r][p]: out[t] = x_t · state[g(t)] for the tokens of every group (trans: the
// second state index is contracted), fp32 rows, for up to three sets in one launch.
struct SmatReadJob {
  const void* x;                   // [bh][T][r] rows (trans: [bh][T][p])
  const float* state;
  float* out;                      // [bh][T][p] (trans: [bh][T][r])
  SmatGroupSpec grp;
  int64_t groups;
  int trans;
};
struct SmatReadArgs {
  SmatReadJob job[3];
  int jobs;
};
// scan (or null): chunk states, NC of r x p to a head, that CTAs of the same launch scan (as smat_launch_scan would).
cudaError_t smat_launch_state_read(const SmatReadArgs& a, int bf16, int64_t Tlen, int bh, int r, int p, int* status,
                                   cudaStream_t st, const SmatScanArgs* scan = nullptr, int64_t NC = 0);

// Both stages of the d = 4 tabulation with the table between them in shared memory (the primes for which it fits).
int smat_tabulate_slab_supported(int q, int64_t state_elems);
cudaError_t smat_launch_tabulate_slab(const void* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh, int* status,
                                      cudaStream_t st);

// The d = 3 tabulation of fp32 tables with the sums in registers (the primes it is instantiated for).
int smat_tabulate_d3_f32_supported(const SmatGeo& geo, int64_t state_elems);
cudaError_t smat_launch_tabulate_d3_f32(const float* in, float* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                        int* status, cudaStream_t st);

// Staged exact tabulation (same sums as Algorithm 2, one coordinate at a time). Slab = 0: not available.
int smat_tabulate_staged_slab(const SmatGeo& geo, int64_t state_elems, int transpose);
// out_bf16 = 1 writes the result table as bf16 (same layout, half the bytes) instead of fp32.
cudaError_t smat_launch_tabulate_staged(const float* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                        int transpose, int out_bf16, cudaStream_t st);

// Tensor-core kernels of the causal branch (bf16, d_k = d_v = 128, 128-token tiles; n and T - n multiples of 128).
bool smat_tc_available();
// S_in[bh][tile] (bf16 [128][128]) = exclusive prefix sum of K_bᵀ V_b over the tiles of each block;
// through = 1 runs one scan over the whole sequence (d = 1), else the scan restarts at token n.
// reverse = 1 gives exclusive suffix sums instead (the scan adjoint, with K, V replaced by Q, dO).
// lam (gated variant): inclusive prefix sums of the log-gates [bh][T]; K then holds the rows rescaled to the end of
// their tile (forward order) or to its start (reverse order), and the running state decays by the tile's total gate.
cudaError_t smat_launch_chunk_scan_tc(const void* K, const void* V, void* Sin_bf16, int64_t T, int bh, int64_t n,
                                      int through, int reverse, int* status, cudaStream_t st, const float* lam = nullptr);
// Within-chunk adjoints on tensor cores (which = 0: dQ, 1: dK, 2: dV), see tile_product_tc_kernel.
cudaError_t smat_launch_chunk_adjoint_tc(int which, const void* Q, const void* K, const void* V, const void* dO,
                                         const void* Sin_bf16, const void* Dbar_bf16, const float* addend,
                                         int64_t add_lo, int64_t add_hi, void* Out, int64_t T, int bh, int* status,
                                         cudaStream_t st, int addend_bf16 = 0);
// The three adjoints of every tile in one launch (all operands of a tile loaded once, both score tiles formed once).
cudaError_t smat_launch_bwd_tiles_fused_tc(const void* Q, const void* K, const void* V, const void* dO,
                                           const void* Sin_bf16, const void* Dbar_bf16, const void* lr_q, const void* lr_k,
                                           const void* lr_v, int64_t n, void* dQ, void* dK, void* dV, int64_t T, int bh,
                                           int* status, cudaStream_t st, const float* lam = nullptr, float* dlam = nullptr);
// O_b = Q_b S_in[b] + tril(Q_b K_bᵀ) V_b (+ ylr rows for tokens >= n_lr).
cudaError_t smat_launch_chunk_output_tc(const void* Q, const void* K, const void* V, const void* Sin_bf16,
                                        const float* ylr, int64_t n_lr, void* O, int64_t T, int bh, int* status,
                                        cudaStream_t st, const float* lam = nullptr);
// Typed read on tensor cores: ylr[t] = q_tᵀ U_type(t) for recent tokens, U kept as bf16 [bh][B][128][128].
// (transposed = 1 contracts the second state index instead: out[t] = state · x_t; grp selects types or profiles)
// (the rows go to `out` as fp32, or to `out_bf16` when that is non-null)
cudaError_t smat_launch_state_read_tc(const void* X, const void* state_bf16, float* out, void* out_bf16, int transposed,
                                      const SmatGroupSpec& grp, int64_t groups, int64_t T, int bh, int* status,
                                      cudaStream_t st);
// Both reads of the per-profile adjoint states in one launch (every state loaded once): out_t[t] = St x_t for rows Xt,
// out_n[t] = Stᵀ x_t for rows Xn; bf16 results.
cudaError_t smat_launch_state_read_dual_tc(const void* Xt, const void* Xn, const void* state_bf16, void* out_t_bf16,
                                           void* out_n_bf16, const SmatGroupSpec& grp, int64_t groups, int64_t T, int bh,
                                           int* status, cudaStream_t st);
// One step of cached decoding: S += k vᵀ, o = qᵀ (U_type + S) for every head (fp32 running state).
cudaError_t smat_launch_decode_step(const void* q, const void* k, const void* v, void* o, float* S, const void* U,
                                    int u_bf16, int in_bf16, int64_t type, int64_t types, int r, int p, int bh,
                                    cudaStream_t st, const float* log_a = nullptr, float* log_g = nullptr);
// d = 3 tabulation from a bf16 profile table on the fp32 ALUs (primes too large for the resident-matrix kernel).
int smat_tabulate_d3_bf16_slab(const SmatGeo& geo, int64_t state_elems);
cudaError_t smat_launch_tabulate_d3_bf16(const void* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                         cudaStream_t st);
// The same on the tensor cores with the Radon matrix generated beside the stream (primes 19 to 53).
int smat_tabulate_d3_wide_supported(const SmatGeo& geo, int64_t state_elems);
cudaError_t smat_launch_tabulate_d3_wide(const void* in, void* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                         int* status, cudaStream_t st);
// bf16 -> fp32 copy of a table (debug export).
// Tabulation on the tensor cores (bf16 tables; d = 3, 4 with a prime small enough for a resident Radon matrix).
int smat_tabulate_tc_supported(const SmatGeo& geo, int64_t state_elems);
int smat_tabulate_tc_layout_ok(int q);   // host-only self-check of the kernel's shared-memory map for prime q
int64_t smat_tabulate_tc_scratch_rows(const SmatGeo& geo);
int64_t smat_tabulate_tc_scratch_elems(const SmatGeo& geo, int64_t state_elems, int bh);
cudaError_t smat_launch_tabulate_tc(const void* in, void* out, void* scratch, const SmatGeo& geo, int64_t state_elems,
                                    int bh, int transpose, int* status, cudaStream_t st, int* launches);
cudaError_t smat_launch_widen_bf16(const void* src_bf16, float* dst, int64_t count, cudaStream_t st);
// Pooling on tensor cores: F[bh][x] = Σ_{t ≡ x (mod P), t < n} k_t v_tᵀ, stored as fp32 or bf16.
cudaError_t smat_launch_pool_tc(const void* K, const void* V, void* F, int out_bf16, const SmatGroupSpec& grp,
                                int64_t groups, int64_t max_tokens, int64_t T, int bh, int* status, cudaStream_t st);
// Gated variant (Sec. 3.2): prefix / suffix sums per head, rescaled copies, decayed chunk scan, gate gradient.
cudaError_t smat_launch_head_scan(const float* in, float* out, int64_t len, int bh, int reverse, cudaStream_t st);
cudaError_t smat_launch_gate_scale(const void* A, const void* B, void* out, const float* lam, int mode, int bf16,
                                   int64_t n, int64_t c, int64_t T, int dim, int bh, cudaStream_t st);
// out1 = A rescaled to its 128-token tile (mode 0: from its start, 1: to its end), out2 = B (t < n) or C rescaled to the
// block boundary (null: skipped); bf16 rows of 128.
cudaError_t smat_launch_gate_scale_pair(const void* A, const void* B, const void* C, void* out1, void* out2, const float* lam,
                                        int mode, int64_t n, int64_t T, int bh, cudaStream_t st);
cudaError_t smat_launch_gated_scan(float* S, const float* lam, int64_t state_elems, int64_t NC, int64_t c, int bh,
                                   int64_t lo0, int64_t hi0, int64_t lo1, int64_t hi1, int reverse, cudaStream_t st);
cudaError_t smat_launch_gate_dlam(const void* Q, const void* dQ, const void* K, const void* dK, float* dlam, int bf16,
                                  int dim, int64_t T, int bh, cudaStream_t st);
// Normalised output (Sec. 2): elementwise steps around the linear pass (see smat_gated.cu).
cudaError_t smat_launch_normalize_step(int step, const void* a, const void* b, void* out, int bf16, int p, int64_t rows,
                                       cudaStream_t st);
// Token lists of user-supplied routing: prof [bh][n] (cells in [0, P)) and type [bh][m] (types in [0, B)) -> CSR lists
// (offsets [bh][G + 1], token positions [bh][count], ascending inside a group).  Keys out of range are dropped.  Parts of
// heavy groups are appended at heavy (null, or room for bh * (count / SMAT_HEAVY_TOKENS)) and added to *heavy_count, zero before.
struct SmatRouteLists {
  int32_t* list;
  int32_t* offs;
  SmatHeavyPart* heavy;
  int32_t* heavy_count;
};
int64_t smat_routing_max_groups();
cudaError_t smat_launch_routing_lists(const int32_t* prof, const int32_t* type, const SmatRouteLists& prof_to,
                                      const SmatRouteLists& type_to, const SmatGeo& geo, int bh, cudaStream_t st);
// Zeroes the row (row_bytes bytes at rows + (bh*T + first + i) * row_bytes) of every token i whose key lies outside [0, G).
cudaError_t smat_launch_zero_unrouted(const int32_t* key, int64_t count, int64_t G, int64_t first, void* rows, int64_t T,
                                      int row_bytes, int bh, cudaStream_t st);
// Two-level causal branch: segment totals, then (after an exclusive scan of the totals, where a block has more than two)
// per-segment fused output.
// Block 0 holds rows0 tokens of every head and block 1 the rows1 after them (0: one block, d = 1); the last tile of a
// block may be partial.
int smat_segment_tiles(int64_t tiles_block0, int64_t tiles_block1, int bh);
void smat_segment_counts(int64_t tiles0, int64_t tiles1, int bh, int L, int* nseg0, int* nseg1);
bool smat_segments_need_scan(int nseg0, int nseg1);
cudaError_t smat_launch_segment_state_tc(const void* K, const void* V, float* totals, int64_t rows0, int64_t rows1,
                                         int nseg0, int nseg1, int bh, int* status, cudaStream_t st, int ones = 0);
// ylr_f32: the long-range rows are fp32 (else bf16).  split: any blocks (else of whole tiles), and the state and the scores enter
// their products as a bf16 part plus a bf16 remainder (with fp32 rows only).  divide: the rows leave divided by their last column,
// which stays as it is, and V's last column counts as one (as in the totals with `ones`).
cudaError_t smat_launch_segment_output_tc(const void* Q, const void* K, const void* V, const float* seg_in,
                                          const void* ylr, int ylr_f32, int split, int64_t n_lr, void* O, int64_t rows0, int64_t rows1,
                                          int nseg0, int nseg1, int bh, int* status, cudaStream_t st,
                                          void* sin_tiles = nullptr, int64_t sin_lo = 0, int64_t sin_hi = 0, int divide = 0);
// Long-range rows without tables (see smat_lines.cu), positional routing, bf16 rows of 128: for every token t of a type (or,
// rows_are_types = 0, of a cell) out1_t = Σ_s (x1_t · y_s) z_s over the tokens s of the cells of its hyperplane (of the types
// through the cell), and with out2 also out2_t = Σ_s (x2_t · z_s) y_s.
struct SmatLineArgs {
  const void *x1, *x2, *y, *z;
  void *out1, *out2;
  int out_f32, rows_are_types;
  int ones;              // Z's last column counts as one (one product, ungated)
  int parts;             // bf16 parts in which a score enters its product: 1, 2 (16 bits) or 3 (all of fp32); more than one only
                         // for one product, ungated
  const float* lam;      // gated: prefix sums of the log-gates; terms are multiplied by exp(λ_recent - λ_distant)
  void* copy;            // null, or where K and V of every distant token are left side by side: token t of head b at
  int64_t copy_head;     // row b * copy_head + t of 512 bytes
  int copy_swap;         // y is V and z is K
  int* mark;             // null, or a word that is set to mark_value
  int mark_value;
  int* clear;            // null, or a status word that is set to zero
};
// Whether the kernel takes the shape, and whether it is the faster way (table_bytes: of an entry of the tables otherwise; trains: a
// backward follows every forward).
bool smat_lines_supported(const SmatGeo& geo, int bh);
bool smat_lines_pay(const SmatGeo& geo, int bh, int table_bytes, bool trains);
// F (types = 0) or U of a pass of a plan that may have formed no tables, as fp32: from K and V that it left where *mark says (1:
// beside, 2: behind), or from `table` where *mark is zero.
cudaError_t smat_launch_line_tables(const SmatGeo& geo, int bh, const int* mark, const void* beside, const void* behind,
                                    const void* table, int table_bf16, int profile_bf16, int types, float* dst, cudaStream_t st);
cudaError_t smat_launch_line_products(const SmatLineArgs& a, const SmatGeo& geo, int bh, cudaStream_t st);
