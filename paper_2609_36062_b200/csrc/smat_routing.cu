// User-supplied routing (Sec. 3, "construction of G": the content-based assignment): the caller gives every distant
// token its profile cell and every recent token its type as integer arrays; this file turns them into the per-group
// token lists (CSR: offsets + token positions, ascending inside a group) that the pooling and routed-read kernels
// walk instead of the positional strides.  Integer work only: a counting sort per (head, kind), stable so that the
// order of the floating-point sums downstream does not depend on thread timing.
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"

namespace {

// What a CTA takes is a chain of passes over its tokens in shared memory, so as many warps as there are counters for, at most 32
// (16 heads of 35,968 tokens, d = 4: 91 us with 8, 66 with 22; 32 heads of 16 K: 48, 35), several keys of a lane in flight, and
// no match.any, which takes a step for every different key of a warp: 35 us and 21.  Equal keys are ranked a key at a time; a
// token at a time, all tokens in one group took 74 us at 35,968 tokens where 60 were taken with match.any and 27 are now, eight groups 73, 66
// and 39, runs of four tokens 81, 74 and 45.
constexpr int ROUTE_THREADS = 1024;
constexpr int ROUTE_AHEAD = 4;   // keys of a lane in flight

// One CTA per (head, kind); kind 0: profiles of the n distant tokens, kind 1: types of the m recent tokens.
// The tokens are cut into W contiguous ranges, one per warp (W as large as shared memory allows, at most 32):
//   1. every warp histograms the keys of its range in its own row of counters (keys outside [0, G) are dropped:
//      such a token belongs to no group)
//   2. totals per group (a heavy group's parts are noted: their order depends on thread timing, but each is a set of rows that
//      some CTA reads on its own), exclusive scan -> offs[0 .. G]; row w then becomes the first slot of group g for warp w's
//      tokens: offs[g] + the counts of the warps before it
//   3. stable placement: every warp walks ITS range in order, 32 tokens at a time; every lane advances the warp's cursor of
//      its token's group, those that find it advanced further rank themselves among the lanes of the same key (one ballot for
//      each such key, at most 16; match.any takes a step for every different key, and nearly all 32 are), and writes its
//      token's position.  Ranges are in token order and each warp's slots follow those of the warps before it, so the list of
//      a group is ascending.
struct RouteParams {
  const int32_t* key[2];   // [bh][count]
  SmatRouteLists to[2];    // lists [bh][count], offsets [bh][G + 1]
  int64_t count[2], G[2], first[2];   // tokens per head, groups, position of the first token of the kind
  int warps;               // W: rows of per-warp counters in shared memory
};

__global__ void __launch_bounds__(ROUTE_THREADS) routing_lists_kernel(const __grid_constant__ RouteParams prm) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ int32_t rows[];     // [1 + W][G + 1]: row 0 totals / offsets, row 1 + w the counters of warp w
  const int kind = blockIdx.y;
  const int64_t bh = blockIdx.x, n = prm.count[kind], G = prm.G[kind], pitch = G + 1;
  const int W = prm.warps;
  const int32_t* key = prm.key[kind] + bh * n;
  const SmatRouteLists& to = prm.to[kind];
  int32_t* list = to.list + bh * n;
  int32_t* offs = to.offs + bh * pitch;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int32_t* total = rows;
  for (int64_t i = tid; i < (1 + W) * pitch; i += ROUTE_THREADS) rows[i] = 0;
  __syncthreads();
  const int64_t per = ((n + W - 1) / W + 31) & ~(int64_t)31;   // tokens per warp range, a multiple of 32
  const int64_t lo = (int64_t)warp * per, hi = lo + per < n ? lo + per : n;
  if (warp < W) {
    int32_t* mine = rows + (1 + warp) * pitch;
    for (int64_t t0 = lo + lane; t0 < hi; t0 += 32 * ROUTE_AHEAD) {
      int32_t k[ROUTE_AHEAD];
#pragma unroll
      for (int i = 0; i < ROUTE_AHEAD; ++i) k[i] = t0 + 32 * i < hi ? key[t0 + 32 * i] : -1;
#pragma unroll
      for (int i = 0; i < ROUTE_AHEAD; ++i)
        if (k[i] >= 0 && k[i] < G) atomicAdd(&mine[k[i]], 1);
    }
  }
  __syncthreads();
  for (int64_t g = tid; g < G; g += ROUTE_THREADS) {
    int32_t sum = 0;
    for (int w = 0; w < W; ++w) sum += rows[(1 + w) * pitch + g];
    total[g + 1] = sum;          // shifted by one: the inclusive scan below leaves the first slot of group g at index g
    if (sum > SMAT_HEAVY_TOKENS && to.heavy) {
      const int32_t parts = (sum - 1) / SMAT_HEAVY_TOKENS, at = atomicAdd(to.heavy_count, parts);   // behind the first
      for (int32_t i = 0; i < parts; ++i) to.heavy[at + i] = SmatHeavyPart{(uint16_t)bh, (uint16_t)g, (uint16_t)(i + 1)};
    }
  }
  __syncthreads();
  __shared__ int32_t warp_sum[ROUTE_THREADS / 32];
  __shared__ int32_t carry;
  if (tid == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 1; base <= G; base += ROUTE_THREADS) {
    const int64_t g = base + tid;
    int32_t x = g <= G ? total[g] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    int32_t before = carry;
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
    if (g <= G) total[g] = before + x;
    __syncthreads();
    if (tid == ROUTE_THREADS - 1) carry = before + x;
    __syncthreads();
  }
  // total[g] = tokens in groups < g (total[0] = 0): the offsets; then the per-warp first slots
  for (int64_t g = tid; g <= G; g += ROUTE_THREADS) offs[g] = total[g];
  for (int64_t g = tid; g < G; g += ROUTE_THREADS) {
    int32_t slot = total[g];
    for (int w = 0; w < W; ++w) {
      const int32_t c = rows[(1 + w) * pitch + g];
      rows[(1 + w) * pitch + g] = slot;
      slot += c;
    }
  }
  __syncthreads();
  if (warp < W) {
    int32_t* cursor = rows + (1 + warp) * pitch;
    const int64_t first = prm.first[kind];
    for (int64_t t0 = lo; t0 < hi; t0 += 32 * ROUTE_AHEAD) {
      int32_t ahead[ROUTE_AHEAD];
#pragma unroll
      for (int i = 0; i < ROUTE_AHEAD; ++i) ahead[i] = t0 + 32 * i + lane < hi ? key[t0 + 32 * i + lane] : -1;
#pragma unroll
      for (int i = 0; i < ROUTE_AHEAD; ++i) {
        const int64_t t = t0 + 32 * i + lane;
        const int32_t k = ahead[i];
        const bool valid = k >= 0 && k < G;
        const int32_t slot = valid ? cursor[k] : 0;
        __syncwarp();
        if (valid) atomicAdd(&cursor[k], 1);
        __syncwarp();
        // keys that met others of their kind: few, but where a group is heavy
        const unsigned same = __ballot_sync(0xffffffffu, valid && cursor[valid ? k : 0] - slot > 1);
        int rank = 0;
        for (unsigned m = same; m;) {   // a step for every different one of these keys, 16 at most
          const int32_t other = __shfl_sync(0xffffffffu, k, __ffs(m) - 1);
          const unsigned peers = __ballot_sync(0xffffffffu, k == other);
          if (k == other) rank = __popc(peers & ((1u << lane) - 1));
          m &= ~peers;
        }
        if (valid) list[slot + rank] = (int32_t)(first + t);
        __syncwarp();
      }
    }
  }
}

// Rows of tokens that belong to no group are never written by a routed read; whoever adds those rows afterwards must
// find zeros there.  One thread per token reads its key; the (rare) token whose key is out of range zeroes its row.
__global__ void zero_unrouted_rows_kernel(const int32_t* key, int64_t count, int64_t G, int64_t first,
                                          uint8_t* rows, int64_t T, int row_bytes, int64_t total) {
  pdl_trigger();
  pdl_wait();
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= total) return;
  const int32_t k = key[w];
  if (k >= 0 && k < G) return;
  const int64_t bh = w / count, t = first + (w - bh * count);
  uint4* dst = reinterpret_cast<uint4*>(rows + (bh * T + t) * row_bytes);
  for (int i = 0; i < row_bytes / 16; ++i) dst[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

cudaError_t smat_launch_zero_unrouted(const int32_t* key, int64_t count, int64_t G, int64_t first, void* rows, int64_t T,
                                      int row_bytes, int bh, cudaStream_t st) {
  const int64_t total = (int64_t)bh * count;
  return smat_launch_pdl(zero_unrouted_rows_kernel, dim3((unsigned)((total + 255) / 256)), 256, 0, st, key, count, G, first,
                         static_cast<uint8_t*>(rows), T, row_bytes, total);
}

// Largest group count the list builder handles (its cursors live in shared memory).
int64_t smat_routing_max_groups() { return 27000; }

cudaError_t smat_launch_routing_lists(const int32_t* prof, const int32_t* type, const SmatRouteLists& prof_to,
                                      const SmatRouteLists& type_to, const SmatGeo& geo, int bh, cudaStream_t st) {
  RouteParams prm;
  prm.key[0] = prof; prm.to[0] = prof_to; prm.count[0] = geo.n; prm.G[0] = geo.P; prm.first[0] = 0;
  prm.key[1] = type; prm.to[1] = type_to; prm.count[1] = geo.m; prm.G[1] = geo.B; prm.first[1] = geo.n;
  const int64_t gmax = geo.P > geo.B ? geo.P : geo.B;
  if (gmax > smat_routing_max_groups()) return cudaErrorInvalidConfiguration;
  int64_t warps = (int64_t)(220 * 1024 / sizeof(int32_t)) / (gmax + 1) - 1;
  if (warps > ROUTE_THREADS / 32) warps = ROUTE_THREADS / 32;
  const int64_t most = geo.n > geo.m ? geo.n : geo.m, useful = (most + 32 * ROUTE_AHEAD - 1) / (32 * ROUTE_AHEAD);
  if (warps > useful) warps = useful;
  if (warps < 1) warps = 1;
  prm.warps = (int)warps;
  const size_t smem = (size_t)(1 + warps) * (gmax + 1) * sizeof(int32_t);
  cudaError_t err = cudaFuncSetAttribute(routing_lists_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  dim3 grid((unsigned)bh, 2);
  return smat_launch_pdl(routing_lists_kernel, grid, ROUTE_THREADS, smem, st, prm);
}
