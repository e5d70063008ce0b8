// Tabulation U = C F for d = 3 (Algorithm 2) with fp32 tables, on the fp32 ALUs with the sums held in registers: fp32
// inputs, and bf16 plans whose blocks are not whole 128-token tiles.
//
// For d = 3 the points are (x1, x2) ∈ F_q², point index x1 + q x2, and the types are the lines
//        slope a < q :  h = a q + b,   { x1 + a x2 = b }        U_h = Σ_{x2} F[(b - a x2) mod q, x2]
//        extra class :  h = q² + b,    { x2 = b }               U_h = Σ_{x1} F[x1, b]
// Two lines share at most one point, so no partial sum is common to two of them: q³ + q² additions per state entry is
// what Algorithm 2 asks for and also the least any add-only scheme can do.  What this kernel organises is where the
// operands come from.  A thread owns EPT neighbouring state entries and, for K slopes at a time, all q offsets: K q
// accumulators.  It walks the q columns (fixed x2) of a slab once per K slopes; every value is loaded from shared memory
// once and added into K accumulators (two entries per instruction), so shared-memory traffic per addition falls by K.
//
// The register index of an accumulator has to be a compile-time constant.  Slopes are therefore grouped as
// a0·{g_0 .. g_{K-1}} with g_i = r^i (r a primitive root of F_q) and a0 = r^{K t} for task t: the sets tile F_q* when K
// divides q - 1.  With x2' = a0 x2 the target offset is b = x1 + g_i x2', which does not depend on a0: every task runs the
// same code and only permutes the order in which it visits the columns (x2 = x2' / a0).  The body is unrolled over all
// columns, q² (K + 1) instructions of 16 bytes: at most 25 KB, inside the instruction cache.  Slope 0 and the extra class
// form one lighter task per slab.
//
// One persistent CTA per SM, 32 EPT entries of every point per slab, as many slabs in shared memory as fit (at most four);
// slabs arrive by TMA, and the warp that finishes the last task of a slab starts the next load into the freed buffer.
// Warps take (slab, task) pairs from a shared counter and write whole rows of 128 EPT bytes.  The least time is the
// tables' bytes: 32 heads of 16,384 entries at q = 17, 1.25 GB, 0.19 ms.  Measured there: 0.229 ms with three slabs (0.257
// while lane 0 alone looked at a slab's barrier; then 0.352 with two slabs), 0.425 for the staged kernel, which keeps its
// sums in shared memory.  16 heads, staged and here: q = 11 0.091, 0.052; q = 13 0.121, 0.070; q = 19 0.299, 0.145;
// 8 heads, q = 23: 0.260, 0.150.
#include <cuda.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_radon.cuh"
#include "smat_tc.cuh"

namespace {

using namespace tc;

__host__ __device__ constexpr int cpow_mod(int base, int e, int q) {
  int r = 1;
  for (int i = 0; i < e; ++i) r = (r * base) % q;
  return r;
}
__host__ __device__ constexpr bool is_primitive_root(int r, int q) {
  int v = 1;
  for (int e = 1; e < q - 1; ++e) {
    v = (v * r) % q;
    if (v == 1) return false;
  }
  return true;
}

// Per-prime constants: K slopes per task (K | q - 1), a primitive root, the entries per thread (two slabs of q² x 128 EPT
// bytes must fit shared memory) and the warps.  EPT K q accumulators and 25 other registers a thread have to leave room
// for enough warps to hide the loads; small primes have the shared-memory bandwidth for K = 2 and twenty warps (q = 11:
// 0.064 ms against 0.075 at K = 5 and sixteen, q = 13: 0.087 against 0.091 at K = 4), large ones do not (q = 17: 0.299
// against 0.257 at K = 4 and twelve, q = 19: 0.275 against 0.206 at K = 3; all of these while lane 0 alone waited).
template <int Q> struct D3Cfg;
template <> struct D3Cfg<11> { static constexpr int K = 2, ROOT = 2, EPT = 2, WARPS = 20; };
template <> struct D3Cfg<13> { static constexpr int K = 2, ROOT = 2, EPT = 2, WARPS = 20; };
template <> struct D3Cfg<17> { static constexpr int K = 4, ROOT = 3, EPT = 2, WARPS = 12; };
template <> struct D3Cfg<19> { static constexpr int K = 3, ROOT = 2, EPT = 2, WARPS = 12; };
template <> struct D3Cfg<23> { static constexpr int K = 2, ROOT = 5, EPT = 1, WARPS = 24; };

template <int Q>
struct D3Layout {
  using Cfg = D3Cfg<Q>;
  static constexpr int K = Cfg::K, EPT = Cfg::EPT;
  static_assert((Q - 1) % K == 0, "slope groups must tile the nonzero slopes");
  static_assert(is_primitive_root(Cfg::ROOT, Q), "ROOT must generate the multiplicative group");
  static constexpr int ENTRIES = 32 * EPT, ROW = ENTRIES * 4;      // entries and bytes per point of a slab
  static constexpr int TASKS = (Q - 1) / K + 1;                    // K nonzero slopes each, and slope 0 with the extra class
  static constexpr int BOXES = (Q * Q + 255) / 256, BOX_ROWS = (Q * Q + BOXES - 1) / BOXES;   // a box holds 256 rows at most
  static constexpr int SLAB_BYTES = BOXES * BOX_ROWS * ROW;
  static constexpr int FIT = (227 * 1024 - 256) / SLAB_BYTES, NBUF = FIT < 4 ? FIT : 4;
  static_assert(NBUF >= 2, "two slabs must fit");
  static constexpr int OFF_BARS = NBUF * SLAB_BYTES;
  static constexpr int SMEM = OFF_BARS + 128;
  static constexpr int THREADS = 32 * Cfg::WARPS;
};

struct D3Params {
  int64_t B, rp;             // type states per head, entries per state
  uint32_t slabs;            // heads * slabs_per_head
  int slabs_per_head;
  float* U;                  // [bh][B][rp]
  int* status;
};

template <int EPT> struct Entries;
template <> struct Entries<1> { using T = float; };
template <> struct Entries<2> { using T = float2; };
__device__ __forceinline__ void acc_add(float& a, float v) { a += v; }
__device__ __forceinline__ void acc_add(float2& a, float2 v) { a = __fadd2_rn(a, v); }
__device__ __forceinline__ void acc_zero(float& a) { a = 0.f; }
__device__ __forceinline__ void acc_zero(float2& a) { a = make_float2(0.f, 0.f); }

// Column x2' = J of every slope group: Q values into K accumulators each.
template <int Q, int J, typename V, int N>
__device__ __forceinline__ void d3_column(V (&acc)[N], const uint8_t* col) {
  using L = D3Layout<Q>;
#pragma unroll
  for (int x1 = 0; x1 < Q; ++x1) {
    const V v = *reinterpret_cast<const V*>(col + x1 * L::ROW);
#pragma unroll
    for (int i = 0; i < L::K; ++i) acc_add(acc[i * Q + (x1 + cpow_mod(D3Cfg<Q>::ROOT, i, Q) * J) % Q], v);
  }
}
template <int Q, int J, typename V, int N>
__device__ __forceinline__ void d3_columns(V (&acc)[N], const uint8_t* slab, int inv, int x2) {
  if constexpr (J < Q) {
    d3_column<Q, J>(acc, slab + x2 * (Q * D3Layout<Q>::ROW));
    x2 += inv;
    if (x2 >= Q) x2 -= Q;
    d3_columns<Q, J + 1>(acc, slab, inv, x2);
  }
}

// One heavy task: the K slopes a0 g_i of one slab.  `release` is called between the last read of the slab and the stores.
template <int Q, typename V, typename Release>
__device__ __forceinline__ void d3_heavy_task(const uint8_t* slab, float* u, int64_t rp, int task, Release release) {
  using L = D3Layout<Q>;
  int a0 = 1;                                      // slopes a0 g_i; columns visited in the order x2 = x2' / a0
  for (int i = 0; i < L::K * task; ++i) a0 = (a0 * D3Cfg<Q>::ROOT) % Q;
  int inv = 1;
  for (int i = 0; i < Q - 2; ++i) inv = (inv * a0) % Q;
  V acc[L::K * Q];
#pragma unroll
  for (int i = 0; i < L::K * Q; ++i) acc_zero(acc[i]);
  d3_columns<Q, 0>(acc, slab, inv, 0);
  __syncwarp();
  release();
  int slope = a0;
#pragma unroll
  for (int i = 0; i < L::K; ++i) {
    float* row = u + (int64_t)slope * Q * rp;
#pragma unroll
    for (int b = 0; b < Q; ++b) *reinterpret_cast<V*>(row + b * rp) = acc[i * Q + b];
    slope = (slope * D3Cfg<Q>::ROOT) % Q;
  }
}

// Slope 0, U[b] = Σ_{x2} F[b, x2], and the extra class, U[q² + x2] = Σ_{x1} F[x1, x2].
template <int Q, typename V, typename Release>
__device__ __forceinline__ void d3_light_task(const uint8_t* slab, float* u, int64_t rp, Release release) {
  using L = D3Layout<Q>;
  V acc[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) acc_zero(acc[i]);
#pragma unroll 1
  for (int x2 = 0; x2 < Q; ++x2) {
    V part[2];
    acc_zero(part[0]); acc_zero(part[1]);
#pragma unroll
    for (int x1 = 0; x1 < Q; ++x1) {
      const V v = *reinterpret_cast<const V*>(slab + (x2 * Q + x1) * L::ROW);
      acc_add(acc[x1], v);
      acc_add(part[x1 & 1], v);
    }
    acc_add(part[0], part[1]);
    *reinterpret_cast<V*>(u + (int64_t)(Q * Q + x2) * rp) = part[0];
  }
  __syncwarp();
  release();
#pragma unroll
  for (int b = 0; b < Q; ++b) *reinterpret_cast<V*>(u + b * rp) = acc[b];
}

template <int Q>
__global__ void __launch_bounds__(D3Layout<Q>::THREADS, 1) tabulate_d3_f32_kernel(const __grid_constant__ CUtensorMap tmF,
                                                                        const D3Params prm) {
  using L = D3Layout<Q>;
  using V = typename Entries<L::EPT>::T;
  extern __shared__ __align__(128) uint8_t smem[];   // 128-byte alignment is all the unswizzled boxes need
  constexpr uint32_t NBUF = L::NBUF;
  uint64_t* slab_full = reinterpret_cast<uint64_t*>(smem + L::OFF_BARS);                 // [4] slab landed
  volatile uint32_t* started = reinterpret_cast<volatile uint32_t*>(slab_full + 4);      // [4] last slab whose load went into a buffer
  int* tasks_done = reinterpret_cast<int*>(slab_full + 6);                               // [4] finished tasks of the slab in a buffer
  int* task_counter = tasks_done + 4;
  volatile int* cta_abort = reinterpret_cast<volatile int*>(task_counter + 1);
  const int lane = threadIdx.x & 31;
  const WaitCtx wc{cta_abort, prm.status};
  const uint32_t my_slabs = prm.slabs > blockIdx.x ? (prm.slabs - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  auto start_load = [&](uint32_t ks) {   // slab ks of this CTA into buffer ks % NBUF; one thread calls this
    // (the last heads first: the kernel before has just written them)
    const uint32_t buf = ks % NBUF, slab = prm.slabs - 1 - (blockIdx.x + ks * gridDim.x), head = slab / (uint32_t)prm.slabs_per_head;
    const int e0 = (int)(slab - head * prm.slabs_per_head) * L::ENTRIES;
    started[buf] = ks;
    mbar_expect_tx(slab_full + buf, L::SLAB_BYTES);   // (rows past the last point arrive as zeros)
#pragma unroll
    for (int b = 0; b < L::BOXES; ++b)
      tma_load_3d(smem + buf * L::SLAB_BYTES + b * L::BOX_ROWS * L::ROW, &tmF, e0, b * L::BOX_ROWS, (int)head, slab_full + buf);
  };
  if (threadIdx.x == 0) {
    *cta_abort = 0;
    *task_counter = 0;
    for (uint32_t b = 0; b < NBUF; ++b) {
      tasks_done[b] = 0;
      started[b] = 0xffffffffu;
      mbar_init(slab_full + b, 1);
    }
    fence_barrier_init();
  }
  __syncthreads();
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0)
    for (uint32_t ks = 0; ks < NBUF && ks < my_slabs; ++ks) start_load(ks);
  const uint32_t total = my_slabs * L::TASKS;
  for (;;) {
    uint32_t id = 0;
    if (lane == 0) id = (uint32_t)atomicAdd(task_counter, 1);
    id = __shfl_sync(0xffffffffu, id, 0);
    if (id >= total) break;
    const uint32_t ks = id / L::TASKS, buf = ks % NBUF;
    const int task = (int)(id - ks * L::TASKS);
    const uint32_t slab = prm.slabs - 1 - (blockIdx.x + ks * gridDim.x), head = slab / (uint32_t)prm.slabs_per_head;
    const int64_t e0 = (int64_t)(slab - head * prm.slabs_per_head) * L::ENTRIES + lane * L::EPT;
    float* u = prm.U + (int64_t)head * prm.B * prm.rp + e0;
    // Loads land out of order, and the warps can hold tasks of more than two slabs: a warp may come to wait for a slab
    // while the load before it into the same buffer is still in flight.  The parity wait would pass at once there (it
    // cannot tell the phase before the one in flight from its own), and the early count would start a second load, a
    // second arrival in one phase.  So a warp first waits until its own slab's load has been started, which is after
    // the phase before it has ended.
    // Then every lane waits for the slab itself: all of them read what the copy engine wrote.
    bool ok = true;
    if (lane == 0) {
      const long long since = clock64();
      while (started[buf] != ks && ok) {
        if (*cta_abort) ok = false;
        if (clock64() - since > wc.limit) { *cta_abort = 1; atomicExch(prm.status, 1); ok = false; }
        __nanosleep(100);
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(slab_full + buf, (ks / NBUF) & 1, wc));
    if (!ok) break;
    const uint8_t* mine = smem + buf * L::SLAB_BYTES + lane * (L::EPT * 4);
    // After its last read a task counts itself done; the one that completes the slab's count owns the buffer and starts
    // the load of the slab NBUF further on (every read of the buffer has returned its value by then).
    auto release = [&]() {
      if (lane == 0) {
        __threadfence_block();
        if (atomicAdd(tasks_done + buf, 1) == L::TASKS - 1) {
          tasks_done[buf] = 0;
          fence_proxy_async();
          if (ks + NBUF < my_slabs) start_load(ks + NBUF);
        }
      }
    };
    if (task + 1 < L::TASKS) d3_heavy_task<Q, V>(mine, u, prm.rp, task, release);
    else d3_light_task<Q, V>(mine, u, prm.rp, release);
  }
  if (lane == 0 && *cta_abort)   // waits were given up: the last load into every buffer has landed all the same
    for (uint32_t b = 0; b < NBUF; ++b)
      if (started[b] != 0xffffffffu) landed(slab_full + b, (started[b] / NBUF) & 1, wc);
}

template <int Q>
cudaError_t launch_d3_f32(const float* in, float* out, const SmatGeo& geo, int64_t rp, int bh, int* status, cudaStream_t st) {
  using L = D3Layout<Q>;
  RadonEncodeFn fn = radon_encode_fn();
  if (!fn) return cudaErrorInvalidValue;
  CUtensorMap map;   // (entry, point, head)
  const cuuint64_t dims[3] = {(cuuint64_t)rp, (cuuint64_t)geo.P, (cuuint64_t)bh};
  const cuuint64_t strides[2] = {(cuuint64_t)rp * 4, (cuuint64_t)geo.P * (cuuint64_t)rp * 4};
  const cuuint32_t box[3] = {(cuuint32_t)L::ENTRIES, (cuuint32_t)L::BOX_ROWS, 1}, estr[3] = {1, 1, 1};
  if (fn(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(in), dims, strides, box, estr,
         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  D3Params prm;
  prm.B = geo.B; prm.rp = rp;
  prm.slabs_per_head = (int)(rp / L::ENTRIES);
  prm.slabs = (uint32_t)bh * (uint32_t)prm.slabs_per_head;
  prm.U = out;
  prm.status = status;
  cudaError_t err = cudaFuncSetAttribute(tabulate_d3_f32_kernel<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM);
  if (err != cudaSuccess) return err;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = prm.slabs < (uint32_t)sms ? prm.slabs : (unsigned)sms;
  return smat_launch_pdl(tabulate_d3_f32_kernel<Q>, dim3(grid), L::THREADS, L::SMEM, st, map, prm);
}

}  // namespace

// 1 when the register-resident d = 3 tabulation of fp32 tables covers this geometry.
int smat_tabulate_d3_f32_supported(const SmatGeo& geo, int64_t state_elems) {
  if (geo.D != 2 || state_elems % 64) return 0;
  return geo.q == 11 || geo.q == 13 || geo.q == 17 || geo.q == 19 || geo.q == 23;
}

cudaError_t smat_launch_tabulate_d3_f32(const float* in, float* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                        int* status, cudaStream_t st) {
  if (!smat_tabulate_d3_f32_supported(geo, state_elems)) return cudaErrorInvalidConfiguration;
  switch (geo.q) {
    case 11: return launch_d3_f32<11>(in, out, geo, state_elems, bh, status, st);
    case 13: return launch_d3_f32<13>(in, out, geo, state_elems, bh, status, st);
    case 17: return launch_d3_f32<17>(in, out, geo, state_elems, bh, status, st);
    case 19: return launch_d3_f32<19>(in, out, geo, state_elems, bh, status, st);
    default: return launch_d3_f32<23>(in, out, geo, state_elems, bh, status, st);
  }
}
