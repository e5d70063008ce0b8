// fp32-ALU kernels of libsmat: the within-chunk tiles of the forward and of the backward pass when no tensor-core
// kernel applies (fp32 inputs, other head widths), the chunk-state scans, the direct form of Algorithm 2 and its
// transpose, and the debug mask.
#include <cuda_bf16.h>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_scan.cuh"
#include "smat_tc.cuh"

namespace {

using tc::cp_async16;
using tc::cp_async_commit;
using tc::cp_async_wait;

// ---- within-chunk tiles ------------------------------------------------------------------------------------------
// Out[i] = Σ_j X_ij P3_j + P4_i · St (+ addend row),   X_ij = P1_i · P2_j where j <= i (upper: j >= i) in i's chunk:
//     O  : P1 = Q,  P2 = K,  P3 = V,  P4 = Q,  St = S_in              dQ : P1 = dO, P2 = V,  P3 = K,  P4 = dO, St = S_inᵀ
//     dK : P1 = V,  P2 = dO, P3 = Q,  P4 = V,  St = D̄ᵀ (upper)        dV : P1 = K,  P2 = Q,  P3 = dO, P4 = K,  St = D̄ (upper)
// (Eq. "local", Eq. "local-adjoint" with the broadcast of the scanned states.)  A CTA takes 32 or 16 rows of one chunk: the
// scores of 64 columns at a time go through shared memory, two operand buffers alternate between the next columns'
// P2 / P3 and the 64-row pieces of the state, fetched while the other one is used.  Everything is fp32.
// One launch serves the forward tile, or the three adjoints (jobs).  What it replaces — scores, state product and
// tile product as separate launches of a general 64 x 64 product, with the score tiles in memory — took 21 launches
// and 259 us for forward + backward of one 512-token head (64 wide, chunk 64).
constexpr int COLS = 64;      // score columns per step, and rows of a state piece
constexpr int TILE_THREADS = 256;

template <typename T, int SD, int OD, int ROWS>
struct TileLayout {
  static constexpr int SROW = SD * (int)sizeof(T) + 16;   // bytes per staged row (padded by one 16-byte chunk)
  static constexpr int OROW = OD * (int)sizeof(T) + 16;
  static constexpr int STROW = OD * 4 + 16;               // one row of a state piece [k][n]
  static constexpr int BUF = COLS * STROW > COLS * (SROW > OROW ? SROW : OROW) ? COLS * STROW : COLS * (SROW > OROW ? SROW : OROW);
  static constexpr int XROW = COLS + 4;                   // floats
  static constexpr int OFF_P4 = ROWS * SROW;
  static constexpr int OFF_A = 2 * ROWS * SROW;
  static constexpr int OFF_B = OFF_A + BUF;
  static constexpr int OFF_X = OFF_B + BUF;
  static constexpr int SMEM = OFF_X + ROWS * XROW * 4;
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void st4(float* p, const float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16* p, const float4 v) {
  *reinterpret_cast<uint2*>(p) = make_uint2(tc::pack_bf16(v.x, v.y), tc::pack_bf16(v.z, v.w));
}
__device__ __forceinline__ float dot4(const float4 a, const float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
__device__ __forceinline__ float4 fma4(float s, const float4 b, float4 a) {
  a.x = fmaf(s, b.x, a.x); a.y = fmaf(s, b.y, a.y); a.z = fmaf(s, b.z, a.z); a.w = fmaf(s, b.w, a.w);
  return a;
}

template <typename T, int SD, int OD, int ROWS>
__global__ void __launch_bounds__(TILE_THREADS, 2) tile_rows_kernel(const __grid_constant__ SmatTileArgs a) {
  using L = TileLayout<T, SD, OD, ROWS>;
  constexpr int SR = ROWS / 16;   // score rows per thread
  extern __shared__ __align__(16) uint8_t smem[];
  pdl_trigger();
  uint8_t *s1 = smem, *s4 = smem + L::OFF_P4, *sA = smem + L::OFF_A, *sB = smem + L::OFF_B;
  float* sX = reinterpret_cast<float*>(smem + L::OFF_X);
  const int blocks = (a.c + ROWS - 1) / ROWS;                 // row blocks of a chunk
  const int per_job = a.NC * blocks;
  const int which = blockIdx.x / per_job, rest = blockIdx.x - which * per_job;
  const SmatTileJob& job = a.job[which];
  const int chunk = rest / blocks, m0 = (rest - chunk * blocks) * ROWS;
  const int64_t bh = blockIdx.y;
  const int rows = a.c - m0 < ROWS ? a.c - m0 : ROWS;
  const int64_t t0 = (int64_t)chunk * a.c;                    // first token of the chunk
  const int64_t row0 = bh * a.T + t0;
  const int tid = threadIdx.x;
  constexpr int OC = OD / 4, RG = TILE_THREADS / OC, RPT = ROWS / RG;   // output columns / 4, row groups, rows per thread
  const int oc = tid % OC, rg = tid / OC;

  auto stage_rows = [&](uint8_t* dst, const void* src, int first, int count, int dim, int pitch) {
    const int chunks = dim * (int)sizeof(T) / 16;
    const uint8_t* base = static_cast<const uint8_t*>(src) + (row0 + first) * dim * (int64_t)sizeof(T);
    for (int i = tid; i < count * chunks; i += TILE_THREADS) {
      const int r = i / chunks, ch = i - r * chunks;
      cp_async16(dst + r * pitch + ch * 16, base + (int64_t)i * 16);
    }
  };
  const float* st = job.st + (bh * a.NC + chunk) * (int64_t)(SD * OD);
  // 64 rows of the state as the product reads it ([k][n], n contiguous)
  auto stage_state = [&](uint8_t* dst, int piece) {
    if (!job.st_trans) {
      for (int i = tid; i < COLS * OC; i += TILE_THREADS) {
        const int k = i / OC, ch = i - k * OC;
        cp_async16(dst + k * L::STROW + ch * 16, st + (int64_t)(piece * COLS + k) * OD + ch * 4);
      }
    } else {   // stored [n][k]: neighbouring lanes take neighbouring n, so that the scattered words hit different banks
      float* d = reinterpret_cast<float*>(dst);
      constexpr int PER = COLS / 4 * OD / TILE_THREADS;
      float4 v[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int i = tid + u * TILE_THREADS, n = i % OD, k4 = i / OD;
        v[u] = ld4(st + (int64_t)n * SD + piece * COLS + k4 * 4);
      }
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int i = tid + u * TILE_THREADS, n = i % OD, k4 = i / OD;
        float* p = d + (k4 * 4) * (L::STROW / 4) + n;
        p[0] = v[u].x; p[L::STROW / 4] = v[u].y; p[2 * (L::STROW / 4)] = v[u].z; p[3 * (L::STROW / 4)] = v[u].w;
      }
    }
  };
  const int kb0 = job.upper ? m0 / COLS : 0;
  const int kb1 = job.upper ? (a.c - 1) / COLS : (m0 + rows - 1) / COLS;
  auto cols_of = [&](int kb) { return a.c - kb * COLS < COLS ? a.c - kb * COLS : COLS; };
  const bool own4 = job.p4 != job.p1;
  float4 acc[RPT];
#pragma unroll
  for (int r = 0; r < RPT; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);

  pdl_wait();
  stage_rows(s1, job.p1, m0, rows, SD, L::SROW);
  if (own4) stage_rows(s4, job.p4, m0, rows, SD, L::SROW);
  stage_rows(sA, job.p2, kb0 * COLS, cols_of(kb0), SD, L::SROW);
  cp_async_commit();
  stage_rows(sB, job.p3, kb0 * COLS, cols_of(kb0), OD, L::OROW);
  cp_async_commit();
  for (int kb = kb0; kb <= kb1; ++kb) {
    const int cols = cols_of(kb);
    cp_async_wait<1>();
    __syncthreads();
    {   // scores: SR rows x four columns per thread
      const int ty = tid >> 4, tx = tid & 15;
      float x[SR][4];
#pragma unroll
      for (int i = 0; i < SR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) x[i][j] = 0.f;
#pragma unroll 4
      for (int k = 0; k < SD; k += 4) {
        float4 av[SR], bv[4];
#pragma unroll
        for (int i = 0; i < SR; ++i) av[i] = ld4(reinterpret_cast<const T*>(s1 + (ty * SR + i) * L::SROW) + k);
#pragma unroll
        for (int j = 0; j < 4; ++j) bv[j] = ld4(reinterpret_cast<const T*>(sA + (tx + 16 * j) * L::SROW) + k);
#pragma unroll
        for (int i = 0; i < SR; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) x[i][j] = dot4(av[i], bv[j], x[i][j]);
      }
#pragma unroll
      for (int i = 0; i < SR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int m = m0 + ty * SR + i, n = kb * COLS + tx + 16 * j;   // positions inside the chunk
          const bool in = m < a.c && n < a.c && (job.upper ? n >= m : n <= m);
          float v = in ? x[i][j] : 0.f;
          if (a.lam && in) {   // gated: decay between the key's and the query's position
            const float* l = a.lam + row0;
            v *= job.upper ? __expf(l[n] - l[m]) : __expf(l[m] - l[n]);
          }
          sX[(ty * SR + i) * L::XROW + tx + 16 * j] = v;
        }
    }
    __syncthreads();
    if (kb < kb1) stage_rows(sA, job.p2, (kb + 1) * COLS, cols_of(kb + 1), SD, L::SROW);
    else stage_state(sA, 0);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < cols; k += 4) {
      float4 xv[RPT], bv[4];
#pragma unroll
      for (int r = 0; r < RPT; ++r) xv[r] = ld4(sX + (rg * RPT + r) * L::XROW + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = ld4(reinterpret_cast<const T*>(sB + (k + j) * L::OROW) + oc * 4);
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        acc[r] = fma4(xv[r].x, bv[0], acc[r]); acc[r] = fma4(xv[r].y, bv[1], acc[r]);
        acc[r] = fma4(xv[r].z, bv[2], acc[r]); acc[r] = fma4(xv[r].w, bv[3], acc[r]);
      }
    }
    __syncthreads();
    if (kb < kb1) stage_rows(sB, job.p3, (kb + 1) * COLS, cols_of(kb + 1), OD, L::OROW);
    else if (SD > COLS) stage_state(sB, 1);
    cp_async_commit();
  }
#pragma unroll
  for (int piece = 0; piece < SD / COLS; ++piece) {
    if (piece == 0) cp_async_wait<1>(); else cp_async_wait<0>();
    __syncthreads();
    const uint8_t* sp = own4 ? s4 : s1;
    const uint8_t* buf = piece ? sB : sA;
#pragma unroll 4
    for (int k = 0; k < COLS; k += 4) {
      float4 av[RPT], bv[4];
#pragma unroll
      for (int r = 0; r < RPT; ++r) av[r] = ld4(reinterpret_cast<const T*>(sp + (rg * RPT + r) * L::SROW) + piece * COLS + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = ld4(reinterpret_cast<const float*>(buf + (k + j) * L::STROW) + oc * 4);
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        acc[r] = fma4(av[r].x, bv[0], acc[r]); acc[r] = fma4(av[r].y, bv[1], acc[r]);
        acc[r] = fma4(av[r].z, bv[2], acc[r]); acc[r] = fma4(av[r].w, bv[3], acc[r]);
      }
    }
  }
  // out in the place of P2 or P3, whose rows every row block of the chunk reads: the blocks are a cluster then, and none
  // stores before all have read
  if (a.together) asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
#pragma unroll
  for (int r = 0; r < RPT; ++r) {
    const int m = rg * RPT + r;
    if (m >= rows) continue;
    const int64_t t = t0 + m0 + m, off = (bh * a.T + t) * OD + oc * 4;
    float4 v = acc[r];
    if (t >= job.acc_lo && t < job.acc_hi) {
      const float4 y = ld4(job.acc + off);
      v.x += y.x; v.y += y.y; v.z += y.z; v.w += y.w;
    }
    st4(static_cast<T*>(job.out) + off, v);
  }
}

// ---- scan --------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) scan_kernel(const __grid_constant__ SmatScanArgs a, int64_t state_elems, int64_t NC) {
  pdl_trigger();
  pdl_wait();
  smat_scan_entries(a, state_elems, NC, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y, blockIdx.z);
}

// ---- Algorithm 2, direct form ------------------------------------------------------------------------
// The CTA copies its slab (E consecutive state entries) of all input states into shared memory, then
// every (output state, entry) pair is summed by one thread.  Offsets aᵀx are maintained by a base-q
// counter: bumping a digit q times returns the running dot product to where it started, so a carry
// needs no correction.
__global__ void __launch_bounds__(256) tabulate_alg2_kernel(const float* __restrict__ in, float* __restrict__ out,
                                                            const SmatGeo geo, int64_t state_elems, int E,
                                                            int transpose) {
  extern __shared__ __align__(16) float slab[];
  const int64_t rows_in = transpose ? geo.B : geo.P;
  const int64_t rows_out = transpose ? geo.P : geo.B;
  const int64_t bh = blockIdx.y;
  const int64_t e0 = (int64_t)blockIdx.x * E;
  const float* src = in + bh * rows_in * state_elems + e0;
  for (int64_t idx = threadIdx.x; idx < rows_in * E; idx += blockDim.x) {
    const int64_t x = idx / E;
    const int e = (int)(idx - x * E);
    slab[idx] = src[x * state_elems + e];
  }
  __syncthreads();
  float* dst = out + bh * rows_out * state_elems + e0;
  const int q = geo.q, D = geo.D;
  for (int64_t item = threadIdx.x; item < rows_out * E; item += blockDim.x) {
    const int64_t row = item / E;
    const int e = (int)(item - row * E);
    float sum = 0.f;
    if (!transpose) {
      // hyperplane `row` = (direction a, offset b): visit its q^(D-1) points
      int32_t a[SMAT_MAX_DIM];
      smat_direction(geo, row / q, a);
      const int b = (int)(row % q);
      int lead = 0;
      while (a[lead] == 0) ++lead;
      int digit[SMAT_MAX_DIM];
      for (int k = 0; k < D; ++k) digit[k] = 0;
      int s = 0;        // Σ over free coordinates of a_k x_k  (mod q)
      int64_t v = 0;    // packed index of the free coordinates
      const int64_t npts = geo.qpow[D - 1];
      for (int64_t it = 0; it < npts; ++it) {
        int xl = b - s;
        if (xl < 0) xl += q;
        sum += slab[(v + (int64_t)xl * geo.qpow[lead]) * E + e];
        for (int k = 0; k < D; ++k) {  // bump the counter over the free coordinates
          if (k == lead) continue;
          s += a[k];
          if (s >= q) s -= q;
          v += geo.qpow[k];
          if (++digit[k] < q) break;
          digit[k] = 0;
          v -= geo.qpow[k + 1];
        }
      }
    } else {
      // point `row`: one hyperplane per direction, offset aᵀx
      int x[SMAT_MAX_DIM];
      int64_t vv = row;
      for (int k = 0; k < D; ++k) { x[k] = (int)(vv % q); vv /= q; }
      for (int lead = 0; lead < D; ++lead) {
        int digit[SMAT_MAX_DIM];
        for (int k = 0; k < D; ++k) digit[k] = 0;
        int dot = x[lead];
        int64_t dir = geo.dir_group_start[lead];
        const int64_t ndir = geo.qpow[D - 1 - lead];
        for (int64_t it = 0; it < ndir; ++it, ++dir) {
          sum += slab[(dir * q + dot) * E + e];
          for (int k = lead + 1; k < D; ++k) {
            dot += x[k];
            if (dot >= q) dot -= q;
            if (++digit[k] < q) break;
            digit[k] = 0;
          }
        }
      }
    }
    dst[row * state_elems + e] = sum;
  }
}

__global__ void mask_kernel(uint8_t* mask, const SmatGeo geo) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= geo.T * geo.T) return;
  mask[idx] = (uint8_t)smat_mask_entry(geo, idx / geo.T, idx % geo.T);
}

}  // namespace

template <typename T, int SD, int OD, int ROWS>
static cudaError_t launch_tile_rows_of(SmatTileArgs a, int bh, cudaStream_t st) {
  const unsigned blocks = (unsigned)((a.c + ROWS - 1) / ROWS);
  const int smem = smat_smem_alone((int64_t)a.jobs * a.NC * blocks * bh, TileLayout<T, SD, OD, ROWS>::SMEM);
  cudaError_t err = cudaFuncSetAttribute(tile_rows_kernel<T, SD, OD, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (err != cudaSuccess) return err;
  const size_t rows = (size_t)bh * a.T * sizeof(T);
  a.together = 0;
  for (int j = 0; j < a.jobs; ++j)
    if (smat_overlap(a.job[j].out, rows * OD, a.job[j].p2, rows * SD) || smat_overlap(a.job[j].out, rows * OD, a.job[j].p3, rows * OD))
      a.together = 1;
  const dim3 grid((unsigned)(a.jobs * a.NC) * blocks, (unsigned)bh);
  return smat_launch_pdl_cluster(tile_rows_kernel<T, SD, OD, ROWS>, grid, TILE_THREADS, smem, a.together ? blocks : 1u, st, a);
}

// 32 rows to a CTA, or 16 while that leaves SMs idle: half the work on the path of a launch that is one round of CTAs.
template <typename T, int SD, int OD>
static cudaError_t launch_tile_rows(const SmatTileArgs& a, int bh, cudaStream_t st) {
  const int64_t ctas = (int64_t)a.jobs * a.NC * ((a.c + 15) / 16) * bh;
  return ctas <= smat_sm_count() ? launch_tile_rows_of<T, SD, OD, 16>(a, bh, st) : launch_tile_rows_of<T, SD, OD, 32>(a, bh, st);
}

cudaError_t smat_launch_tile_rows(const SmatTileArgs& a, int bf16, int score_dim, int out_dim, int bh, cudaStream_t st) {
#define SMAT_TILE(SV, OV)                                                                                     \
  if (score_dim == SV && out_dim == OV)                                                                       \
    return bf16 ? launch_tile_rows<__nv_bfloat16, SV, OV>(a, bh, st) : launch_tile_rows<float, SV, OV>(a, bh, st);
  SMAT_TILE(64, 64) SMAT_TILE(64, 128) SMAT_TILE(128, 64) SMAT_TILE(128, 128)
#undef SMAT_TILE
  return cudaErrorInvalidValue;
}

cudaError_t smat_launch_scan(const SmatScanArgs& a, int64_t state_elems, int64_t NC, int bh, cudaStream_t st) {
  const dim3 grid((unsigned)((state_elems / 4 + 255) / 256), (unsigned)bh, (unsigned)(2 * a.jobs));
  return smat_launch_pdl(scan_kernel, grid, 256, 0, st, a, state_elems, NC);
}

int smat_tabulate_alg2_slab(int64_t rows_in, int64_t state_elems) {
  const int64_t budget = 200 * 1024;
  int E = 128;
  while (E >= 1 && (rows_in * E * 4 > budget || state_elems % E != 0)) E >>= 1;
  return E;
}

cudaError_t smat_launch_tabulate_alg2(const float* in, float* out, const SmatGeo& geo, int64_t state_elems, int bh,
                                      int transpose, cudaStream_t st) {
  const int64_t rows_in = transpose ? geo.B : geo.P;
  const int E = smat_tabulate_alg2_slab(rows_in, state_elems);
  if (E < 1) return cudaErrorInvalidConfiguration;
  const size_t smem = (size_t)rows_in * E * sizeof(float);
  cudaError_t err = cudaFuncSetAttribute(tabulate_alg2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  dim3 grid((unsigned)(state_elems / E), (unsigned)bh);
  tabulate_alg2_kernel<<<grid, 256, smem, st>>>(in, out, geo, state_elems, E, transpose);
  return cudaGetLastError();
}

cudaError_t smat_launch_mask(uint8_t* mask, const SmatGeo& geo, cudaStream_t st) {
  const int64_t total = geo.T * geo.T;
  mask_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(mask, geo);
  return cudaGetLastError();
}
