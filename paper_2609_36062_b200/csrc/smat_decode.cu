// Cached decoding of the recent block (Sec. "Memory-efficient decoding", Theorem "Streaming decoding"):
// once the distant block has been pooled and tabulated, token t >= n is answered from B + 1 states,
//     S_t = S_{t-1} + k_t v_tᵀ ,   o_t = q_tᵀ (U_type(t) + S_t) ,
// and with scalar gates (Sec. 3.2; the table then holds the keys rescaled to the block boundary)
//     S_t = a_t S_{t-1} + k_t v_tᵀ ,   g_t = a_t g_{t-1} ,   o_t = q_tᵀ (g_t U_type(t) + S_t) ,
// O(r p) work per token and head.  One step reads S and one type state and writes S back: it is a stream over
// 3 states per head, so it runs on the plain ALUs with vectorised loads.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"

namespace {

template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T>
__device__ __forceinline__ void store_out(T* p, float v);
template <>
__device__ __forceinline__ void store_out<float>(float* p, float v) { *p = v; }
template <>
__device__ __forceinline__ void store_out<__nv_bfloat16>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Four consecutive entries of a state, past the L1 cache: nothing of it is read twice in a step.
template <typename TU>
__device__ __forceinline__ float4 load_state4(const TU* p);
template <>
__device__ __forceinline__ float4 load_state4<float>(const float* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
template <>
__device__ __forceinline__ float4 load_state4<__nv_bfloat16>(const __nv_bfloat16* p) {
  uint2 w;
  asm volatile("ld.global.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(w.x), "=r"(w.y) : "l"(p));
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}

// One CTA per head and 32 columns of the state (128 bytes of a row), so that even a handful of sequences spreads over
// the SMs.  Thread (row tid / 8, columns 4 (tid % 8)) walks the rows 32 at a time with every load of its share in
// flight before the first use: a CTA's 24 KB are one round trip to memory.  The partial outputs meet by shuffles and
// one row of shared memory per warp (no atomics: the sum's order is fixed).  Bound by the 84 MB a step of 512 heads
// moves: 14.6 us (12.8 at the HBM rate; 15.7 without the prefetch), where one CTA per head with one row pass in flight at
// a time took 22.1.
constexpr int DEC_COLS = 32, DEC_ROWS = 32, DEC_THREADS = 256;

// TOGETHER: the CTAs of a head are a cluster and none writes o or the running gate before all have read q, k and it (gated
// steps, and o in the place of q or k).
template <typename T, typename TU, int PASSES, bool TOGETHER>
__global__ void __launch_bounds__(DEC_THREADS) decode_step_kernel(const T* q, const T* k,
                                                          const T* v, T* o,
                                                          float* S, const TU* U, int64_t type,
                                                          int64_t types, int p, const float* log_a,
                                                          float* log_g) {
  constexpr int r = PASSES * DEC_ROWS;
  __shared__ float part[DEC_THREADS / 32][DEC_COLS];
  pdl_trigger();
  const int bh = blockIdx.y, tid = threadIdx.x, j0 = blockIdx.x * DEC_COLS;
  const int j = j0 + (tid & 7) * 4, i0 = tid >> 3;
  const TU* Ub = U + ((int64_t)bh * types + type) * r * p;
  // the type state is on its way to L2 while the step before finishes (a hint: it reads nothing)
  if (tid < r) asm volatile("prefetch.global.L2 [%0];" ::"l"(Ub + (int64_t)tid * p + j0));
  pdl_wait();
  float* Sh = S + (int64_t)bh * r * p + j;
  const TU* Uh = Ub + j;
  float4 s[PASSES], u[PASSES];
  float qi[PASSES], ki[PASSES];
#pragma unroll
  for (int n = 0; n < PASSES; ++n) {
    const int64_t off = (int64_t)(n * DEC_ROWS + i0) * p;
    s[n] = load_state4<float>(Sh + off);
    u[n] = load_state4<TU>(Uh + off);
  }
#pragma unroll
  for (int n = 0; n < PASSES; ++n) {
    qi[n] = to_f32(q[(int64_t)bh * r + n * DEC_ROWS + i0]);
    ki[n] = to_f32(k[(int64_t)bh * r + n * DEC_ROWS + i0]);
  }
  const T* vrow = v + (int64_t)bh * p + j;
  const float v0 = to_f32(vrow[0]), v1 = to_f32(vrow[1]), v2 = to_f32(vrow[2]), v3 = to_f32(vrow[3]);
  // gated: a = this token's gate, g = the product of the gates since the block boundary (kept as its logarithm)
  float a = 1.f, g = 1.f;
  float lg = 0.f;
  if (TOGETHER && log_a) { lg = log_g[bh] + log_a[bh]; a = __expf(log_a[bh]); g = __expf(lg); }
  float o4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int n = 0; n < PASSES; ++n) {
    s[n].x = fmaf(ki[n], v0, a * s[n].x); s[n].y = fmaf(ki[n], v1, a * s[n].y);
    s[n].z = fmaf(ki[n], v2, a * s[n].z); s[n].w = fmaf(ki[n], v3, a * s[n].w);
    *reinterpret_cast<float4*>(Sh + (int64_t)(n * DEC_ROWS + i0) * p) = s[n];     // S_t = a_t S_{t-1} + k vᵀ
    o4[0] = fmaf(qi[n], fmaf(g, u[n].x, s[n].x), o4[0]); o4[1] = fmaf(qi[n], fmaf(g, u[n].y, s[n].y), o4[1]);
    o4[2] = fmaf(qi[n], fmaf(g, u[n].z, s[n].z), o4[2]); o4[3] = fmaf(qi[n], fmaf(g, u[n].w, s[n].w), o4[3]);
  }
  if (TOGETHER) asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 4; ++c) {   // the four rows a warp holds in each of its passes
    o4[c] += __shfl_xor_sync(0xffffffffu, o4[c], 8);
    o4[c] += __shfl_xor_sync(0xffffffffu, o4[c], 16);
  }
  if ((tid & 31) < 8) *reinterpret_cast<float4*>(&part[tid >> 5][(tid & 7) * 4]) = make_float4(o4[0], o4[1], o4[2], o4[3]);
  __syncthreads();
  if (TOGETHER) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (tid < DEC_COLS) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < DEC_THREADS / 32; ++w) sum += part[w][tid];
    store_out(o + (int64_t)bh * p + j0 + tid, sum);
  }
  if (TOGETHER && log_a && blockIdx.x == 0 && tid == 0) log_g[bh] = lg;
}

template <typename T, typename TU>
cudaError_t launch_step(const void* q, const void* k, const void* v, void* o, float* S, const void* U, int64_t type,
                        int64_t types, int r, int p, int bh, cudaStream_t st, const float* log_a, float* log_g) {
  const unsigned slices = (unsigned)(p / DEC_COLS);
  // o in the place of q or k (o in the place of v needs nothing: a CTA reads just the columns that it writes)
  const size_t in = (size_t)bh * r * sizeof(T), out = (size_t)bh * p * sizeof(T);
  const bool together = log_a || smat_overlap(o, out, q, in) || smat_overlap(o, out, k, in);
  auto kernel = r == 64 ? (together ? decode_step_kernel<T, TU, 2, true> : decode_step_kernel<T, TU, 2, false>)
                        : (together ? decode_step_kernel<T, TU, 4, true> : decode_step_kernel<T, TU, 4, false>);
  return smat_launch_pdl_cluster(kernel, dim3(slices, (unsigned)bh), DEC_THREADS, 0, together ? slices : 1u, st,
                                 static_cast<const T*>(q), static_cast<const T*>(k), static_cast<const T*>(v),
                                 static_cast<T*>(o), S, static_cast<const TU*>(U), type, types, p, log_a, log_g);
}

}  // namespace

// q, k: [bh][r]; v, o: [bh][p] in the plan's input type; S: [bh][r][p] fp32; U: [bh][types][r][p] (bf16 or fp32).
// Gated step: log_a [bh] = log-gates of this token, log_g [bh] = running log of the gates since the boundary (updated).
cudaError_t smat_launch_decode_step(const void* q, const void* k, const void* v, void* o, float* S, const void* U,
                                    int u_bf16, int in_bf16, int64_t type, int64_t types, int r, int p, int bh,
                                    cudaStream_t st, const float* log_a, float* log_g) {
  if ((r != 64 && r != 128) || (p != 64 && p != 128)) return cudaErrorInvalidValue;
  if (!in_bf16)
    return u_bf16 ? cudaErrorInvalidValue : launch_step<float, float>(q, k, v, o, S, U, type, types, r, p, bh, st, log_a, log_g);
  return u_bf16 ? launch_step<__nv_bfloat16, __nv_bfloat16>(q, k, v, o, S, U, type, types, r, p, bh, st, log_a, log_g)
                : launch_step<__nv_bfloat16, float>(q, k, v, o, S, U, type, types, r, p, bh, st, log_a, log_g);
}
