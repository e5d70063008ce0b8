// Small kernels of the scalar-gated variant (Sec. 3.2, Eq. "gated"; Lemma "Gated SMat"): the prefix sum λ of the
// log-gates, the rescaled copies of Q, K, V, dO that carry the query-side and key-side factors, the decayed scan of the
// chunk states and the gate gradient.  Every factor is the exponential of a difference λ_i - λ_j with j <= i, so it lies
// in (0, 1] and nothing can overflow.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "smat_internal.h"
#include "smat_launch.cuh"

namespace {

// Inclusive prefix (reverse = 0) or suffix (reverse = 1) sum of one row of `len` floats per head; one CTA per head, 4096
// values per turn: a warp scans 128 neighbouring values, the warp totals are scanned by shuffles.  Bound by its few
// dependent steps (32 heads of 4096: 7 us alone, 11 with one value per thread and turn and the totals summed one by one).
__global__ void __launch_bounds__(1024) head_scan_kernel(const float* in, float* out, int64_t len, int reverse) {
  pdl_trigger();
  __shared__ float warp_sum[2][32];
  constexpr int PER = 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* src = in + (int64_t)blockIdx.x * len;
  float* dst = out + (int64_t)blockIdx.x * len;
  float carry = 0.f;
  pdl_wait();
  for (int64_t base = 0, turn = 0; base < len; base += 1024 * PER, turn ^= 1) {
    const int64_t k0 = base + warp * 32 * PER + lane;
    float x[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int64_t k = k0 + 32 * i;
      x[i] = k < len ? src[reverse ? len - 1 - k : k] : 0.f;
    }
    float run = 0.f;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, x[i], d);
        if (lane >= d) x[i] += y;
      }
      x[i] += run;
      run = __shfl_sync(0xffffffffu, x[i], 31);
    }
    if (lane == 31) warp_sum[turn][warp] = run;
    __syncthreads();
    float tot = warp_sum[turn][lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, tot, d);
      if (lane >= d) tot += y;
    }
    // the warps before this one, taken from the scan itself: their sum as (sum through this warp) - (this warp's values)
    // loses the low bits of theirs wherever one strong gate outweighs them, for the tokens before that gate too
    const float prev = __shfl_sync(0xffffffffu, tot, warp ? warp - 1 : 0);
    const float before = carry + (warp ? prev : 0.f);
    carry += __shfl_sync(0xffffffffu, tot, 31);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int64_t k = k0 + 32 * i;
      if (k < len) dst[reverse ? len - 1 - k : k] = before + x[i];
    }
  }
}

// Rescaled copy of token rows: out[t] = src[t] * f(t), dim values per row, in the plan's dtype.
//   mode 0 (query side of a chunk)   : f = exp(λ_t - λ_{s(t)-1}),  s(t) = first token of t's chunk (λ_{-1} = 0)
//   mode 1 (key side of a chunk)     : f = exp(λ_{e(t)} - λ_t),    e(t) = last token of t's chunk
//   mode 2 (the block boundary)      : t <  n: src = A, f = exp(λ_{n-1} - λ_t)   (key side, folded into Z_j)
//                                      t >= n: src = B, f = exp(λ_t - λ_{n-1})   (query side, on the read)
template <typename T>
__global__ void gate_scale_kernel(const T* A, const T* B, T* out,
                                  const float* lam, int mode, int64_t n, int64_t c, int64_t Tlen, int dim,
                                  int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  const int64_t bh = row / Tlen, t = row - bh * Tlen;
  const float* l = lam + bh * Tlen;
  float f;
  const T* src = A;
  if (mode == 0) {
    const int64_t s = t - t % c;
    f = __expf(l[t] - (s > 0 ? l[s - 1] : 0.f));
  } else if (mode == 1) {
    const int64_t e = t - t % c + c - 1;
    f = __expf(l[e] - l[t]);
  } else if (t < n) {
    f = __expf(l[n - 1] - l[t]);
  } else {
    f = __expf(l[t] - l[n - 1]);
    src = B;
  }
  if (dim % 128 == 0) {   // four consecutive elements per lane: 8-byte (bf16) or 16-byte (fp32) accesses
    for (int i = lane * 4; i < dim; i += 128) {
      __align__(16) T v[4];
      if (sizeof(T) == 2) *reinterpret_cast<uint2*>(v) = *reinterpret_cast<const uint2*>(src + row * dim + i);
      else *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(src + row * dim + i);
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = (T)((float)v[k] * f);
      if (sizeof(T) == 2) *reinterpret_cast<uint2*>(out + row * dim + i) = *reinterpret_cast<const uint2*>(v);
      else *reinterpret_cast<uint4*>(out + row * dim + i) = *reinterpret_cast<const uint4*>(v);
    }
    return;
  }
  for (int i = lane; i < dim; i += 32) out[row * dim + i] = (T)((float)src[row * dim + i] * f);
}

// Both rescaled copies a tensor-core pass needs, from one read of their rows (bf16, 128 columns):
//   out1[t] = A[t] * f(t), the query side (mode 0) or key side (mode 1) of t's 128-token tile;
//   out2[t] = (t < n ? B : C)[t] * f(t) at the block boundary (null: d = 1, no long-range branch).
// Sixteen lanes per row, eight rows in flight per warp.  32 heads of 4096 tokens (117 MB): 0.021 ms, where two launches
// with 8 bytes per lane and one row per warp took 0.056.
constexpr int SCALE_ROWS = 4;   // rows per half warp
__device__ __forceinline__ uint4 scale8(const uint4 v, float f) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(__uint_as_float(w[i] << 16) * f, __uint_as_float(w[i] & 0xffff0000u) * f);
    o[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
__global__ void __launch_bounds__(256) gate_scale_pair_kernel(const uint4* A, const uint4* B, const uint4* C, uint4* out1,
                                                              uint4* out2, const float* lam, int mode, int64_t n,
                                                              int64_t Tlen, int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x & 31, col = lane & 15;
  uint4 a[SCALE_ROWS], b[SCALE_ROWS];
  float f1[SCALE_ROWS], f2[SCALE_ROWS];
#pragma unroll
  for (int u = 0; u < SCALE_ROWS; ++u) {
    const int64_t row = (warp * SCALE_ROWS + u) * 2 + (lane >> 4);
    if (row >= rows) continue;
    const int64_t bh = row / Tlen, t = row - bh * Tlen;
    const float* l = lam + bh * Tlen;
    const uint4* src2 = t < n ? B : C;
    a[u] = A[row * 16 + col];
    b[u] = a[u];
    if (out2 && src2 != A) b[u] = src2[row * 16 + col];
    const int64_t t0 = t & ~(int64_t)127;
    f1[u] = mode == 0 ? __expf(l[t] - (t0 > 0 ? l[t0 - 1] : 0.f)) : __expf(l[t0 + 127] - l[t]);
    if (out2) f2[u] = t < n ? __expf(l[n - 1] - l[t]) : __expf(l[t] - l[n - 1]);
  }
#pragma unroll
  for (int u = 0; u < SCALE_ROWS; ++u) {
    const int64_t row = (warp * SCALE_ROWS + u) * 2 + (lane >> 4);
    if (row >= rows) continue;
    out1[row * 16 + col] = scale8(a[u], f1[u]);
    if (out2) out2[row * 16 + col] = scale8(b[u], f2[u]);
  }
}

// Decayed exclusive scan of per-chunk states in place: walking the chunks of a range in order (or in reverse),
//   out[b] = running;  running = γ_b running + in[b],   γ_b = exp(λ_{e(b)} - λ_{s(b)-1}) = the product of chunk b's gates.
// Forward this is S_in (Lemma "Gated SMat": the carried state is decayed by every chunk it passes); in reverse it is the
// adjoint recursion of the same scan.
__global__ void __launch_bounds__(256) gated_scan_kernel(float* S, const float* lam, int64_t state_elems,
                                                         int64_t NC, int64_t c, int64_t lo0, int64_t hi0, int64_t lo1,
                                                         int64_t hi1, int reverse) {
  pdl_trigger();
  pdl_wait();
  const int64_t e4 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e4 * 4 >= state_elems) return;
  const int64_t bh = blockIdx.y;
  const int64_t lo = blockIdx.z ? lo1 : lo0, hi = blockIdx.z ? hi1 : hi0;
  float4* base = reinterpret_cast<float4*>(S + bh * NC * state_elems) + e4;
  const float* l = lam + bh * NC * c;
  const int64_t stride4 = state_elems / 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t k = 0; k < hi - lo; ++k) {
    const int64_t b = reverse ? hi - 1 - k : lo + k;
    const float4 v = base[b * stride4];
    base[b * stride4] = acc;
    const float g = __expf(l[b * c + c - 1] - (b > 0 ? l[b * c - 1] : 0.f));
    acc.x = g * acc.x + v.x; acc.y = g * acc.y + v.y; acc.z = g * acc.z + v.z; acc.w = g * acc.w + v.w;
  }
}

// dλ_t = q_t·dQ_t - k_t·dK_t (every edge's contribution enters once as a query and once as a key); one warp per token.
template <typename T>
__global__ void gate_dlam_kernel(const T* Q, const T* dQ, const T* K,
                                 const T* dK, float* dlam, int dim, int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  float s = 0.f;
  for (int i = lane; i < dim; i += 32)
    s += (float)Q[row * dim + i] * (float)dQ[row * dim + i] - (float)K[row * dim + i] * (float)dK[row * dim + i];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  if (lane == 0) dlam[row] = s;
}

}  // namespace

cudaError_t smat_launch_head_scan(const float* in, float* out, int64_t len, int bh, int reverse, cudaStream_t st) {
  return smat_launch_pdl(head_scan_kernel, dim3((unsigned)bh), 1024, 0, st, in, out, len, reverse);
}

cudaError_t smat_launch_gate_scale(const void* A, const void* B, void* out, const float* lam, int mode, int bf16,
                                   int64_t n, int64_t c, int64_t T, int dim, int bh, cudaStream_t st) {
  const int64_t rows = (int64_t)bh * T;
  const unsigned blocks = (unsigned)((rows * 32 + 255) / 256);
  if (bf16)
    return smat_launch_pdl(gate_scale_kernel<__nv_bfloat16>, dim3(blocks), 256, 0, st, static_cast<const __nv_bfloat16*>(A),
                           static_cast<const __nv_bfloat16*>(B), static_cast<__nv_bfloat16*>(out), lam, mode, n, c, T, dim, rows);
  return smat_launch_pdl(gate_scale_kernel<float>, dim3(blocks), 256, 0, st, static_cast<const float*>(A),
                         static_cast<const float*>(B), static_cast<float*>(out), lam, mode, n, c, T, dim, rows);
}

cudaError_t smat_launch_gate_scale_pair(const void* A, const void* B, const void* C, void* out1, void* out2, const float* lam,
                                        int mode, int64_t n, int64_t T, int bh, cudaStream_t st) {
  const int64_t rows = (int64_t)bh * T, warps = (rows + 2 * SCALE_ROWS - 1) / (2 * SCALE_ROWS);
  return smat_launch_pdl(gate_scale_pair_kernel, dim3((unsigned)((warps + 7) / 8)), 256, 0, st, static_cast<const uint4*>(A),
                         static_cast<const uint4*>(B), static_cast<const uint4*>(C), static_cast<uint4*>(out1),
                         static_cast<uint4*>(out2), lam, mode, n, T, rows);
}

cudaError_t smat_launch_gated_scan(float* S, const float* lam, int64_t state_elems, int64_t NC, int64_t c, int bh,
                                   int64_t lo0, int64_t hi0, int64_t lo1, int64_t hi1, int reverse, cudaStream_t st) {
  const int ranges = (hi1 > lo1) ? 2 : 1;
  dim3 grid((unsigned)((state_elems / 4 + 255) / 256), (unsigned)bh, (unsigned)ranges);
  return smat_launch_pdl(gated_scan_kernel, grid, 256, 0, st, S, lam, state_elems, NC, c, lo0, hi0, lo1, hi1, reverse);
}

cudaError_t smat_launch_gate_dlam(const void* Q, const void* dQ, const void* K, const void* dK, float* dlam, int bf16,
                                  int dim, int64_t T, int bh, cudaStream_t st) {
  const int64_t rows = (int64_t)bh * T;
  const unsigned blocks = (unsigned)((rows * 32 + 255) / 256);
  if (bf16)
    return smat_launch_pdl(gate_dlam_kernel<__nv_bfloat16>, dim3(blocks), 256, 0, st, static_cast<const __nv_bfloat16*>(Q),
                           static_cast<const __nv_bfloat16*>(dQ), static_cast<const __nv_bfloat16*>(K),
                           static_cast<const __nv_bfloat16*>(dK), dlam, dim, rows);
  return smat_launch_pdl(gate_dlam_kernel<float>, dim3(blocks), 256, 0, st, static_cast<const float*>(Q),
                         static_cast<const float*>(dQ), static_cast<const float*>(K), static_cast<const float*>(dK), dlam, dim,
                         rows);
}

// ---- normalised output (Sec. 2: augmented value v̄ = [v; 1], one final division) ------------------------------------
namespace {

// Four consecutive elements of a row, as one 8-byte (bf16) or 16-byte (fp32) access.
template <typename T>
struct Quad {
  __align__(16) T v[4];
  __device__ __forceinline__ void load(const T* src) {
    if (sizeof(T) == 2) *reinterpret_cast<uint2*>(v) = *reinterpret_cast<const uint2*>(src);
    else *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(src);
  }
  __device__ __forceinline__ void store(T* dst) const {
    if (sizeof(T) == 2) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(v);
    else *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(v);
  }
};

// The three row kernels below take one warp per row; rows whose length is a multiple of 128 move four elements per lane
// and access (the elementwise form was bound by its 2-byte accesses and per-element index arithmetic).

// V̄ = V with its last column set to one.
template <typename T>
__global__ void augment_value_kernel(const T* V, T* Vbar, int p, int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  if (p % 128 == 0) {
    for (int i = lane * 4; i < p; i += 128) {
      Quad<T> q;
      q.load(V + row * p + i);
      if (i + 4 == p) q.v[3] = (T)1.0f;
      q.store(Vbar + row * p + i);
    }
    return;
  }
  for (int i = lane; i < p; i += 32) Vbar[row * p + i] = i == p - 1 ? (T)1.0f : V[row * p + i];
}

// O = ȳ_{1:p-1} / ȳ_p, and the normaliser ȳ_p itself in the last column.  One warp per row.
template <typename T>
__global__ void normalize_rows_kernel(const T* Y, T* O, int p, int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  const float den = (float)Y[row * p + p - 1];
  const float inv = 1.0f / den;
  if (p % 128 == 0) {
    for (int i = lane * 4; i < p; i += 128) {
      Quad<T> q;
      q.load(Y + row * p + i);
#pragma unroll
      for (int k = 0; k < 4; ++k) q.v[k] = i + k == p - 1 ? (T)den : (T)((float)q.v[k] * inv);
      q.store(O + row * p + i);
    }
    return;
  }
  for (int i = lane; i < p; i += 32) O[row * p + i] = i == p - 1 ? (T)den : (T)((float)Y[row * p + i] * inv);
}

// Upstream of the linear pass from the upstream of the normalised output (the backward of the final division):
//   dȳ_c = dO_c / z (c < p-1),   dȳ_p = dO_p - Σ_{c<p-1} dO_c O_c / z,   z = the normaliser kept in O's last column.
template <typename T>
__global__ void normalize_adjoint_kernel(const T* O, const T* dO, T* dY, int p,
                                         int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  const float inv = 1.0f / (float)O[row * p + p - 1];
  float dot = 0.f;
  if (p % 128 == 0) {
    float last = 0.f;   // dO of the normaliser column (held by the lane that owns the row's last quad)
    for (int i = lane * 4; i < p; i += 128) {
      Quad<T> g, o;
      g.load(dO + row * p + i);
      o.load(O + row * p + i);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (i + k == p - 1) { last = (float)g.v[k]; continue; }
        dot += (float)g.v[k] * (float)o.v[k];
        g.v[k] = (T)((float)g.v[k] * inv);
      }
      if (i + 4 != p) g.store(dY + row * p + i);
      else {   // the last quad waits for the row's dot product
#pragma unroll
        for (int k = 0; k < 3; ++k) dY[row * p + i + k] = g.v[k];
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, d);
    if (lane == ((p - 4) % 128) / 4) dY[row * p + p - 1] = (T)(last - dot * inv);
    return;
  }
  for (int i = lane; i < p - 1; i += 32) {
    const float g = (float)dO[row * p + i];
    dot += g * (float)O[row * p + i];
    dY[row * p + i] = (T)(g * inv);
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, d);
  if (lane == 0) dY[row * p + p - 1] = (T)((float)dO[row * p + p - 1] - dot * inv);
}

// The ones column of V̄ is a constant: its gradient is dropped.
template <typename T>
__global__ void clear_last_column_kernel(T* dV, int p, int64_t rows) {
  pdl_trigger();
  pdl_wait();
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row < rows) dV[row * p + p - 1] = (T)0.0f;
}

template <typename T>
cudaError_t normalize_step(int step, const void* a, const void* b, void* out, int p, int64_t rows, cudaStream_t st) {
  const unsigned warp_blocks = (unsigned)((rows * 32 + 255) / 256);
  if (step == 0)
    return smat_launch_pdl(augment_value_kernel<T>, dim3(warp_blocks), 256, 0, st, static_cast<const T*>(a),
                           static_cast<T*>(out), p, rows);
  if (step == 1)
    return smat_launch_pdl(normalize_rows_kernel<T>, dim3(warp_blocks), 256, 0, st, static_cast<const T*>(a),
                           static_cast<T*>(out), p, rows);
  if (step == 2)
    return smat_launch_pdl(normalize_adjoint_kernel<T>, dim3(warp_blocks), 256, 0, st, static_cast<const T*>(a),
                           static_cast<const T*>(b), static_cast<T*>(out), p, rows);
  return smat_launch_pdl(clear_last_column_kernel<T>, dim3((unsigned)((rows + 255) / 256)), 256, 0, st, static_cast<T*>(out),
                         p, rows);
}

}  // namespace

// step 0: out = V̄ from a = V;  1: out = O from a = ȳ;  2: out = dȳ from a = O, b = dO;  3: out (dV) last column := 0
cudaError_t smat_launch_normalize_step(int step, const void* a, const void* b, void* out, int bf16, int p, int64_t rows,
                                       cudaStream_t st) {
  return bf16 ? normalize_step<__nv_bfloat16>(step, a, b, out, p, rows, st) : normalize_step<float>(step, a, b, out, p, rows, st);
}
