// HBM-streaming kernels of the long-range branch, written as persistent CTAs around bulk asynchronous
// copies (TMA, one-dimensional, no multicast):
//   pool_stream_kernel       : state[g] = Σ_{tokens of g} a_tᵀ b_t ; each finished 64 KB state leaves through a
//                              bulk store while the next group's tokens are already in flight        (Algorithm 1, step 2)
//   state_read_stream_kernel : out[t] = x_t · state[g(t)] for the few tokens of every group; states arrive through
//                              bulk loads                                                             (Algorithm 1, step 4)
// Both are bound by the one pass over the table they write or read.
#include <cuda_bf16.h>

#include <type_traits>

#include "smat_internal.h"
#include "smat_launch.cuh"
#include "smat_scan.cuh"
#include "smat_tc.cuh"

namespace {

using tc::smem_u32;

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ float4 fma4(float s, const float4 b, float4 a) {
  a.x = fmaf(s, b.x, a.x); a.y = fmaf(s, b.y, a.y); a.z = fmaf(s, b.z, a.z); a.w = fmaf(s, b.w, a.w);
  return a;
}
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&raw.x);
  const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&raw.y);
  return make_float4(__low2float(lo), __high2float(lo), __low2float(hi), __high2float(hi));
}

using tc::bulk_load;
using tc::cp_async16;
using tc::cp_async_commit;
using tc::cp_async_wait;

__device__ __forceinline__ void bulk_store(void* gmem, const void* smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gmem), "r"(smem_u32(smem)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void bulk_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// ---- pooling ----------------------------------------------------------------------------------------------------
// The items of all jobs in one list: job j's (head, group) pairs follow those of job j - 1.
struct PoolList {
  SmatPoolArgs a;
  int64_t first[5];        // first item of job j; first[jobs] = all items
};

// One pass of the kernel: up to TK tokens of one item.
template <int TK>
struct PoolCursor {
  const PoolList* l;
  int64_t item, stride;
  int job;
  int64_t bh, k0, cnt;
  SmatTokens tk;
  __device__ PoolCursor(const PoolList& list, int64_t first, int64_t step) : l(&list), item(first), stride(step) { load(); }
  __device__ bool valid() const { return item < l->first[l->a.jobs]; }
  __device__ void load() {
    k0 = 0; cnt = 0; job = 0;
    if (!valid()) return;
    while (item >= l->first[job + 1]) ++job;
    const int64_t at = item - l->first[job];
    bh = smat_div(at, l->a.job[job].groups);
    tk = smat_group_tokens(l->a.job[job].grp, bh, at - bh * l->a.job[job].groups);
    cnt = tk.cnt;
  }
  __device__ bool last() const { return k0 + TK >= cnt; }
  __device__ int tokens() const { const int64_t left = cnt - k0; return (int)(left < TK ? (left > 0 ? left : 0) : TK); }
  __device__ void next() {
    if (last()) { item += stride; load(); } else k0 += TK;
  }
};

// Two token buffers alternate over the passes, also inside a group of many tokens: the next pass's rows (of the same
// group or of the next item) travel while this pass is summed.
// clear (or null): the status word (and the mark behind it) of a pass that begins with this launch, which waits for nothing that could fail.
// TK: tokens staged per pass.
template <int R, int PD, typename T, int TK>
__global__ void __launch_bounds__(256) pool_stream_kernel(const __grid_constant__ PoolList list, int64_t Tlen, int* clear) {
  constexpr int NJ4 = PD / 4;
  constexpr int NG = 256 / NJ4;
  constexpr int NS = R / NG;
  constexpr int RC = R * (int)sizeof(T) / 16, PC = PD * (int)sizeof(T) / 16;  // 16-byte chunks per row
  extern __shared__ __align__(128) uint8_t smem_raw[];
  float* outb = reinterpret_cast<float*>(smem_raw);                  // [R*PD]
  T* a_raw = reinterpret_cast<T*>(smem_raw + R * PD * 4);            // [2][TK][R]
  T* b_raw = a_raw + 2 * TK * R;                                     // [2][TK][PD]
  pdl_trigger();
  const int tid = threadIdx.x;
  const int j4 = tid % NJ4, ig = tid / NJ4;

  auto fetch = [&](const PoolCursor<TK>& c, int buf) {
    if (c.valid()) {
      const int kn = c.tokens();
      const T* Ab = static_cast<const T*>(list.a.job[c.job].a) + c.bh * Tlen * R;
      const T* Bb = static_cast<const T*>(list.a.job[c.job].b) + c.bh * Tlen * PD;
      for (int idx = tid; idx < kn * RC; idx += 256) {
        const int k = idx / RC, ch = idx - k * RC;
        cp_async16(reinterpret_cast<uint8_t*>(a_raw + (buf * TK + k) * R) + ch * 16,
                   reinterpret_cast<const uint8_t*>(Ab + c.tk.at(c.k0 + k) * R) + ch * 16);
      }
      for (int idx = tid; idx < kn * PC; idx += 256) {
        const int k = idx / PC, ch = idx - k * PC;
        cp_async16(reinterpret_cast<uint8_t*>(b_raw + (buf * TK + k) * PD) + ch * 16,
                   reinterpret_cast<const uint8_t*>(Bb + c.tk.at(c.k0 + k) * PD) + ch * 16);
      }
    }
    cp_async_commit();
  };

  pdl_wait();   // (the token lists of a routed call come from the kernel before)
  if (clear && blockIdx.x == 0 && tid == 0) clear[0] = clear[1] = 0;
  PoolCursor<TK> cur(list, blockIdx.x, gridDim.x);
  fetch(cur, 0);
  float4 acc[NS];
  for (int n = 0; cur.valid(); ++n) {
    const int buf = n & 1;
    PoolCursor<TK> nxt = cur;
    nxt.next();
    fetch(nxt, buf ^ 1);
    cp_async_wait<1>();
    __syncthreads();
    if (cur.k0 == 0) {
#pragma unroll
      for (int s = 0; s < NS; ++s) acc[s] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int kn = cur.tokens();
    const T* as = a_raw + buf * TK * R;
    const T* bs = b_raw + buf * TK * PD;
    // a thread owns NS neighbouring rows, so that their factors come four to a load (one by one they took as many
    // shared-memory cycles as everything else: 32 heads, 289 states of 9 tokens, 0.138 ms against 0.122)
    for (int k = 0; k < kn; ++k) {
      const float4 b4 = load4(bs + k * PD + j4 * 4);
#pragma unroll
      for (int s = 0; s < NS; s += 4) {
        const float4 a4 = load4(as + k * R + ig * NS + s);
        acc[s] = fma4(a4.x, b4, acc[s]); acc[s + 1] = fma4(a4.y, b4, acc[s + 1]);
        acc[s + 2] = fma4(a4.z, b4, acc[s + 2]); acc[s + 3] = fma4(a4.w, b4, acc[s + 3]);
      }
    }
    if (cur.last()) {
      // the previous item's bulk store reads the same buffer: it must have finished reading (the other CTA
      // resident on this SM keeps the memory pipe busy meanwhile)
      if (tid == 0) bulk_store_wait_read<0>();
      __syncthreads();
#pragma unroll
      for (int s = 0; s < NS; ++s) *reinterpret_cast<float4*>(outb + (ig * NS + s) * PD + j4 * 4) = acc[s];
      tc::fence_proxy_async();
      __syncthreads();
      if (tid == 0) bulk_store(list.a.job[cur.job].state + (cur.item - list.first[cur.job]) * (int64_t)(R * PD), outb, R * PD * 4);
    } else {
      __syncthreads();   // the buffer just read is the next fetch's target
    }
    cur = nxt;
  }
  if (tid == 0) bulk_store_wait_all();
  cp_async_wait<0>();
}

// ---- routed read ----------------------------------------------------------------------------------------------------
struct ReadList {
  SmatReadArgs a;
  int64_t first[4];
  // Chunk states that the tile kernel behind the read will want scanned: the first scan_ctas CTAs of the launch do that, where
  // the pass is a sequence of launches of a few CTAs each and bound by their number.
  SmatScanArgs scan;
  int64_t NC;
  int32_t scan_x, scan_y, scan_ctas;   // CTAs per head and (job, range); heads; all of them
};

// Two CTAs share an SM; each owns one 64 KB state buffer, so one CTA's contraction overlaps the other's bulk load.  A state
// of 32 KB or more arrives in two halves of rows.  Where a group is one pass of five to eight tokens they are contracted one
// after the other, and the next state's first half is fetched in between (d = 3, seven or eight tokens to a group, bf16 with
// fp32 tables, heads of 2688 tokens: 24 of them 263 -> 258 us a pass, 8 of them 116.5 -> 112.6).  That costs a barrier, which
// shorter passes do not earn back and groups of several passes would pay in each (8 heads of 2048, d = 2, fp32, half of the
// tokens in one group, forward and backward: 2000 us so, 2100 with every pass in halves).
template <int R, int PD, typename T>
struct ReadLayout {
  static constexpr int KT = 8;                              // tokens per pass over a state
  static constexpr int NJ4 = PD / 4, NG = 256 / NJ4;
  static constexpr int XM = R > PD ? R : PD;
  static constexpr int RED = KT * R > NG * KT * PD ? KT * R : NG * KT * PD;
  static constexpr int SMEM = R * PD * 4 + RED * 4 + 2 * KT * XM * (int)sizeof(T) + KT * XM * 4 + 64;
};

template <int R, int PD, typename T>
__global__ void __launch_bounds__(256, 2) state_read_stream_kernel(const __grid_constant__ ReadList list, int64_t Tlen,
                                                                   int* status) {
  using L = ReadLayout<R, PD, T>;
  constexpr int KT = L::KT, NJ4 = L::NJ4, NG = L::NG;
  constexpr int RPG = R / NG, RPH = RPG / 2;   // a thread's rows of a state, and of a half
  constexpr bool HALVES = RPH >= 4;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  float* Sb = reinterpret_cast<float*>(smem_raw);        // [R*PD]
  float* red = Sb + R * PD;                              // [RED]
  T* Xraw = reinterpret_cast<T*>(red + L::RED);          // [2][KT][XM] raw rows of the first KT tokens of an item
  float* Xs = reinterpret_cast<float*>(Xraw + 2 * KT * L::XM);  // [KT][XM]
  uint64_t* bar = reinterpret_cast<uint64_t*>(Xs + KT * L::XM);   // [2] a half of the state has landed
  volatile int* cta_abort = reinterpret_cast<volatile int*>(bar + 2);
  pdl_trigger();
  const tc::WaitCtx wc{cta_abort, status};
  const int tid = threadIdx.x;
  if ((int)blockIdx.x < list.scan_ctas) {
    pdl_wait();
    const int x = blockIdx.x % list.scan_x, yz = blockIdx.x / list.scan_x;
    smat_scan_entries(list.scan, R * PD, list.NC, x * 256 + tid, yz % list.scan_y, yz / list.scan_y);
    return;
  }
  const int j4 = tid % NJ4, ig = tid / NJ4;
  constexpr uint32_t LBYTES = HALVES ? R * PD * 2 : R * PD * 4;   // a load: half a state, or all of it
  const int64_t items = list.first[list.a.jobs], cta = blockIdx.x - list.scan_ctas, ctas = gridDim.x - list.scan_ctas;
  auto job_of = [&](int64_t item) {
    int j = 0;
    while (item >= list.first[j + 1]) ++j;
    return j;
  };
  auto tokens_of = [&](int64_t item, int j, int64_t* bh) {
    const int64_t at = item - list.first[j];
    *bh = smat_div(at, list.a.job[j].groups);
    return smat_group_tokens(list.a.job[j].grp, *bh, at - *bh * list.a.job[j].groups);
  };
  auto state_of = [&](int64_t item) {
    const int j = job_of(item);
    return list.a.job[j].state + (item - list.first[j]) * (int64_t)(R * PD);
  };
  auto prefetch_x = [&](int64_t item, int buf) {
    if (item < items) {
      const int j = job_of(item);
      int64_t bh;
      const SmatTokens tk = tokens_of(item, j, &bh);
      const int xd = list.a.job[j].trans ? PD : R, xc = xd * (int)sizeof(T) / 16;   // 16-byte chunks per x row
      const int kn = (int)(tk.cnt < KT ? tk.cnt : KT);
      const T* Xb = static_cast<const T*>(list.a.job[j].x) + bh * Tlen * xd;
      for (int idx = tid; idx < kn * xc; idx += 256) {
        const int k = idx / xc, c = idx - k * xc;
        cp_async16(reinterpret_cast<uint8_t*>(Xraw + (buf * KT + k) * L::XM) + c * 16,
                   reinterpret_cast<const uint8_t*>(Xb + tk.at(k) * xd) + c * 16);
      }
    }
    cp_async_commit();
  };

  if (tid == 0) {
    *cta_abort = 0;
    tc::mbar_init(bar, 1);
    tc::mbar_init(bar + 1, 1);
    tc::fence_barrier_init();
  }
  uint32_t loads[2] = {0, 0};   // started ones (thread 0)
  auto load_half = [&](int64_t item, int h) {
    tc::mbar_expect_tx(bar + h, LBYTES);
    bulk_load(Sb + h * (R * PD / 2), state_of(item) + h * (R * PD / 2), LBYTES, bar + h);
    ++loads[h];
  };
  auto load_state = [&](int64_t item) {
    load_half(item, 0);
    if (HALVES) load_half(item, 1);
  };
  pdl_wait();
  if (tid == 0 && cta < items) load_state(cta);
  prefetch_x(cta, 0);
  __syncthreads();
  int n = 0;
  for (int64_t item = cta; item < items; item += ctas, ++n) {
    const int buf = n & 1;
    const int j = job_of(item);
    int64_t bh;
    const SmatTokens tk = tokens_of(item, j, &bh);
    const int64_t cnt = tk.cnt, nxt = item + ctas;
    const int trans = list.a.job[j].trans, xd = trans ? PD : R, od = trans ? R : PD;
    const T* Xb = static_cast<const T*>(list.a.job[j].x) + bh * Tlen * xd;
    float* out = list.a.job[j].out + bh * Tlen * od;
    const float4* S4 = reinterpret_cast<const float4*>(Sb);
    const bool split = HALVES && !trans && cnt > 4 && cnt <= KT;
    prefetch_x(nxt, buf ^ 1);
    cp_async_wait<1>();
    __syncthreads();
    for (int64_t k0 = 0; k0 == 0 || k0 < cnt; k0 += KT) {   // (a state without tokens is waited for and passed over)
      const int kn = (int)((cnt - k0) < KT ? (cnt - k0) : KT);
      for (int idx = tid; idx < KT * xd; idx += 256) {
        const int k = idx / xd, i = idx - k * xd;
        float v = 0.f;
        if (k < kn) v = k0 == 0 ? to_float(Xraw[(buf * KT + k) * L::XM + i]) : to_float(Xb[tk.at(k0 + k) * xd + i]);
        Xs[k * L::XM + i] = v;
      }
      // (block-wide barriers follow: all go on, or none)
      const bool ok = __syncthreads_and(k0 > 0 || (tc::mbar_wait(bar, n & 1, wc) && (split || !HALVES || tc::mbar_wait(bar + 1, n & 1, wc)))) != 0;
      if (!ok || cnt == 0) break;
      if (!trans) {
        // KK: tokens of the pass, rounded up: nine tokens are a pass of eight and one of two (32 heads of 5056 tokens, d = 3,
        // normalised: the pass 651 us with eight to every one, 615 so)
        auto contract = [&](auto tokens) {
          constexpr int KK = decltype(tokens)::value;
          float4 acc[KK];
#pragma unroll
          for (int k = 0; k < KK; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          // four rows at a time, so that a token's factors are one load (32 heads, 307 states, bf16: 0.185 -> 0.177 ms)
          auto rows = [&](int first, int count) {
#pragma unroll 2
            for (int s = 0; s < count; s += 4) {
              const int i = first + s;
              const float4 u0 = S4[i * NJ4 + j4], u1 = S4[(i + 1) * NJ4 + j4], u2 = S4[(i + 2) * NJ4 + j4], u3 = S4[(i + 3) * NJ4 + j4];
#pragma unroll
              for (int k = 0; k < KK; ++k) {
                const float4 x = *reinterpret_cast<const float4*>(Xs + k * L::XM + i);
                acc[k] = fma4(x.x, u0, acc[k]); acc[k] = fma4(x.y, u1, acc[k]);
                acc[k] = fma4(x.z, u2, acc[k]); acc[k] = fma4(x.w, u3, acc[k]);
              }
            }
          };
          if (HALVES && KK == KT && split) {
            rows(ig * RPH, RPH);
            if (!__syncthreads_and(tc::mbar_wait(bar + 1, n & 1, wc))) return false;
            if (tid == 0 && nxt < items) load_half(nxt, 0);   // every thread is past its reads of the first half
            rows(R / 2 + ig * RPH, RPH);
          } else {
            rows(ig * RPG, RPG);
          }
#pragma unroll
          for (int k = 0; k < KK; ++k) *reinterpret_cast<float4*>(red + (ig * KT + k) * PD + j4 * 4) = acc[k];
          return true;
        };
        const bool done = kn > 4 ? contract(std::integral_constant<int, 8>{})
                                 : (kn > 2 ? contract(std::integral_constant<int, 4>{}) : contract(std::integral_constant<int, 2>{}));
        if (!done) break;
        __syncthreads();
        if (split && tid == 0 && nxt < items) load_half(nxt, 1);
        for (int idx = tid; idx < kn * NJ4; idx += 256) {   // the row groups' partial rows meet in shared memory
          const int k = idx / NJ4, c = idx - k * NJ4;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int w = 0; w < NG; ++w) {
            const float4 p = *reinterpret_cast<const float4*>(red + (w * KT + k) * PD + c * 4);
            v.x += p.x; v.y += p.y; v.z += p.z; v.w += p.w;
          }
          *reinterpret_cast<float4*>(out + tk.at(k0 + k) * PD + c * 4) = v;
        }
      } else {
#pragma unroll 2
        for (int s = 0; s < RPG; ++s) {
          const int i = ig * RPG + s;
          const float4 u = S4[i * NJ4 + j4];
          float part[KT];
#pragma unroll
          for (int k = 0; k < KT; ++k) {
            const float4 x4 = *reinterpret_cast<const float4*>(Xs + k * L::XM + j4 * 4);
            part[k] = u.x * x4.x + u.y * x4.y + u.z * x4.z + u.w * x4.w;
          }
#pragma unroll
          for (int off = NJ4 / 2; off > 0; off >>= 1)
#pragma unroll
            for (int k = 0; k < KT; ++k) part[k] += __shfl_xor_sync(0xffffffffu, part[k], off);
          if (j4 == 0)
#pragma unroll
            for (int k = 0; k < KT; ++k) red[k * R + i] = part[k];
        }
        __syncthreads();
        for (int idx = tid; idx < kn * R; idx += 256) {
          const int k = idx / R, i = idx % R;
          out[tk.at(k0 + k) * R + i] = red[k * R + i];
        }
      }
      __syncthreads();
    }
    // every thread is past its reads of the state buffer: fetch the next item's state
    if (!split && tid == 0 && nxt < items && !*cta_abort) load_state(nxt);
  }
  if (tid == 0) {   // (a barrier that never saw a load lets parity 1 pass)
    tc::landed(bar, (loads[0] + 1) & 1, wc);
    tc::landed(bar + 1, (loads[1] + 1) & 1, wc);
  }
  cp_async_wait<0>();
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

int smat_sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

namespace {

template <int R, int PD, typename T, int TK>
cudaError_t launch_pool_tk(const PoolList& list, int64_t Tlen, int* clear, cudaStream_t st) {
  const int64_t items = list.first[list.a.jobs];
  const size_t smem = smat_smem_alone(items, R * PD * 4 + 2 * TK * (R + PD) * (int)sizeof(T));
  cudaError_t err = set_smem(pool_stream_kernel<R, PD, T, TK>, smem);
  if (err != cudaSuccess) return err;
  const int per_sm = smem <= 110 * 1024 ? 2 : 1;
  const int64_t grid = items < (int64_t)smat_sm_count() * per_sm ? items : (int64_t)smat_sm_count() * per_sm;
  return smat_launch_pdl(pool_stream_kernel<R, PD, T, TK>, dim3((unsigned)grid), 256, smem, st, list, Tlen, clear);
}

// As long as every item has an SM of its own the time is one item's way through the passes: 64 tokens to a pass there (a
// chunk of 64 is one round of loads instead of four: forward and backward of one 512-token head, d = 2, fp32, 45.9 -> 37.2 us
// together with the 16-row tiles); else few, so that two CTAs share an SM.
template <int R, int PD, typename T>
cudaError_t launch_pool(const PoolList& list, int64_t Tlen, int* clear, cudaStream_t st) {
  if (list.first[list.a.jobs] <= smat_sm_count()) return launch_pool_tk<R, PD, T, 64>(list, Tlen, clear, st);
  return launch_pool_tk<R, PD, T, sizeof(T) == 2 ? 32 : 16>(list, Tlen, clear, st);
}

template <int R, int PD, typename T>
cudaError_t launch_read(const ReadList& list, int64_t Tlen, int* status, cudaStream_t st) {
  const size_t smem = ReadLayout<R, PD, T>::SMEM;
  cudaError_t err = set_smem(state_read_stream_kernel<R, PD, T>, smem);
  if (err != cudaSuccess) return err;
  const int64_t items = list.first[list.a.jobs];
  const int per_sm = smem <= 112 * 1024 ? 2 : 1;
  const int64_t grid = items < (int64_t)smat_sm_count() * per_sm ? items : (int64_t)smat_sm_count() * per_sm;
  return smat_launch_pdl(state_read_stream_kernel<R, PD, T>, dim3((unsigned)(grid + list.scan_ctas)), 256, smem, st, list, Tlen, status);
}

}  // namespace

cudaError_t smat_launch_pool(const SmatPoolArgs& a, int bf16, int64_t Tlen, int bh, int r, int p, int* clear, cudaStream_t st) {
  PoolList list;
  list.a = a;
  list.first[0] = 0;
  for (int j = 0; j < a.jobs; ++j) list.first[j + 1] = list.first[j] + a.job[j].groups * bh;
#define SMAT_POOL(RV, PV)                                                                                          \
  if (r == RV && p == PV)                                                                                          \
    return bf16 ? launch_pool<RV, PV, __nv_bfloat16>(list, Tlen, clear, st) : launch_pool<RV, PV, float>(list, Tlen, clear, st);
  SMAT_POOL(128, 128) SMAT_POOL(64, 64) SMAT_POOL(64, 128) SMAT_POOL(128, 64)
#undef SMAT_POOL
  return cudaErrorInvalidValue;
}

cudaError_t smat_launch_state_read(const SmatReadArgs& a, int bf16, int64_t Tlen, int bh, int r, int p, int* status,
                                   cudaStream_t st, const SmatScanArgs* scan, int64_t NC) {
  ReadList list{};
  list.a = a;
  if (scan) {
    list.scan = *scan; list.NC = NC;
    list.scan_x = (r * p / 4 + 255) / 256; list.scan_y = bh;
    list.scan_ctas = list.scan_x * bh * 2 * scan->jobs;
  }
  list.first[0] = 0;
  for (int j = 0; j < a.jobs; ++j) list.first[j + 1] = list.first[j] + a.job[j].groups * bh;
#define SMAT_READ(RV, PV)                                                                        \
  if (r == RV && p == PV)                                                                        \
    return bf16 ? launch_read<RV, PV, __nv_bfloat16>(list, Tlen, status, st)                     \
                : launch_read<RV, PV, float>(list, Tlen, status, st);
  SMAT_READ(128, 128) SMAT_READ(64, 64) SMAT_READ(64, 128) SMAT_READ(128, 64)
#undef SMAT_READ
  return cudaErrorInvalidValue;
}
