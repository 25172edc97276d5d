// Kernels of the options beyond the default pipeline: the value norms of the v-norm variant
// (App. A.1.3) and the position order of the kept tokens.
#include "kvc_internal.cuh"
#include "value_norm.cuh"

namespace kvc {
namespace {

// (a stream: past L1, L2 fetches 256 bytes at a time)
__device__ __forceinline__ uint4 ld_once(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// ||v|| of every value row, where the scoring kernel does not take it along (fp32, explicit maps, strides it cannot take).  Bound
// by HBM: V is read once.  A warp per row with half of its lanes idle and one load in flight took 807 us for
// 1.07 GB (1.3 TB/s); this form takes 182 us (5.9 TB/s; 191 with plain loads, 4 rows per lane 192).
template <typename T, int kLpr>
__global__ void __launch_bounds__(256)
value_norm_kernel(LayerPtrs vp, float* __restrict__ vnorm, int Bt, int Hkv, long long segs, long long N, long long vs0,
                  long long vs1, long long vs2) {
  grid_dependency_wait();
  constexpr int kGroups = 32 / kLpr;                         // rows a warp loads at once
  const int lane = threadIdx.x & 31, sub = lane & (kLpr - 1), grp = lane / kLpr;
  const long long first = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * kNormBlock<kLpr>;
  for (long long seg = blockIdx.y; seg < segs; seg += gridDim.y) {      // (l * Bt + b) * Hkv + h
    const int h = (int)(seg % Hkv);
    const int b = (int)(seg / Hkv % Bt);
    const int l = (int)(seg / Hkv / Bt);
    const T* base = reinterpret_cast<const T*>(vp.p[l]) + b * vs0 + h * vs1;
    uint4 w[kNormRows];
#pragma unroll
    for (int u = 0; u < kNormRows; ++u) {
      const long long c = min(first + grp + u * kGroups, N - 1);
      w[u] = ld_once(reinterpret_cast<const uint4*>(base + c * vs2) + sub);
    }
    norm_store<T, kLpr>(w, vnorm + seg * N, first, N);
  }
}

template <typename T, int kLpr>
kvc_status launch_norm_t(const Problem& P, const LayerPtrs& v, float* vnorm, cudaStream_t st) {
  const long long per_cta = 8LL * kNormBlock<kLpr>;
  const long long segs = (long long)P.L * P.Bt * P.Hkv;
  const dim3 grid((unsigned)((P.N + per_cta - 1) / per_cta), (unsigned)(segs < 65535 ? segs : 65535));
  KVC_CUDA(launch_dependent(value_norm_kernel<T, kLpr>, grid, dim3(256), 0, st, v, vnorm, P.Bt, P.Hkv, segs, P.N,
                            P.kvs[0], P.kvs[1], P.kvs[2]));
  KVC_LAUNCH_CHECK("value_norm_kernel");
  return KVC_OK;
}

// One CTA per (layer, sequence, head): marks the kept positions in a bitmap (one bit per token; in shared memory up to
// kOrderSharedN tokens, else in global scratch), then writes the marked positions back in ascending order.  Bound by latency:
// marks in shared memory do not travel to L2 (256 heads of 16384, a quarter kept: 13.7 -> 8.6 us).
constexpr int kOrderThreads = 512;
// 32 KB of marks: four CTAs of 512 threads per SM fill it and fit, without a launch attribute.  (64 heads, a quarter kept, at the
// line: 66 us in shared memory for 262144 tokens, 97 us in the workspace for 262148.)
constexpr long long kOrderSharedN = 262144;

template <bool kShared>
__global__ void __launch_bounds__(kOrderThreads)
order_kept_kernel(int32_t* __restrict__ idx, const int32_t* __restrict__ n_keep, uint32_t* __restrict__ bitmap,
                  int L, int Bt, int Hkv, long long N, int per_head) {
  __shared__ uint32_t warp_tot[kOrderThreads / 32];
  __shared__ uint32_t carry;
  extern __shared__ uint32_t order_bits[];
  grid_dependency_wait();
  const long long seg = blockIdx.x;                   // (l * Bt + b) * Hkv + h
  const int h = (int)(seg % Hkv);
  const int b = (int)((seg / Hkv) % Bt);
  const int l = (int)(seg / ((long long)Hkv * Bt));
  const long long n = per_head ? n_keep[((long long)b * L + l) * Hkv + h] : n_keep[(long long)b * L + l];
  int32_t* row = idx + seg * N;
  const long long words = (N + 31) / 32;
  uint32_t* bits = kShared ? order_bits : bitmap + seg * words;
  for (long long i = threadIdx.x; i < words; i += kOrderThreads) bits[i] = 0u;
  __syncthreads();
  for (long long k0 = threadIdx.x; k0 < n; k0 += 4 * kOrderThreads) {
    int32_t c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i] = k0 + i * kOrderThreads < n ? row[k0 + i * kOrderThreads] : -1;
#pragma unroll
    for (int i = 0; i < 4; ++i) if (c[i] >= 0) atomicOr(&bits[c[i] >> 5], 1u << (c[i] & 31));
  }
  if (threadIdx.x == 0) carry = 0u;
  __syncthreads();
  // every thread takes one bitmap word per round; exclusive prefix of the popcounts over the CTA
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (long long w0 = 0; w0 < words; w0 += kOrderThreads) {
    const long long wi = w0 + threadIdx.x;
    uint32_t word = wi < words ? bits[wi] : 0u;
    const uint32_t cnt = __popc(word);
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    uint32_t before = carry;
    for (int wv = 0; wv < warp; ++wv) before += warp_tot[wv];
    uint32_t pos = before + incl - cnt;
    while (word) {
      const int bit = __ffs(word) - 1;
      word &= word - 1;
      row[pos++] = (int32_t)(wi * 32 + bit);
    }
    __syncthreads();
    if (threadIdx.x == kOrderThreads - 1) carry = before + incl;
    __syncthreads();
  }
}

// Head-sharded scoring: the local part of Eq. 16's sum over the KV heads, and the mean added back.  Streams: a thread takes
// four neighbouring tokens with 16-byte accesses where the rows allow it (kVec: N a multiple of 4), one otherwise;
// blockIdx.y = (layer, sequence), so that no index has to be divided.  (32 layers, 2 heads, N = 32768, one token per thread and
// a 64-bit division: 8.0 and 6.3 us, the scaling 3.9; so: 3.7, 3.8 and 2.2.)
template <bool kVec>
__global__ void __launch_bounds__(256)
head_sum_kernel(const float* __restrict__ s, float* __restrict__ head_sum, int Hkv, long long N) {
  grid_dependency_wait();
  const long long c = ((long long)blockIdx.x * 256 + threadIdx.x) * (kVec ? 4 : 1);
  if (c >= N) return;
  const float* base = s + (long long)blockIdx.y * Hkv * N + c;
  if constexpr (kVec) {
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int h = 0; h < Hkv; ++h) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(base + (long long)h * N));
      sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
    }
    *reinterpret_cast<float4*>(head_sum + (long long)blockIdx.y * N + c) = sum;
  } else {
    float sum = 0.f;
#pragma unroll 4
    for (int h = 0; h < Hkv; ++h) sum += __ldg(base + (long long)h * N);
    head_sum[(long long)blockIdx.y * N + c] = sum;
  }
}

// (blockIdx.z: the head)
template <bool kVec>
__global__ void __launch_bounds__(256)
add_head_mean_kernel(float* __restrict__ s, const float* __restrict__ head_sum, int Hkv, float inv_total, long long N) {
  grid_dependency_wait();
  const long long c = ((long long)blockIdx.x * 256 + threadIdx.x) * (kVec ? 4 : 1);
  if (c >= N) return;
  float* at = s + ((long long)blockIdx.y * Hkv + blockIdx.z) * N + c;
  const float* sum = head_sum + (long long)blockIdx.y * N + c;
  if constexpr (kVec) {
    const float4 m = __ldg(reinterpret_cast<const float4*>(sum));
    float4 v = *reinterpret_cast<const float4*>(at);
    v.x += m.x * inv_total; v.y += m.y * inv_total; v.z += m.z * inv_total; v.w += m.w * inv_total;
    *reinterpret_cast<float4*>(at) = v;
  } else {
    *at += __ldg(sum) * inv_total;
  }
}

template <bool kVec>
__global__ void __launch_bounds__(256)
scale_kernel(float* __restrict__ x, long long n, float f) {
  grid_dependency_wait();
  const long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * (kVec ? 4 : 1);
  if (i >= n) return;
  if constexpr (kVec) {
    float4 v = *reinterpret_cast<const float4*>(x + i);
    v.x *= f; v.y *= f; v.z *= f; v.w *= f;
    *reinterpret_cast<float4*>(x + i) = v;
  } else {
    x[i] *= f;
  }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

kvc_status launch_head_sum(const Problem& P, const float* scores, float* head_sum, cudaStream_t st) {
  const bool vec = P.N % 4 == 0 && aligned16(scores) && aligned16(head_sum);
  const long long per = vec ? 1024 : 256;
  KVC_CUDA(launch_dependent(vec ? head_sum_kernel<true> : head_sum_kernel<false>,
                            dim3((unsigned)((P.N + per - 1) / per), (unsigned)(P.L * P.Bt)), dim3(256), 0, st, scores, head_sum,
                            P.Hkv, P.N));
  KVC_LAUNCH_CHECK("head_sum_kernel");
  return KVC_OK;
}

kvc_status launch_add_head_mean(const Problem& P, float* scores, const float* head_sum, int heads_total,
                                cudaStream_t st) {
  const bool vec = P.N % 4 == 0 && aligned16(scores) && aligned16(head_sum);
  const long long per = vec ? 1024 : 256;
  KVC_CUDA(launch_dependent(vec ? add_head_mean_kernel<true> : add_head_mean_kernel<false>,
                            dim3((unsigned)((P.N + per - 1) / per), (unsigned)(P.L * P.Bt), (unsigned)P.Hkv), dim3(256), 0, st,
                            scores, head_sum, P.Hkv, 1.0f / (float)heads_total, P.N));
  KVC_LAUNCH_CHECK("add_head_mean_kernel");
  return KVC_OK;
}

kvc_status launch_scale(float* x, long long n, float f, cudaStream_t st) {
  if (n <= 0) return KVC_OK;
  const bool vec = n % 4 == 0 && aligned16(x);
  const long long per = vec ? 1024 : 256;
  KVC_CUDA(launch_dependent(vec ? scale_kernel<true> : scale_kernel<false>, dim3((unsigned)((n + per - 1) / per)), dim3(256), 0, st,
                            x, n, f));
  KVC_LAUNCH_CHECK("scale_kernel");
  return KVC_OK;
}

kvc_status launch_value_norm(const Problem& P, const LayerPtrs& v, float* vnorm, cudaStream_t st) {
  if (P.dtype == KVC_BF16)
    return P.d == 128 ? launch_norm_t<__nv_bfloat16, 16>(P, v, vnorm, st) : launch_norm_t<__nv_bfloat16, 8>(P, v, vnorm, st);
  return P.d == 128 ? launch_norm_t<float, 32>(P, v, vnorm, st) : launch_norm_t<float, 16>(P, v, vnorm, st);
}

size_t order_kept_workspace_bytes(const Problem& P) {
  return align_up((size_t)P.L * P.Bt * P.Hkv * (size_t)((P.N + 31) / 32) * sizeof(uint32_t));
}

kvc_status launch_order_kept(const Problem& P, int32_t* idx, const int32_t* n_keep, bool per_head,
                             void* ws, size_t ws_bytes, cudaStream_t st) {
  if (ws_bytes < order_kept_workspace_bytes(P)) {
    set_error("order_kept: workspace too small");
    return KVC_ERR_WORKSPACE;
  }
  const long long segs = (long long)P.L * P.Bt * P.Hkv;
  const bool shared = P.N <= kOrderSharedN;
  const size_t smem = shared ? (size_t)((P.N + 31) / 32) * sizeof(uint32_t) : 0;
  KVC_CUDA(launch_dependent(shared ? order_kept_kernel<true> : order_kept_kernel<false>, dim3((unsigned)segs), dim3(kOrderThreads),
                            smem, st, idx, n_keep,
                            reinterpret_cast<uint32_t*>(ws), P.L, P.Bt, P.Hkv, P.N, per_head ? 1 : 0));
  KVC_LAUNCH_CHECK("order_kept_kernel");
  return KVC_OK;
}

}  // namespace kvc
