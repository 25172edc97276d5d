// Token-importance scoring on the CUDA cores (Eqs. 3, 14-16).
//
// This is the shape-agnostic path: fp32 or bf16 inputs, head_dim 64 or 128, any window length,
// any GQA map.  Where the logits of a (layer, sequence, KV head) fit a bounded buffer they are computed once and kept
// (second part of this file); otherwise, and for few rows over many tokens, it makes two sweeps over K.  Sweep 1 produces, for every query row, the
// log-sum-exp of its logits over the visible keys (per-chunk partials, then a combine kernel).
// Sweep 2 recomputes the logits and emits exp(s - lse) -- the softmax weight of Eq. 3 -- reduced
// over the window rows (Eq. 14) and over the query heads of the KV head (Eq. 15).  A last kernel
// adds the mean over KV heads (Eq. 16).  Logits are kept in the log2 domain so that every
// exponential is a single ex2.
#include <math.h>

#include "kvc_internal.cuh"

namespace kvc {
namespace {

constexpr int kThreads = 128;     // one token per thread
constexpr int kRowTile = 32;      // query rows staged in shared memory at a time
constexpr int kChunkIters = 8;    // sweep-1 chunk = kChunkIters * kThreads tokens
constexpr float kLog2e = 1.4426950408889634f;

struct ScoreParams {
  int L, Bt, Hq, Hkv, w;
  long long N, q_pos0;
  long long qs0, qs1, qs2, kvs0, kvs1, kvs2;
  float scale_log2e;
  int agg_task, agg_group;
  int nchunks;
};

struct KvOfQ {
  int16_t kv[kMaxQHeads];
};

template <typename T>
__device__ inline void load_row(const T* __restrict__ src, float* dst, int D);

template <>
__device__ inline void load_row<float>(const float* __restrict__ src, float* dst, int D) {
  const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
  for (int i = 0; i < 64; ++i) {
    if (i * 4 < D) {
      float4 v = __ldg(s4 + i);
      dst[i * 4 + 0] = v.x; dst[i * 4 + 1] = v.y; dst[i * 4 + 2] = v.z; dst[i * 4 + 3] = v.w;
    }
  }
}

template <>
__device__ inline void load_row<__nv_bfloat16>(const __nv_bfloat16* __restrict__ src, float* dst, int D) {
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    if (i * 8 < D) {
      uint4 v = __ldg(s4 + i);
      uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        dst[i * 8 + 2 * e + 0] = __uint_as_float(u[e] << 16);          // bf16 -> fp32 is exact
        dst[i * 8 + 2 * e + 1] = __uint_as_float(u[e] & 0xffff0000u);
      }
    }
  }
}

__device__ inline float to_float(float x) { return x; }
__device__ inline float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

// Stage rows [r0, r0 + rt) of one query head into shared memory as fp32.
template <typename T, int D>
__device__ inline void stage_q(const T* __restrict__ qhead, long long row_stride, int r0, int rt,
                               float* Qs) {
  for (int i = threadIdx.x; i < rt * D; i += kThreads) {
    int r = i / D, t = i - r * D;
    Qs[i] = to_float(qhead[(long long)(r0 + r) * row_stride + t]);
  }
}

template <int D>
__device__ inline float dot_row(const float* __restrict__ Qrow, const float* kr) {
  const float4* q4 = reinterpret_cast<const float4*>(Qrow);
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
  for (int i = 0; i < D / 4; ++i) {
    float4 qv = q4[i];  // same address for the whole warp: a broadcast
    a0 = fmaf(qv.x, kr[4 * i + 0], a0);
    a1 = fmaf(qv.y, kr[4 * i + 1], a1);
    a2 = fmaf(qv.z, kr[4 * i + 2], a2);
    a3 = fmaf(qv.w, kr[4 * i + 3], a3);
  }
  return (a0 + a1) + (a2 + a3);
}

__device__ inline float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ inline float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sweep 1: per (layer, sequence, query head, token chunk) the running (max, sum-exp) of every
// window row over the chunk's visible keys, in the log2 domain.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
score_stats_kernel(ScoreParams P, KvOfQ map, LayerPtrs qp, LayerPtrs kp, float2* __restrict__ partial) {
  __shared__ __align__(16) float Qs[kRowTile * D];
  __shared__ float sm_m[kRowTile][kThreads / 32];
  __shared__ float sm_l[kRowTile][kThreads / 32];

  const int chunk = blockIdx.x, j = blockIdx.y, lb = blockIdx.z;
  const int l = lb / P.Bt, b = lb - l * P.Bt;
  const int h = map.kv[j];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T* kbase = reinterpret_cast<const T*>(kp.p[l]) + b * P.kvs0 + h * P.kvs1;
  const T* qbase = reinterpret_cast<const T*>(qp.p[l]) + b * P.qs0 + j * P.qs1;
  const long long c_begin = (long long)chunk * (kChunkIters * kThreads);

  for (int r0 = 0; r0 < P.w; r0 += kRowTile) {
    const int rt = min(kRowTile, P.w - r0);
    __syncthreads();
    stage_q<T, D>(qbase, P.qs2, r0, rt, Qs);
    for (int i = threadIdx.x; i < kRowTile * (kThreads / 32); i += kThreads) {
      (&sm_m[0][0])[i] = -INFINITY;
      (&sm_l[0][0])[i] = 0.f;
    }
    __syncthreads();
    for (int it = 0; it < kChunkIters; ++it) {
      const long long c = c_begin + (long long)it * kThreads + threadIdx.x;
      if (c_begin + (long long)it * kThreads >= P.N) break;  // uniform for the block
      const bool valid = c < P.N;
      float kr[D];
      if (valid) {
        load_row<T>(kbase + c * P.kvs2, kr, D);
      } else {
#pragma unroll
        for (int i = 0; i < D; ++i) kr[i] = 0.f;
      }
      for (int r = 0; r < rt; ++r) {
        float s = dot_row<D>(Qs + r * D, kr) * P.scale_log2e;
        const bool vis = valid && (c <= P.q_pos0 + r0 + r);
        s = vis ? s : -INFINITY;
        const float m_w = warp_max(s);
        const float m_old = sm_m[r][warp];
        const float m_new = fmaxf(m_old, m_w);
        const float e = (m_new == -INFINITY) ? 0.f : exp2f(s - m_new);
        const float l_w = warp_sum(e);
        __syncwarp();
        if (lane == 0 && m_new > -INFINITY) {
          sm_l[r][warp] = sm_l[r][warp] * exp2f(m_old - m_new) + l_w;
          sm_m[r][warp] = m_new;
        }
        __syncwarp();
      }
    }
    __syncthreads();
    if (threadIdx.x < rt) {
      const int r = threadIdx.x;
      float M = -INFINITY;
#pragma unroll
      for (int wv = 0; wv < kThreads / 32; ++wv) M = fmaxf(M, sm_m[r][wv]);
      float Lsum = 0.f;
      if (M > -INFINITY) {
#pragma unroll
        for (int wv = 0; wv < kThreads / 32; ++wv) Lsum += sm_l[r][wv] * exp2f(sm_m[r][wv] - M);
      }
      const long long row = ((long long)lb * P.Hq + j) * P.w + r0 + r;
      partial[row * P.nchunks + chunk] = make_float2(M, Lsum);
    }
  }
}

// Combine the chunk partials of one query row into lse2 = log2(sum_c 2^{s2_c}).
__global__ void score_lse_kernel(const float2* __restrict__ partial, float* __restrict__ lse2,
                                 long long rows, int nchunks) {
  const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows) return;
  const float2* p = partial + row * nchunks;
  float M = -INFINITY;
  for (int i = 0; i < nchunks; ++i) M = fmaxf(M, p[i].x);
  float Lsum = 0.f;
  for (int i = 0; i < nchunks; ++i)
    if (p[i].x > -INFINITY) Lsum += p[i].y * exp2f(p[i].x - M);
  lse2[row] = M + log2f(Lsum);
}

// Sweep 2: S_group[l, b, h, c] (Eqs. 14-15) from the logits and the rows' log-sum-exp.
template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
score_emit_kernel(ScoreParams P, GroupMap gm, LayerPtrs qp, LayerPtrs kp,
                  const float* __restrict__ lse2, float* __restrict__ s_group) {
  __shared__ __align__(16) float Qs[kRowTile * D];
  __shared__ float Ls[kRowTile];

  const int h = blockIdx.y, lb = blockIdx.z;
  const int l = lb / P.Bt, b = lb - l * P.Bt;
  const long long c = (long long)blockIdx.x * kThreads + threadIdx.x;
  const bool valid = c < P.N;
  const T* kbase = reinterpret_cast<const T*>(kp.p[l]) + b * P.kvs0 + h * P.kvs1;

  float kr[D];
  if (valid) {
    load_row<T>(kbase + c * P.kvs2, kr, D);
  } else {
#pragma unroll
    for (int i = 0; i < D; ++i) kr[i] = 0.f;
  }

  const int members = gm.begin[h + 1] - gm.begin[h];
  float gacc = (P.agg_group == KVC_AGG_MAX) ? -INFINITY : 0.f;
  for (int mi = 0; mi < members; ++mi) {
    const int j = gm.qh[gm.begin[h] + mi];
    const T* qbase = reinterpret_cast<const T*>(qp.p[l]) + b * P.qs0 + j * P.qs1;
    const float* lrow = lse2 + ((long long)lb * P.Hq + j) * P.w;
    float tacc = (P.agg_task == KVC_AGG_MAX) ? -INFINITY : 0.f;
    for (int r0 = 0; r0 < P.w; r0 += kRowTile) {
      const int rt = min(kRowTile, P.w - r0);
      __syncthreads();
      stage_q<T, D>(qbase, P.qs2, r0, rt, Qs);
      if (threadIdx.x < rt) Ls[threadIdx.x] = lrow[r0 + threadIdx.x];
      __syncthreads();
      for (int r = 0; r < rt; ++r) {
        const float s = dot_row<D>(Qs + r * D, kr) * P.scale_log2e;
        const bool vis = valid && (c <= P.q_pos0 + r0 + r);
        const float t = vis ? s - Ls[r] : -INFINITY;     // log2 of the attention weight
        if (P.agg_task == KVC_AGG_MAX) tacc = fmaxf(tacc, t);
        else tacc += exp2f(t);
      }
    }
    const float s_task = (P.agg_task == KVC_AGG_MAX) ? exp2f(tacc) : tacc / (float)P.w;
    if (P.agg_group == KVC_AGG_MAX) gacc = fmaxf(gacc, s_task);
    else gacc += s_task;
  }
  if (P.agg_group == KVC_AGG_MEAN) gacc /= (float)members;
  if (valid) s_group[((long long)lb * P.Hkv + h) * P.N + c] = gacc;
}

// ---- one product, its logits kept -----------------------------------------------------------------
// The sweeps above compute every logit twice, and one token per thread makes them wait for the broadcast reads of
// Q (a 16-byte read per four multiplications and thread).  Where the logits of a (layer, sequence, KV head) fit the
// workspace, they are computed once, by a register-tiled product, and kept in a buffer of at most kLogitsCap bytes;
// the statistics and the emission then read them.  Units are taken in groups that fill the buffer.  Every sum is
// taken in the order of the sweeps (four partial products per logit, the butterfly over 32 tokens, 8 such steps per
// warp and chunk), so the scores are the same bit for bit.  fp32, 16 layers, N = 3001, 32 / 8 heads of 128, w = 32:
// 1342 us for the two sweeps, 406 us so (the product 314; it cannot take less than 175: 128 multiply-adds a clock and
// SM).  A larger buffer (96 MB) gains 1 %, smaller ones mean more and shorter launches.
constexpr int kTileTok = 128, kHalfTok = kTileTok / 2, kLogitThreads = 256;
template <int kTT> constexpr int kLogitTileRows = kTT == 8 ? 128 : 32;
constexpr size_t kLogitsCap = (size_t)64 << 20;

struct LogitParams {
  int Bt, Hkv, w, max_rows;                     // max_rows: of a unit (the largest group's)
  long long N, np, q_pos0;                      // np: row stride of the buffer
  long long qs0, qs1, qs2, kvs0, kvs1, kvs2;
  float scale_log2e;
  int agg_task, agg_group, nchunks, unit0;      // unit0: first unit of the group
};

// Two fp32 lanes in one 64-bit register: d = a * b + c in both.
__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float2 unpack_f2(unsigned long long p) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
  return r;
}
// Four elements of a row to four floats in shared memory: asynchronously, or through registers where they are converted.
__device__ __forceinline__ void stage4(float* dst, const float* row, int v) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(row + 4 * v) : "memory");
}
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* row, int v) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(row) + v);
  *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                                                __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}

// dots[unit - unit0][row][token] = <q row, k token>.  Work items are (unit, 128 rows, 128 tokens), tokens fastest, dealt
// to the CTAs in even stretches, so that a CTA keeps its Q rows and streams K tiles through two buffers.  The tokens of an
// item are two halves of four warps, one on each scheduler, that wait for each other only where the Q rows change, and there
// the second half starts one sweep later: one half multiplies while the other stores and waits for its tile (325 -> 314 us
// in the case above; 320 without the delayed start).  8 x 8 logits per thread; the four partial products of a logit are taken two at a time (a packed pair), in two sweeps over the
// tile.  Bound by the multiply-adds (128 clocks of a scheduler per warp and step of two elements); the operand reads
// are what a smaller register tile would wait for: an 8-byte read costs the SM 2 clocks where neighbouring lanes read
// different addresses (the 8 tokens) and 1 where they share one (the 8 rows), 96 for four warps' steps.  (4 x 4 logits
// with all four products at once: 423 us in the case above.)  Rows are padded by 16 bytes to spread a read over the banks.
// kTT = 2: two tokens per thread, items of 32 rows, for units of few rows and for problems that would leave SMs idle (the tiny
// fp32 configuration: 8.2 -> 5.7 us).
template <typename T, int D, int kTT>
__global__ void __launch_bounds__(kLogitThreads, 1)
score_logits_kernel(LogitParams P, GroupMap gm, LayerPtrs qp, LayerPtrs kp, float* __restrict__ dots, int row_tiles,
                    int tok_tiles, int items, int* __restrict__ status) {
  constexpr int kPitch = D + 4, kVec = D / 4, kTileRow = kLogitTileRows<kTT>;
  constexpr int kTokGroups = kHalfTok / (8 * kTT);             // a half's warps side by side over its tokens
  extern __shared__ __align__(16) float gsm[];
  float* const Qs = gsm;
  float* const Ks = gsm + kTileRow * kPitch;                   // two buffers
  grid_dependency_wait();
  if (status != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *status = 0;      // (nothing here can fail on the device)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int half_id = warp >> 2, ht = threadIdx.x & 127;      // four warps, one on each scheduler
  const int tok = half_id * kHalfTok + (warp & 3) % kTokGroups * (8 * kTT) + (lane & 7);   // tokens tok + 8 i
  const int row0 = (warp & 3) / kTokGroups * 32, row = row0 + (lane >> 3);   // rows row + 4 j
  const int i0 = (int)((long long)items * blockIdx.x / gridDim.x), i1 = (int)((long long)items * (blockIdx.x + 1) / gridDim.x);
  auto load_k = [&](int item, float* dst) {
    const int ur = item / tok_tiles, tt = item - ur * tok_tiles;
    const int unit = P.unit0 + ur / row_tiles;
    const int h = unit % P.Hkv, lb = unit / P.Hkv;
    const T* base = reinterpret_cast<const T*>(kp.p[lb / P.Bt]) + (lb % P.Bt) * P.kvs0 + h * P.kvs1;
#pragma unroll 4
    for (int i = ht; i < kHalfTok * kVec; i += kLogitThreads / 2) {
      const int t = half_id * kHalfTok + i / kVec, v = i % kVec;
      stage4(dst + t * kPitch + 4 * v, base + min((long long)tt * kTileTok + t, P.N - 1) * P.kvs2, v);
    }
  };
  if (i0 < i1) load_k(i0, Ks);
  int cur = -1, rows = 0, r0 = 0;                              // the (unit, rows) whose Q is here
  for (int item = i0; item < i1; ++item) {
    float* const buf = Ks + ((item - i0) & 1) * (kTileTok * kPitch);
    const int ur = item / tok_tiles, tt = item - ur * tok_tiles;
    const bool fresh = ur != cur;
    if (fresh) {
      if (cur >= 0) __syncthreads();                           // the Q rows here have been read
      cur = ur;
      const int unit = P.unit0 + ur / row_tiles;
      const int h = unit % P.Hkv, lb = unit / P.Hkv;
      rows = (gm.begin[h + 1] - gm.begin[h]) * P.w;
      r0 = (ur % row_tiles) * kTileRow;
      const T* base = reinterpret_cast<const T*>(qp.p[lb / P.Bt]) + (lb % P.Bt) * P.qs0;
#pragma unroll 4
      for (int i = threadIdx.x; i < kTileRow * kVec; i += kLogitThreads) {
        const int rr = min(r0 + i / kVec, rows - 1), v = i % kVec;
        const int j = gm.qh[gm.begin[h] + rr / P.w];
        stage4(Qs + (i / kVec) * kPitch + 4 * v, base + j * P.qs1 + (long long)(rr % P.w) * P.qs2, v);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
    } else {
      asm volatile("cp.async.wait_all;" ::: "memory");
      asm volatile("bar.sync %0, 128;" ::"r"(1 + half_id) : "memory");
    }
    // this half's tile is here, and the one before has been read
    if (item + 1 < i1) load_k(item + 1, Ks + ((item + 1 - i0) & 1) * (kTileTok * kPitch));
    const bool delay = kTT == 8 && fresh && item + 1 < i1;     // (the same in all threads; with a single item it only costs)
    if (delay && half_id == 1) asm volatile("bar.sync 3, 256;" ::: "memory");
    if (r0 + row0 >= rows) {
      if (delay && half_id == 0) asm volatile("bar.arrive 3, 256;" ::: "memory");
    } else {
      const float* kq = buf + tok * kPitch;
      const float* qq = Qs + row * kPitch;
      unsigned long long acc[kTT][8];                            // [token][row]: two partial products
      float first[kTT][8];                                       // the sum of the first two
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (half == 1 && delay && half_id == 0) asm volatile("bar.arrive 3, 256;" ::: "memory");
#pragma unroll
        for (int i = 0; i < kTT; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
#pragma unroll 4
        for (int v = 0; v < kVec; ++v) {
          unsigned long long kv[kTT];
#pragma unroll
          for (int i = 0; i < kTT; ++i) kv[i] = *reinterpret_cast<const unsigned long long*>(kq + i * 8 * kPitch + 4 * v + 2 * half);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const unsigned long long qv = *reinterpret_cast<const unsigned long long*>(qq + j * 4 * kPitch + 4 * v + 2 * half);
#pragma unroll
            for (int i = 0; i < kTT; ++i) acc[i][j] = ffma2(qv, kv[i], acc[i][j]);
          }
        }
        if (half == 0) {
#pragma unroll
          for (int i = 0; i < kTT; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) { const float2 x = unpack_f2(acc[i][j]); first[i][j] = x.x + x.y; }
        }
      }
      const long long t0 = (long long)tt * kTileTok + tok;
      float* out = dots + ((long long)(ur / row_tiles) * P.max_rows + r0 + row) * P.np + t0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (r0 + row + 4 * j < rows) {
#pragma unroll
          for (int i = 0; i < kTT; ++i) {
            const float2 y = unpack_f2(acc[i][j]);
            if (t0 + 8 * i < P.N) out[(long long)(4 * j) * P.np + 8 * i] = first[i][j] + (y.x + y.y);
          }
        }
      }
    }
  }
}

// The log-sum-exp (base 2) of four rows of a unit.  Eight lanes per row, four neighbouring tokens each; a warp takes 8 steps
// of 32 tokens, 128 apart, as a warp of score_stats_kernel does; the four "warps" of a chunk and then the chunks are folded
// as there.  Bound by the load / shuffle unit: 16-byte loads (8 per lane, 4 lines each, where 4-byte ones were 32), and the 8
// steps' butterflies together: at each distance a lane passes on half of its steps and keeps the sums of the others, so that lane
// i ends with step i (28 shuffles for the sums, 7 for the maxima; one step at a time takes 24 and 24 with one token per lane
// and load).  The additions are those of the butterfly.  (49 million logits: 65 -> 55 us.)
// kSplit: blockIdx.z takes per_slice of the chunks only and leaves their statistics in `partial` [row][chunk] for
// score_fold_stats_kernel (see LogitPlan).
constexpr int kRowStatWarps = 4;
template <bool kSplit>
__global__ void __launch_bounds__(kRowStatWarps * 32)
score_row_stats_kernel(LogitParams P, GroupMap gm, const float* __restrict__ dots, float* __restrict__ lse2,
                       float2* __restrict__ partial, int per_slice) {
  extern __shared__ float2 st_sm[];                            // [4 * chunks][4 rows]
  grid_dependency_wait();
  const int unit = P.unit0 + blockIdx.y;
  const int h = unit % P.Hkv;
  const int rows = (gm.begin[h + 1] - gm.begin[h]) * P.w;
  const int r0 = blockIdx.x * 4;
  if (r0 >= rows) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 7, rl = lane >> 3;
  const int r = min(r0 + rl, rows - 1);
  const float* src = dots + ((long long)blockIdx.y * P.max_rows + r) * P.np;
  const long long vis = min(P.N - 1, P.q_pos0 + r % P.w);      // the last token the row sees
  __shared__ __align__(16) float step_max[kRowStatWarps][4][kChunkIters];
  __shared__ __align__(16) float2 step_sum[kRowStatWarps][4][kChunkIters];   // (factor of the sum so far, sum of the step)
  const int chunk0 = kSplit ? (int)blockIdx.z * per_slice : 0;
  const int chunks = kSplit ? min(per_slice, P.nchunks - chunk0) : P.nchunks;
  for (int p = warp; p < 4 * chunks; p += kRowStatWarps) {
    const long long base = (long long)(chunk0 + (p >> 2)) * (kChunkIters * kThreads) + (p & 3) * 32 + 4 * sub;
    const float* at = src + base;
    float s[kChunkIters][4];
    if (base + (kChunkIters - 1) * kThreads + 3 <= vis) {      // all of them are there and seen
#pragma unroll
      for (int it = 0; it < kChunkIters; ++it) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(at + it * kThreads));
        s[it][0] = x.x * P.scale_log2e; s[it][1] = x.y * P.scale_log2e; s[it][2] = x.z * P.scale_log2e; s[it][3] = x.w * P.scale_log2e;
      }
    } else {
      const int left = (int)max(-1LL, min(vis - base, (long long)kChunkIters * kThreads));   // offsets up to here count
#pragma unroll
      for (int it = 0; it < kChunkIters; ++it) {
        const int o = it * kThreads;
        const float4 x = o <= left ? __ldg(reinterpret_cast<const float4*>(at + o)) : make_float4(0.f, 0.f, 0.f, 0.f);
        s[it][0] = o <= left ? x.x * P.scale_log2e : -INFINITY;
        s[it][1] = o + 1 <= left ? x.y * P.scale_log2e : -INFINITY;
        s[it][2] = o + 2 <= left ? x.z * P.scale_log2e : -INFINITY;
        s[it][3] = o + 3 <= left ? x.w * P.scale_log2e : -INFINITY;
      }
    }
    // the maximum of step `sub`, then of the steps up to it
    float mw[kChunkIters];
#pragma unroll
    for (int it = 0; it < kChunkIters; ++it) mw[it] = fmaxf(fmaxf(s[it][0], s[it][1]), fmaxf(s[it][2], s[it][3]));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const bool up = sub & o;
#pragma unroll
      for (int k = 0; k < o; ++k)
        mw[k] = fmaxf(up ? mw[k + o] : mw[k], __shfl_xor_sync(0xffffffffu, up ? mw[k] : mw[k + o], o));
    }
    float m = mw[0];
#pragma unroll
    for (int o = 1; o < kChunkIters; o <<= 1) {
      const float x = __shfl_up_sync(0xffffffffu, m, o, kChunkIters);
      m = fmaxf(m, x);                                         // (a lane without a source gets its own)
    }
    const float m_below = __shfl_up_sync(0xffffffffu, m, 1, kChunkIters), m_before = sub ? m_below : -INFINITY;
    step_max[warp][rl][sub] = m;
    __syncwarp();
    float ms[kChunkIters];
#pragma unroll
    for (int it = 0; it < kChunkIters; it += 4) *reinterpret_cast<float4*>(ms + it) = *reinterpret_cast<const float4*>(&step_max[warp][rl][it]);
#pragma unroll
    for (int it = 0; it < kChunkIters; ++it)
#pragma unroll
      for (int i = 0; i < 4; ++i) s[it][i] = (ms[it] == -INFINITY) ? 0.f : exp2f(s[it][i] - ms[it]);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {                          // distances 16, 8, 4 of the butterfly
      const bool up = sub & o;
#pragma unroll
      for (int k = 0; k < o; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          s[k][i] = (up ? s[k + o][i] : s[k][i]) + __shfl_xor_sync(0xffffffffu, up ? s[k][i] : s[k + o][i], o);
    }
    const float l_w = (s[0][0] + s[0][2]) + (s[0][1] + s[0][3]);   // 2 and 1
    step_sum[warp][rl][sub] = make_float2(m == -INFINITY ? 0.f : exp2f(m_before - m), l_w);
    __syncwarp();
    if (sub == kChunkIters - 1) {                              // (its maximum is that of all steps)
      float lsum = 0.f;
#pragma unroll
      for (int it = 0; it < kChunkIters; ++it) {
        const float2 x = step_sum[warp][rl][it];
        lsum = fmaf(lsum, x.x, x.y);
      }
      st_sm[p * 4 + rl] = make_float2(m, lsum);
    }
    __syncwarp();
  }
  __syncthreads();
  // per chunk: the four warps' statistics
  for (int i = threadIdx.x; i < chunks * 4; i += kRowStatWarps * 32) {
    const int ch = i >> 2, rr = i & 3;
    float M = -INFINITY;
#pragma unroll
    for (int wv = 0; wv < 4; ++wv) M = fmaxf(M, st_sm[(ch * 4 + wv) * 4 + rr].x);
    float Lsum = 0.f;
    if (M > -INFINITY) {
#pragma unroll
      for (int wv = 0; wv < 4; ++wv) {
        const float2 v = st_sm[(ch * 4 + wv) * 4 + rr];
        Lsum += v.y * exp2f(v.x - M);
      }
    }
    if (kSplit) {
      if (r0 + rr < rows) partial[((long long)blockIdx.y * P.max_rows + r0 + rr) * P.nchunks + chunk0 + ch] = make_float2(M, Lsum);
    } else {
      st_sm[ch * 16 + rr] = make_float2(M, Lsum);              // (read by nobody else: slot wv = 0 of this chunk and row)
    }
  }
  if (kSplit) return;
  __syncthreads();
  if (threadIdx.x < 4 && r0 + threadIdx.x < rows) {
    float M = -INFINITY;
    for (int i = 0; i < P.nchunks; ++i) M = fmaxf(M, st_sm[i * 16 + threadIdx.x].x);
    float Lsum = 0.f;
    for (int i = 0; i < P.nchunks; ++i) {
      const float2 v = st_sm[i * 16 + threadIdx.x];
      if (v.x > -INFINITY) Lsum += v.y * exp2f(v.x - M);
    }
    lse2[(long long)blockIdx.y * P.max_rows + r0 + threadIdx.x] = M + log2f(Lsum);
  }
}

// The chunks' statistics of a row folded to its log-sum-exp, a warp per row: the lanes fetch 32 chunks at a time, the sum is
// taken in the order of the chunks, as score_row_stats_kernel takes it.
__global__ void __launch_bounds__(kThreads)
score_fold_stats_kernel(LogitParams P, GroupMap gm, const float2* __restrict__ partial, float* __restrict__ lse2) {
  grid_dependency_wait();
  const int h = (P.unit0 + blockIdx.y) % P.Hkv;
  const int row = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= (gm.begin[h + 1] - gm.begin[h]) * P.w) return;
  const float2* src = partial + ((long long)blockIdx.y * P.max_rows + row) * P.nchunks;
  float M = -INFINITY;
  for (int i = lane; i < P.nchunks; i += 32) M = fmaxf(M, __ldg(&src[i].x));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float Lsum = 0.f;
  for (int i0 = 0; i0 < P.nchunks; i0 += 32) {
    const float2 v = i0 + lane < P.nchunks ? __ldg(src + i0 + lane) : make_float2(-INFINITY, 0.f);
    const float f = exp2f(v.x - M);                            // (0 where no key is seen, and there the sum is 0 too)
#pragma unroll
    for (int i = 0; i < 32; ++i) Lsum += __shfl_sync(0xffffffffu, v.y, i) * __shfl_sync(0xffffffffu, f, i);
  }
  if (lane == 0) lse2[(long long)blockIdx.y * P.max_rows + row] = M + log2f(Lsum);
}

// Eqs. 14-15 from the kept logits: four tokens per thread, 16 rows in flight.  kMean: agg_task is the mean.
template <bool kMean>
__global__ void __launch_bounds__(kThreads)
score_emit_logits_kernel(LogitParams P, GroupMap gm, const float* __restrict__ dots, const float* __restrict__ lse2,
                         float* __restrict__ s_group) {
  __shared__ float neg_lse[kThreads];
  grid_dependency_wait();
  const int unit = P.unit0 + blockIdx.y;
  const int h = unit % P.Hkv;
  const long long c = ((long long)blockIdx.x * kThreads + threadIdx.x) * 4;
  const int members = gm.begin[h + 1] - gm.begin[h];
  // (a thread behind the end reads the last four tokens again)
  const float4* src = reinterpret_cast<const float4*>(dots + (long long)blockIdx.y * P.max_rows * P.np + min(c, P.np - 4));
  const float* lse = lse2 + (long long)blockIdx.y * P.max_rows;
  const long long step = P.np / 4;
  const int all_from = (int)min((long long)P.w, max(0LL, c + 3 - P.q_pos0));      // window rows from here on see all four tokens
  float gacc[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) gacc[e] = (P.agg_group == KVC_AGG_MAX) ? -INFINITY : 0.f;
  for (int mi = 0; mi < members; ++mi) {
    float tacc[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) tacc[e] = kMean ? 0.f : -INFINITY;
    for (int r0 = 0; r0 < P.w; r0 += kThreads) {
      const int nr = min(kThreads, P.w - r0);
      __syncthreads();
      if (threadIdx.x < nr) neg_lse[threadIdx.x] = -__ldg(lse + threadIdx.x);
      __syncthreads();
      auto row = [&](const float4 d, const int r, const bool masked) {
        const float nl = neg_lse[r];
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float t = fmaf(dv[e], P.scale_log2e, nl);              // log2 of the attention weight
          if (masked && c + e > P.q_pos0 + r0 + r) t = -INFINITY;
          if (kMean) tacc[e] += exp2f(t); else tacc[e] = fmaxf(tacc[e], t);
        }
      };
      int r = 0;
      for (; r + 16 <= nr; r += 16) {
        float4 d[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) d[i] = __ldg(src + i * step);
        src += 16 * step;
        if (r0 + r >= all_from) {
#pragma unroll
          for (int i = 0; i < 16; ++i) row(d[i], r + i, false);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) row(d[i], r + i, true);
        }
      }
      for (; r < nr; ++r) { row(__ldg(src), r, true); src += step; }
      lse += nr;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float s_task = kMean ? tacc[e] / (float)P.w : exp2f(tacc[e]);
      gacc[e] = (P.agg_group == KVC_AGG_MAX) ? fmaxf(gacc[e], s_task) : gacc[e] + s_task;
    }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (P.agg_group == KVC_AGG_MEAN) gacc[e] /= (float)members;
    if (c + e < P.N) s_group[(long long)unit * P.N + c + e] = gacc[e];
  }
}

// The kernel below for up to kAugHeads = 8 (4) KV heads: a thread has all heads' group aggregates of its token in registers, reads
// the row tiles' parts of all heads together and writes every score once.  Bound by HBM / L2: parts once, scores once.
// (28 layers, 4 heads, 4 row tiles, N = 131072: 129 -> 56 us; 32 layers, 8 heads, 16 row tiles, N = 4096: 43 -> 19.)
template <int kAugHeads, bool kParts>
__global__ void __launch_bounds__(256, !kParts ? 6 : kAugHeads == 8 ? 4 : 7)
score_augment_heads_kernel(float* __restrict__ s, const float* __restrict__ parts, int row_tiles, int tiles_per_head,
                           int agg_task, int w, const float* __restrict__ vnorm, int G, int agg_group, int augment, int Hkv,
                           long long N) {
  grid_dependency_wait();
  const long long c = (long long)blockIdx.x * 256 + threadIdx.x;
  if (c >= N) return;
  const long long at = (long long)blockIdx.y * Hkv * N + c;            // blockIdx.y = (layer, sequence)
  float* base = s + at;
  float acc[kAugHeads];
  if constexpr (kParts) {
    const long long tile_stride = (long long)gridDim.y * Hkv * N;       // one [L*Bt*Hkv][N] block per row tile
    const float* p = parts + at;
    auto fetch = [&](int t, float (&v)[kAugHeads]) {
#pragma unroll
      for (int h = 0; h < kAugHeads; ++h) v[h] = h < Hkv ? __ldg(p + t * tile_stride + (long long)h * N) : 0.f;
    };
    if (tiles_per_head > 1) {
#pragma unroll
      for (int h = 0; h < kAugHeads; ++h) acc[h] = (agg_group == KVC_AGG_MAX) ? -INFINITY : 0.f;
      for (int j = 0; j < row_tiles / tiles_per_head; ++j) {             // the query heads of the group
        float ht[kAugHeads];
        fetch(j * tiles_per_head, ht);
#pragma unroll 2
        for (int t = 1; t < tiles_per_head; ++t) {
          float v[kAugHeads];
          fetch(j * tiles_per_head + t, v);
#pragma unroll
          for (int h = 0; h < kAugHeads; ++h) ht[h] = (agg_task == KVC_AGG_MAX) ? fmaxf(ht[h], v[h]) : ht[h] + v[h];
        }
#pragma unroll
        for (int h = 0; h < kAugHeads; ++h) {
          if (agg_task == KVC_AGG_MEAN) ht[h] = ht[h] / (float)w;
          acc[h] = (agg_group == KVC_AGG_MAX) ? fmaxf(acc[h], ht[h]) : acc[h] + ht[h];
        }
      }
    } else {
      fetch(0, acc);
#pragma unroll 2
      for (int t = 1; t < row_tiles; ++t) {
        float v[kAugHeads];
        fetch(t, v);
#pragma unroll
        for (int h = 0; h < kAugHeads; ++h) acc[h] = (agg_group == KVC_AGG_MAX) ? fmaxf(acc[h], v[h]) : acc[h] + v[h];
      }
    }
#pragma unroll
    for (int h = 0; h < kAugHeads; ++h) if (agg_group == KVC_AGG_MEAN) acc[h] = acc[h] / (float)G;
  } else {
#pragma unroll
    for (int h = 0; h < kAugHeads; ++h) acc[h] = h < Hkv ? base[(long long)h * N] : 0.f;
  }
  if (vnorm != nullptr) {
#pragma unroll
    for (int h = 0; h < kAugHeads; ++h) if (h < Hkv) acc[h] *= __ldg(vnorm + at + (long long)h * N);
  }
  float mean = 0.f;
  if (augment) {
    float sum = 0.f;
#pragma unroll
    for (int h = 0; h < kAugHeads; ++h) if (h < Hkv) sum += acc[h];
    mean = sum / (float)Hkv;
#pragma unroll
    for (int h = 0; h < kAugHeads; ++h) acc[h] += mean;
  }
#pragma unroll
  for (int h = 0; h < kAugHeads; ++h) if (h < Hkv) base[(long long)h * N] = acc[h];
}

// Eq. 16: S[h, c] = S_group[h, c] + (1/Hkv) sum_i S_group[i, c], in place.  With row tiles, first
// Eq. 15 from the tiles' partial aggregates (sum or max over the tile's query heads), in tile order.
// With vnorm (App. A.1.3), the group aggregate is multiplied by the token's value norm before Eq. 16.
// With tiles_per_head > 1 (windows longer than 128 rows) a row tile holds one query head's partial
// Eq. 14 -- the maximum or the sum of the attention weights over the tile's rows -- and Eq. 14 is
// completed over the head's tiles (the sum divided by w) before Eq. 15, heads in ascending order.
__global__ void score_augment_kernel(float* __restrict__ s, const float* __restrict__ parts, int row_tiles,
                                     int tiles_per_head, int agg_task, int w, const float* __restrict__ vnorm, int G,
                                     int agg_group, int augment, int Hkv, long long N, long long total) {
  grid_dependency_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const long long lb = i / N, c = i - lb * N;
  float* base = s + lb * Hkv * N + c;
  if (row_tiles > 1 || vnorm != nullptr) {
    const long long tile_stride = (total / N) * Hkv * N;          // one [L*Bt*Hkv][N] block per row tile
    const float* pbase = parts + lb * Hkv * N + c;
    for (int h = 0; h < Hkv; ++h) {
      float acc;
      if (row_tiles > 1 && tiles_per_head > 1) {
        acc = (agg_group == KVC_AGG_MAX) ? -INFINITY : 0.f;
        for (int j = 0; j < row_tiles / tiles_per_head; ++j) {       // the query heads of the group
          float ht = pbase[(long long)(j * tiles_per_head) * tile_stride + (long long)h * N];
          for (int t = 1; t < tiles_per_head; ++t) {
            const float v = pbase[(long long)(j * tiles_per_head + t) * tile_stride + (long long)h * N];
            ht = (agg_task == KVC_AGG_MAX) ? fmaxf(ht, v) : ht + v;
          }
          if (agg_task == KVC_AGG_MEAN) ht = ht / (float)w;
          acc = (agg_group == KVC_AGG_MAX) ? fmaxf(acc, ht) : acc + ht;
        }
        if (agg_group == KVC_AGG_MEAN) acc = acc / (float)G;
      } else if (row_tiles > 1) {
        acc = pbase[(long long)h * N];
        for (int t = 1; t < row_tiles; ++t) {
          const float v = pbase[(long long)t * tile_stride + (long long)h * N];
          acc = (agg_group == KVC_AGG_MAX) ? fmaxf(acc, v) : acc + v;
        }
        if (agg_group == KVC_AGG_MEAN) acc = acc / (float)G;
      } else {
        acc = base[(long long)h * N];
      }
      if (vnorm != nullptr) acc *= vnorm[lb * Hkv * N + (long long)h * N + c];
      base[(long long)h * N] = acc;
    }
  }
  if (!augment) return;
  float sum = 0.f;
  for (int h = 0; h < Hkv; ++h) sum += base[(long long)h * N];
  const float mean = sum / (float)Hkv;
  for (int h = 0; h < Hkv; ++h) base[(long long)h * N] += mean;
}

template <typename T, int D>
kvc_status run(const Problem& P, const GroupMap& gm, const LayerPtrs& q, const LayerPtrs& k,
               float* scores, float2* partial, float* lse2, int nchunks, cudaStream_t st) {
  ScoreParams sp;
  sp.L = P.L; sp.Bt = P.Bt; sp.Hq = P.Hq; sp.Hkv = P.Hkv; sp.w = P.w;
  sp.N = P.N; sp.q_pos0 = P.q_pos0;
  sp.qs0 = P.qs[0]; sp.qs1 = P.qs[1]; sp.qs2 = P.qs[2];
  sp.kvs0 = P.kvs[0]; sp.kvs1 = P.kvs[1]; sp.kvs2 = P.kvs[2];
  sp.scale_log2e = P.scale * kLog2e;
  sp.agg_task = P.agg_task; sp.agg_group = P.agg_group;
  sp.nchunks = nchunks;
  KvOfQ map;
  for (int h = 0; h < P.Hkv; ++h)
    for (int i = gm.begin[h]; i < gm.begin[h + 1]; ++i) map.kv[gm.qh[i]] = (int16_t)h;

  const long long rows = (long long)P.L * P.Bt * P.Hq * P.w;
  score_stats_kernel<T, D><<<dim3(nchunks, P.Hq, P.L * P.Bt), kThreads, 0, st>>>(sp, map, q, k, partial);
  KVC_LAUNCH_CHECK("score_stats_kernel");
  score_lse_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(partial, lse2, rows, nchunks);
  KVC_LAUNCH_CHECK("score_lse_kernel");
  score_emit_kernel<T, D><<<dim3((unsigned)((P.N + kThreads - 1) / kThreads), P.Hkv, P.L * P.Bt),
                            kThreads, 0, st>>>(sp, gm, q, k, lse2, scores);
  KVC_LAUNCH_CHECK("score_emit_kernel");
  return KVC_OK;
}

// Few rows over many tokens: the two sweeps.  They are bound by reading K twice then, while the product multiplies 32 rows whatever
// there are, and for bf16 its operands wait for their conversion.  The line rises with the tokens (short contexts of
// few units do not fill the SMs with sweeps).  Product over sweeps, fp32 with one query head per KV head: 256K tokens of 64,
// 2 rows 1.16, 3 rows 1.05, 4 rows 0.96; of 128, 1 row 1.12, 2 rows 1.03, 3 rows 0.96; with two query heads 0.89 and
// less.  bf16: 256K tokens of 64, 5 rows 1.12, 8 rows 0.88, two heads of 1 row 1.23, of 3 rows 0.95; 1M tokens, 8 rows 1.22,
// two heads of 4 rows 1.05, of 6 rows 0.91, four heads of 1 row 1.02, of 2 rows 0.90.
bool few_rows(const Problem& P) {
  struct Line { long long tokens; int rows; };
  static constexpr Line kBf16[] = {{2048 << 10, 13}, {768 << 10, 10}, {352 << 10, 8}, {224 << 10, 6}, {112 << 10, 3}};
  static constexpr Line kF32[] = {{3072 << 10, 5}, {352 << 10, 4}, {224 << 10, 3}, {112 << 10, 2}};
  const long long tokens = (long long)P.L * P.Bt * P.Hkv * P.N, rows = (long long)P.max_group * P.w;
  if (P.dtype == KVC_BF16) {
    for (const Line& at : kBf16) if (tokens >= at.tokens) return rows + 2 * (P.max_group - 1) <= at.rows;
  } else if (P.max_group == 1) {
    for (const Line& at : kF32) if (tokens >= at.tokens) return rows * (P.d / 64) <= at.rows;
  }
  return false;
}

// How the units are cut into groups whose logits fit the buffer; units_per_group = 0: the two sweeps, because one unit alone does
// not fit, has few rows, or because the problem belongs to the tensor cores and gets here only when its strides do not suit them.
struct LogitPlan {
  long long np, units;
  int max_rows, units_per_group;
  int slices, per_slice;        // of the statistics: how many CTAs share the chunks of a row, and the chunks of each
  size_t dots_bytes, lse_bytes, partial_bytes;
};
LogitPlan logit_plan(const Problem& P) {
  LogitPlan p;
  p.np = (P.N + 3) / 4 * 4;
  p.units = (long long)P.L * P.Bt * P.Hkv;
  const long long rows = (long long)P.max_group * P.w;
  const long long unit_bytes = rows * p.np * (long long)sizeof(float);
  const long long nchunks = (P.N + kChunkIters * kThreads - 1) / (kChunkIters * kThreads);
  p.max_rows = (int)rows;
  p.units_per_group = 0;
  p.slices = 1;
  p.per_slice = (int)nchunks;
  p.dots_bytes = p.lse_bytes = p.partial_bytes = 0;
  if (unit_bytes > (long long)kLogitsCap || score_sm100_shape_ok(P) || few_rows(P)) return p;
  const long long per = (long long)kLogitsCap / unit_bytes < 65535 ? (long long)kLogitsCap / unit_bytes : 65535;
  const long long groups = (p.units + per - 1) / per;
  p.units_per_group = (int)((p.units + groups - 1) / groups);   // groups of even size
  p.dots_bytes = align_up((size_t)p.units_per_group * unit_bytes);
  p.lse_bytes = align_up((size_t)p.units_per_group * rows * sizeof(float));
  // A CTA of the statistics takes four rows over the whole context; where these CTAs are few and the context is long, slices of
  // the chunks instead, about eight CTAs per SM, for one small launch more.  (A constant stands for the SMs: the workspace must not
  // depend on the device.  fp32, heads of 64: 32 rows of 65536 tokens 107 -> 27 us per call, 16 units of 64 rows of 262144 tokens
  // 8740 -> 2388; with 4 chunks it costs what it gains; half and twice as many slices are within 1 %.)
  constexpr long long kStatCtas = 8 * 148;
  const long long ctas = (long long)p.units_per_group * ((rows + 3) / 4);
  if (ctas * 2 <= kStatCtas && nchunks >= 5) {
    const long long want = kStatCtas / ctas;
    p.per_slice = (int)((nchunks + want - 1) / want);
    p.slices = (int)((nchunks + p.per_slice - 1) / p.per_slice);
    p.partial_bytes = align_up((size_t)p.units_per_group * rows * nchunks * sizeof(float2));
  }
  return p;
}

template <typename T, int D, int kTT>
kvc_status run_logits_t(const Problem& P, const GroupMap& gm, const LayerPtrs& q, const LayerPtrs& k, float* scores,
                      const LogitPlan& pl, int sms, char* ws, int* device_status, cudaStream_t st) {
  constexpr int kTileRow = kLogitTileRows<kTT>;
  constexpr int kSmem = (2 * kTileTok + kTileRow) * (D + 4) * (int)sizeof(float);
  KVC_CUDA(cudaFuncSetAttribute(score_logits_kernel<T, D, kTT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
  const int row_tiles = (pl.max_rows + kTileRow - 1) / kTileRow;
  const int tok_tiles = (int)((P.N + kTileTok - 1) / kTileTok);
  LogitParams lp;
  lp.Bt = P.Bt; lp.Hkv = P.Hkv; lp.w = P.w; lp.max_rows = pl.max_rows;
  lp.N = P.N; lp.np = pl.np; lp.q_pos0 = P.q_pos0;
  lp.qs0 = P.qs[0]; lp.qs1 = P.qs[1]; lp.qs2 = P.qs[2];
  lp.kvs0 = P.kvs[0]; lp.kvs1 = P.kvs[1]; lp.kvs2 = P.kvs[2];
  lp.scale_log2e = P.scale * kLog2e;
  lp.agg_task = P.agg_task; lp.agg_group = P.agg_group;
  lp.nchunks = (int)((P.N + kChunkIters * kThreads - 1) / (kChunkIters * kThreads));
  const auto stat_kernel = pl.slices > 1 ? score_row_stats_kernel<true> : score_row_stats_kernel<false>;
  // (at most 28 chunks: unsliced with 5 and more of them are only groups of 593 CTAs and more, whose logits fill the buffer with
  // 28 290 tokens a row; slices hold a 1184th of the buffer each, rounded up)
  const size_t stat_smem = (size_t)pl.per_slice * 16 * sizeof(float2);
  float* dots = reinterpret_cast<float*>(ws);
  float* lse2 = reinterpret_cast<float*>(ws + pl.dots_bytes);
  float2* partial = reinterpret_cast<float2*>(ws + pl.dots_bytes + pl.lse_bytes);
  for (long long u0 = 0; u0 < pl.units; u0 += pl.units_per_group) {
    const unsigned n = (unsigned)(pl.units - u0 < pl.units_per_group ? pl.units - u0 : pl.units_per_group);
    lp.unit0 = (int)u0;
    const long long items = (long long)n * row_tiles * tok_tiles;
    KVC_CUDA(launch_dependent(score_logits_kernel<T, D, kTT>, dim3((unsigned)(items < sms ? items : sms)), dim3(kLogitThreads),
                              (size_t)kSmem, st, lp, gm, q, k, dots, row_tiles, tok_tiles, (int)items, device_status));
    KVC_LAUNCH_CHECK("score_logits_kernel");
    KVC_CUDA(launch_dependent(stat_kernel, dim3((unsigned)((pl.max_rows + 3) / 4), n, (unsigned)pl.slices),
                              dim3(kRowStatWarps * 32), stat_smem, st, lp, gm, (const float*)dots, lse2, partial, pl.per_slice));
    KVC_LAUNCH_CHECK("score_row_stats_kernel");
    if (pl.slices > 1) {
      KVC_CUDA(launch_dependent(score_fold_stats_kernel, dim3((unsigned)((pl.max_rows + kThreads / 32 - 1) / (kThreads / 32)), n),
                                dim3(kThreads), 0, st, lp, gm, (const float2*)partial, lse2));
      KVC_LAUNCH_CHECK("score_fold_stats_kernel");
    }
    KVC_CUDA(launch_dependent(P.agg_task == KVC_AGG_MEAN ? score_emit_logits_kernel<true> : score_emit_logits_kernel<false>,
                              dim3((unsigned)((P.N + 4 * kThreads - 1) / (4 * kThreads)), n), dim3(kThreads), 0, st, lp, gm,
                              (const float*)dots, (const float*)lse2, scores));
    KVC_LAUNCH_CHECK("score_emit_logits_kernel");
  }
  return KVC_OK;
}

template <typename T, int D>
kvc_status run_logits(const Problem& P, const GroupMap& gm, const LayerPtrs& q, const LayerPtrs& k, float* scores,
                      const LogitPlan& pl, char* ws, int* device_status, cudaStream_t st) {
  int dev = 0, sms = 0;
  KVC_CUDA(cudaGetDevice(&dev));
  KVC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // (in items of 32 rows the product reads twice the operands per multiply-add: only where items of 128 rows would be mostly
  // empty or fewer than the SMs)
  const long long items = (long long)pl.units_per_group * ((pl.max_rows + 127) / 128) * ((P.N + kTileTok - 1) / kTileTok);
  if (pl.max_rows <= 32 || items < sms) return run_logits_t<T, D, 2>(P, gm, q, k, scores, pl, sms, ws, device_status, st);
  return run_logits_t<T, D, 8>(P, gm, q, k, scores, pl, sms, ws, device_status, st);
}

}  // namespace

static int generic_nchunks(const Problem& P) {
  const long long per = (long long)kChunkIters * kThreads;
  return (int)((P.N + per - 1) / per);
}

size_t score_generic_workspace_bytes(const Problem& P) {
  const LogitPlan pl = logit_plan(P);
  if (pl.units_per_group > 0) return pl.dots_bytes + pl.lse_bytes + pl.partial_bytes;
  const size_t rows = (size_t)P.L * P.Bt * P.Hq * P.w;
  return align_up(rows * generic_nchunks(P) * sizeof(float2)) + align_up(rows * sizeof(float));
}

kvc_status launch_score_augment(const Problem& P, float* scores, const float* parts, int row_tiles,
                                int tiles_per_head, const float* vnorm, cudaStream_t st) {
  if (!P.augment && row_tiles <= 1 && vnorm == nullptr) return KVC_OK;
  if (P.Hkv <= 8) {
    const auto kernel = row_tiles > 1 ? (P.Hkv <= 4 ? score_augment_heads_kernel<4, true> : score_augment_heads_kernel<8, true>)
                                      : score_augment_heads_kernel<8, false>;
    KVC_CUDA(launch_dependent(kernel, dim3((unsigned)((P.N + 255) / 256), (unsigned)(P.L * P.Bt)), dim3(256), 0,
                              st, scores, parts, row_tiles, tiles_per_head, P.agg_task, P.w, vnorm, P.max_group, P.agg_group,
                              P.augment, P.Hkv, P.N));
    KVC_LAUNCH_CHECK("score_augment_heads_kernel");
    return KVC_OK;
  }
  const long long total = (long long)P.L * P.Bt * P.N;
  KVC_CUDA(launch_dependent(score_augment_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, st,
                            scores, parts, row_tiles, tiles_per_head, P.agg_task, P.w, vnorm, P.max_group, P.agg_group,
                            P.augment, P.Hkv, P.N, total));
  KVC_LAUNCH_CHECK("score_augment_kernel");
  return KVC_OK;
}

kvc_status launch_score_generic(const Problem& P, const GroupMap& gm, const LayerPtrs& q,
                                const LayerPtrs& k, float* scores, const float* vnorm, int* device_status, void* ws,
                                size_t ws_bytes, cudaStream_t st) {
  if (ws_bytes < score_generic_workspace_bytes(P)) {
    set_error("score: workspace too small");
    return KVC_ERR_WORKSPACE;
  }
  const LogitPlan pl = logit_plan(P);
  if (pl.units_per_group > 0) {
    char* w = reinterpret_cast<char*>(ws);
    kvc_status r;
    if (P.dtype == KVC_BF16)
      r = P.d == 64 ? run_logits<__nv_bfloat16, 64>(P, gm, q, k, scores, pl, w, device_status, st)
                    : run_logits<__nv_bfloat16, 128>(P, gm, q, k, scores, pl, w, device_status, st);
    else
      r = P.d == 64 ? run_logits<float, 64>(P, gm, q, k, scores, pl, w, device_status, st) : run_logits<float, 128>(P, gm, q, k, scores, pl, w, device_status, st);
    if (r != KVC_OK) return r;
    return launch_score_augment(P, scores, nullptr, 1, 1, vnorm, st);
  }
  if (device_status) KVC_CUDA(cudaMemsetAsync(device_status, 0, sizeof(int), st));
  const size_t rows = (size_t)P.L * P.Bt * P.Hq * P.w;
  const int nchunks = generic_nchunks(P);
  float2* partial = reinterpret_cast<float2*>(ws);
  float* lse2 = reinterpret_cast<float*>(reinterpret_cast<char*>(ws) +
                                         align_up(rows * nchunks * sizeof(float2)));
  kvc_status s;
  if (P.dtype == KVC_BF16) {
    if (P.d == 64) s = run<__nv_bfloat16, 64>(P, gm, q, k, scores, partial, lse2, nchunks, st);
    else s = run<__nv_bfloat16, 128>(P, gm, q, k, scores, partial, lse2, nchunks, st);
  } else {
    if (P.d == 64) s = run<float, 64>(P, gm, q, k, scores, partial, lse2, nchunks, st);
    else s = run<float, 128>(P, gm, q, k, scores, partial, lse2, nchunks, st);
  }
  if (s != KVC_OK) return s;
  return launch_score_augment(P, scores, nullptr, 1, 1, vnorm, st);
}

}  // namespace kvc
