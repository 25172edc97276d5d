// Layer-adaptive budget allocation (Eqs. 20-22).
//
// Per sequence, the pool P holds the L * N composite scores; the B largest are kept and N_l is
// how many of them lie in layer l.  Because composite[l, :] is non-increasing, the kept set of a
// layer is a prefix, so the answer is fixed by the B-th largest pooled value T:
//   N_l = #{k : I[l, k] > T}  +  (a share of the entries equal to T, handed out in layer order
//                                 until the budget is met -- the total order (I desc, l asc, k asc)).
// Two ways to T, both over the 32-bit order-preserving keys:
//   * pools of up to 256 rows: one kernel, one CTA per sequence, which only ever looks at a few
//     thousand entries.  Every row keeps a window of positions that must hold its boundary; per
//     round the CTA samples each window at equal distances, and the samples' weighted ranks (their
//     block sizes as weights) bracket T between two sample values, which cuts every window to the
//     blocks between them.  A value with so many copies that the windows stop shrinking is located
//     exactly in every row (32-way searches) and either is T or leaves the windows; when at most
//     2048 entries are left T is read off them.  The rounds are bounded; past the bound T is found
//     by bisection over the key range with exact counts.
//   * larger pools: a most-significant-digit radix select -- four histogram passes over the pool
//     (each CTA re-derives the prefix chosen so far from the previous passes' global histograms),
//     then one small kernel does the per-row searches and the tie hand-out.
//
// The rows of the pool are the layers (Eqs. 20-22) or, for the unstructured variant of App. A.2,
// the (layer, head) pairs with the heads' sorted scores as rows.  With a per-layer minimum m the
// first m entries of every row are kept outright and stay out of the pool.
#include <atomic>

#include "kvc_internal.cuh"

namespace kvc {
namespace {

constexpr int kRadix = 256;
constexpr int kHistThreads = 256;
constexpr int kItemsPerThread = 16;

// Select state after `passes` completed passes: the key prefix (high bits) and the rank that is
// still to be located inside that prefix bucket.  rank is 1-based among ascending keys.
// Where row r of sequence b starts: rows are layers of composite [L, Bt, N] (heads_per_row = 1) or
// (layer, head) pairs of sorted scores [L, Bt, Hkv, N] (heads_per_row = Hkv).
__device__ __forceinline__ long long row_start(long long r, int b, int Bt, int hpr, long long N) {
  const long long l = r / hpr, h = r - l * hpr;
  return ((l * Bt + b) * hpr + h) * N;
}

struct SelectState {
  uint32_t prefix;
  unsigned long long rank;
};

// hist: [4][256] counts of digit (MSD first) among keys whose higher digits equal the prefix.
// Walks the completed passes: in each, the digit whose cumulative count first reaches the rank.
// Cooperative: the first 256 threads of the block take one bin each (blockDim.x >= 256); the
// result is valid in every thread after the call.  `scratch` is 16 words of shared memory.
__device__ inline SelectState derive_state(const unsigned int* __restrict__ hist_b, int passes,
                                           unsigned long long rank0, unsigned long long* scratch) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  SelectState s;
  s.prefix = 0;
  s.rank = rank0;
  for (int p = 0; p < passes; ++p) {
    unsigned long long c = 0, incl = 0;
    if (tid < kRadix) {
      c = hist_b[p * kRadix + tid];
      incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
      }
      if (lane == 31) scratch[warp] = incl;
    }
    __syncthreads();
    if (tid == 0) { scratch[8] = kRadix - 1; scratch[9] = 0; }     // default: the last digit
    __syncthreads();
    if (tid < kRadix) {
      unsigned long long before = 0;
      for (int wv = 0; wv < warp; ++wv) before += scratch[wv];
      incl += before;
      const unsigned long long excl = incl - c;
      if (excl < s.rank && s.rank <= incl) { scratch[8] = (unsigned long long)tid; scratch[9] = excl; }
    }
    __syncthreads();
    if (s.rank > 0) {
      const unsigned long long total_last = scratch[9];
      s.prefix |= (uint32_t)scratch[8] << (24 - 8 * p);
      // when the rank lies beyond the total (cannot happen for a valid budget) the last digit
      // was kept with nothing subtracted
      s.rank -= total_last;
    }
    __syncthreads();
  }
  return s;
}

// Clears the histograms of all passes (a kernel rather than a memset, so that it can be launched
// as a programmatic dependent of whatever ran before).
__global__ void __launch_bounds__(1024)
select_clear_kernel(unsigned int* __restrict__ hist) {
  grid_dependency_wait();
  hist[(size_t)blockIdx.x * 4 * kRadix + threadIdx.x] = 0u;
}

// R rows per sequence, each of N entries of which the first `floor` are out of the pool; `budget`
// is what is left to hand out among the others.
__global__ void __launch_bounds__(kHistThreads)
select_hist_kernel(const float* __restrict__ composite, unsigned int* __restrict__ hist, int pass,
                   int R, int Bt, int hpr, long long N, long long floor, long long budget) {
  __shared__ unsigned int sh[kRadix];
  __shared__ unsigned long long scratch[16];
  grid_dependency_wait();
  const int b = blockIdx.y;
  unsigned int* hist_b = hist + (size_t)b * 4 * kRadix;
  for (int i = threadIdx.x; i < kRadix; i += kHistThreads) sh[i] = 0;
  const SelectState st = derive_state(hist_b, pass, (unsigned long long)budget, scratch);
  __syncthreads();
  const uint32_t prefix = st.prefix;
  const int shift = 24 - 8 * pass;
  const uint32_t hi_mask = (pass == 0) ? 0u : (0xffffffffu << (shift + 8));
  const long long M = N - floor;                       // pooled entries per row
  const long long total = (long long)R * M;
  const long long tile = (long long)kHistThreads * kItemsPerThread;
  for (long long t0 = (long long)blockIdx.x * tile; t0 < total; t0 += (long long)gridDim.x * tile) {
    // pooled index -> (row, position) once per tile, then by steps of the block width
    long long i = t0 + threadIdx.x;
    long long r = i / M, kk = i - r * M;
    long long base = row_start(r, b, Bt, hpr, N) + floor;      // (recomputed only when the row changes)
    // all of the thread's loads first ...
    float v[kItemsPerThread];
#pragma unroll
    for (int it = 0; it < kItemsPerThread; ++it) {
      v[it] = 0.f;
      if (i < total) v[it] = composite[base + kk];
      i += kHistThreads;
      kk += kHistThreads;
      if (kk >= M) {
        while (kk >= M) { kk -= M; ++r; }
        base = row_start(r, b, Bt, hpr, N) + floor;
      }
    }
    // ... then the bins.  Consecutive lanes hold consecutive entries of a non-increasing row: equal digits
    // come in runs, and only the first lane of a run adds (its length) to the bin.
    i = t0 + threadIdx.x;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int it = 0; it < kItemsPerThread; ++it, i += kHistThreads) {
      uint32_t digit = 0x100u;                                  // not in the bucket / beyond the pool
      if (i < total) {
        const uint32_t key = score_to_key(v[it]);
        if ((key & hi_mask) == prefix) digit = (key >> shift) & 0xffu;
      }
      const uint32_t prev = __shfl_up_sync(0xffffffffu, digit, 1);
      const bool head = lane == 0 || prev != digit;
      const uint32_t heads = __ballot_sync(0xffffffffu, head);
      if (head && digit < 0x100u) {
        const uint32_t later = lane == 31 ? 0u : (heads >> (lane + 1));
        atomicAdd(&sh[digit], (unsigned int)(later ? __ffs(later) : 32 - lane));
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kRadix; i += kHistThreads)
    if (sh[i]) atomicAdd(&hist_b[pass * kRadix + i], sh[i]);
}

// One warp, kRowsAtOnce non-increasing rows: per row the number of its n entries with key < T (strictly better) and with
// key <= T, by 32-way searches (every step probes 32 positions at once).  The searches -- the first index with key >= T, and
// with key > T, of every row -- take their steps together, so that their loads are in flight at the same time (one after the
// other, a row at a time: 100 rows of 5000 of one value 20.5 us, so 15.4).
template <int kRowsAtOnce>
__device__ __forceinline__ void count_rows_warp(const float* const* row, const uint32_t* n, uint32_t T,
                                                uint32_t* lt, uint32_t* le) {
  constexpr int kS = 2 * kRowsAtOnce;
  const uint32_t lane = threadIdx.x & 31;
  uint32_t lo[kS], hi[kS];                     // the answers lie in [lo, hi]
#pragma unroll
  for (int i = 0; i < kS; ++i) { lo[i] = 0u; hi[i] = n[i >> 1]; }
  for (;;) {
    uint32_t step[kS], key[kS];
    bool there[kS], more = false;
#pragma unroll
    for (int i = 0; i < kS; ++i) {
      step[i] = (hi[i] - lo[i] + 31u) / 32u;                   // probe lo + (lane + 1) * step - 1
      const uint32_t off = (lane + 1u) * step[i] - 1u;         // (all ones where nothing is left)
      there[i] = off < hi[i] - lo[i];
      key[i] = there[i] ? score_to_key(row[i >> 1][lo[i] + off]) : 0u;
      more = more || lo[i] < hi[i];
    }
    if (!more) break;
#pragma unroll
    for (int i = 0; i < kS; ++i) {
      const bool before = there[i] && ((i & 1) == 0 ? key[i] < T : key[i] <= T);   // "the probe sorts before the boundary"
      const uint32_t n_before = __popc(__ballot_sync(0xffffffffu, before));        // (a prefix of the lanes: the row is sorted)
      if (lo[i] >= hi[i]) continue;
      // the boundary lies after probe n_before - 1 and at or before probe n_before
      const uint32_t left = hi[i] - lo[i];
      const uint32_t last = n_before == 32u ? left : min(left, (n_before + 1u) * step[i] - 1u);
      hi[i] = lo[i] + last;
      lo[i] += min(left, n_before * step[i]);
    }
  }
#pragma unroll
  for (int r = 0; r < kRowsAtOnce; ++r) { lt[r] = lo[2 * r]; le[r] = lo[2 * r + 1]; }
}

// `budget` is again what is left to hand out beyond the rows' first `floor` entries.
__global__ void __launch_bounds__(1024)
select_finish_kernel(const float* __restrict__ composite,
                     const unsigned int* __restrict__ hist, int R, int Bt, int hpr, long long N,
                     long long floor, long long budget, int32_t* __restrict__ n_keep,
                     long long* __restrict__ offsets) {
  extern __shared__ long long s_cnt[];               // [R] strictly better than T, [R] at least as good
  long long* s_gt = s_cnt;
  long long* s_ge = s_cnt + R;
  __shared__ unsigned long long scratch[16];
  grid_dependency_wait();
  const int b = blockIdx.x;
  const SelectState st = derive_state(hist + (size_t)b * 4 * kRadix, 4, (unsigned long long)budget, scratch);
  const uint32_t T = st.prefix;
  const int warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  for (int r = warp; r < R; r += n_warps) {
    const float* const row[1] = {composite + row_start(r, b, Bt, hpr, N) + floor};
    const uint32_t n[1] = {budget > 0 ? (uint32_t)(N - floor) : 0u};
    uint32_t gt[1], ge[1];
    count_rows_warp<1>(row, n, T, gt, ge);
    if ((threadIdx.x & 31) == 0) { s_gt[r] = gt[0]; s_ge[r] = ge[0]; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long used = 0;
    for (int r = 0; r < R; ++r) used += s_gt[r];
    long long rem = budget - used;     // entries equal to T still to hand out, in row order
    long long off = 0;
    for (int r = 0; r < R; ++r) {
      long long take = s_ge[r] - s_gt[r];
      if (take > rem) take = rem;
      if (take < 0) take = 0;
      rem -= take;
      const long long n = floor + s_gt[r] + take;
      n_keep[(long long)b * R + r] = (int32_t)n;
      offsets[(long long)b * (R + 1) + r] = off;
      off += n;
    }
    offsets[(long long)b * (R + 1) + R] = off;
  }
}


// ------------------------------------------------------------------------------------------------
// Selection on the sorted rows themselves: one CTA per sequence, no scratch in global memory.
//
// Bound by latency and by the instructions of one CTA: a round is one round trip to L2 for the samples and a few
// block-wide steps on them.  It takes four samples per thread (64 per row for up to 32 rows, 8 for 256) and finds the
// two bracketing sample values by a weighted radix select: a histogram of the block sizes over 2048 equal steps of the
// samples' key range, a scan, and again inside the bracketing bins while these still hold more than a 128th of the
// windows.  (Sorting 1024 samples took 4300 of a round's 9000 clocks and the last step's sort 8000: the kernel takes
// 12.7 us on 32 rows of 32768 where that took 20.2, 10.8 on 32 rows of 1000 where it took 15.5, and 25 on
// 256 rows of 8192 where the six launches of the histogram passes took 72.  With 1024 threads a round is longer, 5200
// clocks for a level of the select alone: all warps issue the same instructions, half of them for samples not needed.)
// ------------------------------------------------------------------------------------------------
constexpr int kSelThreads = 512;
constexpr int kSelItems = 4;              // samples (or, in the last step, entries) per thread
constexpr int kSelMaxRows = 256;          // rows of a pool this kernel takes (fewer samples per row as the rows grow)
constexpr int kSelBits = 11;              // a level of the select; three make up a key
constexpr int kSelBins = 1 << kSelBits;   // four per thread
constexpr int kSelDefaultRounds = 40;     // sampling rounds and exact steps together, before the bisection takes over

struct SelectShared {
  uint32_t hist[kSelBins];                      // block sizes of the samples per bin
  long long base[kSelMaxRows];                  // where the rows' pooled entries start (for the searches)
  int lo[kSelMaxRows], hi[kSelMaxRows];         // the rows' windows: positions < lo are better than T, >= hi worse
  int gt[kSelMaxRows], ge[kSelMaxRows];         // the answer: entries better than T, and at least as good
  int off[kSelMaxRows + 1];                     // running sum of the window lengths (last step)
  int clt[kSelMaxRows], cle[kSelMaxRows];       // entries better than T, at least as good, in the windows (last step)
  uint32_t warp_tot[kSelThreads / 32];
  unsigned long long tot_lt, tot_le;
  uint32_t bin[2], below[2], weight[2];         // of a level: the bin a target falls into, what lies before it, what is in it
  uint32_t rank, width;                         // T is the rank-th best entry inside the windows (1-based); their total length
  uint32_t slack, taken, new_width;
  uint32_t kmin, kmax;                          // range of the round's sample keys
};

// Inclusive sum over the block in thread order.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, SelectShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  if (lane == 31) sh.warp_tot[warp] = v;        // (the previous scan's totals were read before the caller's last barrier)
  __syncthreads();
  return v + __reduce_add_sync(0xffffffffu, lane < warp ? sh.warp_tot[lane] : 0u);
}

// A bracket being narrowed: the keys base .. base + 2^bits - 1 hold the target-th unit of weight (1-based), `target`
// counted from base on.
struct Bracket {
  uint32_t base, target;
  int bits;
  bool active;
};

// One level for the brackets A and B, which are at the same place (B may be the same as A for a single one): histogram
// over kSelBins equal steps, scan, descend into each one's bin.  A bracket stops being active when its bin is one key
// or holds at most `enough`.  `unit`: what most of a lane's items weigh; runs of lanes with the same bin and unit are added
// by their first lane (`other_unit`: the lane's unit differs from its neighbour's; with a run per row, rows of few values all
// added to the same bins; this and the searches two rows at a time: 128 rows of 20000 of four values 31.8 -> 24.7 us).
__device__ __forceinline__ void select_level(SelectShared& sh, const uint32_t (&key)[kSelItems], const uint32_t (&wgt)[kSelItems],
                                          uint32_t unit, bool other_unit, Bracket& A, Bracket& B, uint32_t enough) {
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t base = A.base;
  const int bits = A.bits, shift = bits > kSelBits ? bits - kSelBits : 0;
  const uint32_t reach = bits >= 32 ? 0xffffffffu : (1u << bits) - 1u;
  *reinterpret_cast<uint4*>(&sh.hist[tid * 4]) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSelItems; ++i) {
    const uint32_t rel = key[i] - base;
    const bool in = wgt[i] > 0 && key[i] >= base && rel <= reach;
    const uint32_t d = in ? rel >> shift : 0xffffffffu;
    const uint32_t prev = __shfl_up_sync(0xffffffffu, d, 1);
    const bool head = lane == 0 || other_unit || prev != d;
    const uint32_t heads = __ballot_sync(0xffffffffu, head);
    if (in) {
      if (head) {
        const uint32_t later = lane == 31 ? 0u : heads >> (lane + 1);
        atomicAdd(&sh.hist[d], unit * (uint32_t)(later ? __ffs(later) : 32 - lane));
      }
      if (wgt[i] != unit) atomicAdd(&sh.hist[d], wgt[i] - unit);       // (modulo 2^32)
    }
  }
  __syncthreads();
  const uint4 h4 = *reinterpret_cast<const uint4*>(&sh.hist[tid * 4]);
  const uint32_t h[4] = {h4.x, h4.y, h4.z, h4.w};
  const uint32_t sum = h[0] + h[1] + h[2] + h[3];
  const uint32_t top = block_scan(sum, sh);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const Bracket& X = q == 0 ? A : B;
    uint32_t before = top - sum;
    if (X.active && before < X.target && X.target <= top) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (before < X.target && X.target <= before + h[j]) { sh.bin[q] = tid * 4 + j; sh.below[q] = before; sh.weight[q] = h[j]; }
        before += h[j];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    Bracket& X = q == 0 ? A : B;
    if (!X.active) continue;
    X.base = base + (sh.bin[q] << shift);
    X.target -= sh.below[q];
    X.bits = shift;
    X.active = shift > 0 && sh.weight[q] > enough;
  }
}

__device__ __forceinline__ int bits_of_range(uint32_t lo, uint32_t hi) { return hi > lo ? 32 - __clz(hi - lo) : 0; }

// Exact position of key T in every row's window (32-way searches, two rows at a time per warp): gt / ge of
// the row as absolute pool positions, and their sums over the rows relative to the windows.
__device__ inline void locate_in_windows(const float* __restrict__ composite, SelectShared& sh, int R, uint32_t T) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) { sh.tot_lt = 0; sh.tot_le = 0; }
  __syncthreads();
  constexpr int kWarps = kSelThreads / 32;
  for (int r0 = warp; r0 < R; r0 += 2 * kWarps) {
    const float* row[2];
    uint32_t n[2], lt[2], le[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = r0 + i * kWarps;
      row[i] = nullptr;
      n[i] = 0u;
      if (r < R) {
        row[i] = composite + sh.base[r] + sh.lo[r];
        n[i] = (uint32_t)max(0, sh.hi[r] - sh.lo[r]);
      }
    }
    count_rows_warp<2>(row, n, T, lt, le);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = r0 + i * kWarps;
      if (r < R && lane == 0) {
        sh.gt[r] = sh.lo[r] + (int)lt[i];
        sh.ge[r] = sh.lo[r] + (int)le[i];
        atomicAdd(&sh.tot_lt, (unsigned long long)lt[i]);
        atomicAdd(&sh.tot_le, (unsigned long long)le[i]);
      }
    }
  }
  __syncthreads();
}

// (the host keeps R * (N - floor) below 2^32)
// kFew: up to kSelFewRows rows, which take their start out of shared memory throughout
constexpr int kSelFewRows = 8;
template <bool kFew>
__global__ void __launch_bounds__(kSelThreads)
select_sorted_kernel(const float* __restrict__ composite, int R, int Bt, int hpr, long long N, long long floor,
                     long long budget, int max_rounds, int32_t* __restrict__ n_keep,
                     long long* __restrict__ offsets) {
  __shared__ __align__(16) SelectShared sh;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int M = (int)(N - floor);                      // pooled entries per row
  // threads per row in a round: 16 for up to 32 rows, 2 for 256; kSelItems samples each
  int tshift = 4;
  while ((kSelThreads >> tshift) < R) --tshift;
  const int tpr = 1 << tshift, sshift = tshift + 2;
  static_assert(kSelItems == 4, "sshift");
  const int r = tid >> tshift, sub = tid & (tpr - 1);  // this thread's row and its place among the row's threads
  const int rr0 = r < R ? r : 0, rl0 = kFew ? 0 : rr0 / hpr;
  const float* row = composite + (((long long)rl0 * Bt + b) * hpr + (rr0 - rl0 * hpr)) * N + floor;
  if (tid < R) {
    const int rl = tid / hpr;                          // (32-bit: the 64-bit division of row_start is slow)
    sh.base[tid] = (((long long)rl * Bt + b) * hpr + (tid - rl * hpr)) * N + floor;
    sh.lo[tid] = 0; sh.hi[tid] = M; sh.gt[tid] = 0; sh.ge[tid] = 0;
  }
  if (tid == 0) {
    sh.width = (uint32_t)((unsigned long long)R * (unsigned long long)M);
    sh.rank = budget < (long long)R * M ? (uint32_t)budget : sh.width;
    sh.kmin = 0xffffffffu;
    sh.kmax = 0u;
    sh.slack = sh.taken = sh.new_width = 0u;
  }
  __syncthreads();
  if (kFew) row = composite + sh.base[rr0];
  grid_dependency_wait();                              // (everything above overlapped the end of the kernel before this one)
  if (budget > 0 && M > 0) {
    bool found = false;                                // sh.gt / sh.ge hold the answer
    for (int round = 0; round < max_rounds; ++round) {
      const uint32_t width = sh.width, rank = sh.rank;
      if (width <= kSelThreads * kSelItems) break;
      // this thread's samples: the last (worst) entries of blocks kSelItems * sub .. of its row's window
      int lo = 0, w = 0, s = 0;
      uint32_t key[kSelItems], wgt[kSelItems];
      if (r < R) {
        lo = sh.lo[r];
        w = sh.hi[r] - lo;
        s = (int)(((unsigned)w + (1u << sshift) - 1u) >> sshift);
      }
#pragma unroll
      for (int i = 0; i < kSelItems; ++i) {
        key[i] = 0xffffffffu;
        wgt[i] = 0u;
        const long long b0 = (long long)(kSelItems * sub + i) * s;
        if (b0 < w) {
          const int b1 = (int)min(b0 + s, (long long)w);
          wgt[i] = (uint32_t)(b1 - (int)b0);
          key[i] = score_to_key(row[lo + b1 - 1]);
        }
      }
      {
        uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
        for (int i = 0; i < kSelItems; ++i)
          if (wgt[i]) { kmin = min(kmin, key[i]); kmax = max(kmax, key[i]); }
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        const uint32_t hidden = __reduce_add_sync(0xffffffffu, sub == 0 && w > 0 ? (uint32_t)(s - 1) : 0u);   // in partial blocks
        if (lane == 0) { atomicMin(&sh.kmin, kmin); atomicMax(&sh.kmax, kmax); atomicAdd(&sh.slack, hidden); }
      }
      __syncthreads();
      // upper bracket: the first sample value whose whole blocks already hold `rank` entries: T is at least as good.
      // lower bracket: sample values for which even whole blocks plus one partial block per row hold fewer than
      // `rank` entries at least as good: T is worse than those, the ones before the first that may hold them.
      const uint32_t slack = sh.slack;
      Bracket A = {sh.kmin, rank, bits_of_range(sh.kmin, sh.kmax), true};
      Bracket B = {sh.kmin, rank > slack ? rank - slack : 0u, A.bits, rank > slack};
      const bool has_lo = B.active;
      const uint32_t enough = width / 128;
      const bool other_unit = __shfl_up_sync(0xffffffffu, s, 1) != s;
      // (at most three levels each: 11 + 11 + 10 bits)
      for (int level = 0; level < 6 && (A.active || B.active); ++level) {
        // together as long as they are at the same place, then the upper one first
        const bool one = A.active, two = !A.active || (B.active && A.base == B.base && A.bits == B.bits);
        Bracket X = one ? A : B, Y = B;
        X.active = one;
        Y.active = two;
        select_level(sh, key, wgt, (uint32_t)s, other_unit, X, Y, enough);
        if (one) A = X;
        if (two) B = Y;
      }
      const uint32_t reach = A.bits >= 32 ? 0xffffffffu : (1u << A.bits) - 1u;
      const uint32_t khi = A.base > 0xffffffffu - reach ? 0xffffffffu : A.base + reach;   // T <= khi
      const uint32_t klo = B.base;                     // T is worse than the sample values before klo
      // samples of the row on the good side of either bracket
      uint32_t good = 0u;                              // two counts in one word
#pragma unroll
      for (int i = 0; i < kSelItems; ++i)
        if (wgt[i]) good += (key[i] <= khi ? 0x10000u : 0u) + (has_lo && key[i] < klo ? 1u : 0u);
      for (int o = tpr >> 1; o > 0; o >>= 1) good += __shfl_xor_sync(0xffffffffu, good, o);
      uint32_t took = 0u, left = 0u;
      if (r < R && sub == 0 && w > 0) {
        const long long jlo = good & 0xffffu, jhi = good >> 16;
        const int nlo = lo + (int)min((long long)s * jlo, (long long)w);
        const int nhi = lo + (int)min((long long)s * (jhi + 1), (long long)w);
        sh.lo[r] = nlo;
        sh.hi[r] = nhi;
        took = (uint32_t)(nlo - lo);                   // entries now known to be better than T
        left = (uint32_t)(nhi - nlo);
      }
      took = __reduce_add_sync(0xffffffffu, took);
      left = __reduce_add_sync(0xffffffffu, left);
      if (lane == 0) { atomicAdd(&sh.taken, took); atomicAdd(&sh.new_width, left); }
      __syncthreads();
      const uint32_t new_width = sh.new_width, new_rank = rank - sh.taken;
      __syncthreads();
      if (tid == 0) {
        sh.width = new_width;
        sh.rank = new_rank;
        sh.kmin = 0xffffffffu;
        sh.kmax = 0u;
        sh.slack = sh.taken = sh.new_width = 0u;
      }
      __syncthreads();
      if (new_width > width / 2) {
        // the windows did not shrink: some value has very many copies.  Locate the upper bracket exactly.
        locate_in_windows(composite, sh, R, khi);
        const uint32_t lt = (uint32_t)sh.tot_lt, le = (uint32_t)sh.tot_le;
        __syncthreads();
        if (new_rank > lt && new_rank <= le && A.bits == 0) { found = true; break; }   // it is T
        if (new_rank <= lt) {                                         // T is better: the copies leave the windows
          if (tid < R) sh.hi[tid] = sh.gt[tid];
          if (tid == 0) sh.width = lt;
        } else if (new_rank > le) {                                   // T is worse
          if (tid < R) sh.lo[tid] = sh.ge[tid];
          if (tid == 0) { sh.rank = new_rank - le; sh.width = new_width - le; }
        } else {                                                      // T is not worse
          if (tid < R) sh.hi[tid] = sh.ge[tid];
          if (tid == 0) sh.width = le;
        }
        __syncthreads();
      }
    }
    if (!found) {
      __syncthreads();
      const uint32_t width = sh.width, rank = sh.rank;
      if (width <= kSelThreads * kSelItems) {
        // few enough entries left: all of them are looked at, T is the rank-th
        const uint32_t end = block_scan(tid < R ? (uint32_t)(sh.hi[tid] - sh.lo[tid]) : 0u, sh);
        if (tid < R) { sh.off[tid + 1] = (int)end; sh.clt[tid] = 0; sh.cle[tid] = 0; }
        if (tid == 0) sh.off[0] = 0;
        __syncthreads();
        uint32_t key[kSelItems], wgt[kSelItems];
        int at[kSelItems];
        uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
        for (int i = 0; i < kSelItems; ++i) {
          const int e = i * kSelThreads + tid;
          key[i] = 0xffffffffu;
          wgt[i] = 0u;
          at[i] = 0;
          if (e < (int)width) {
            int x = 0, y = R - 1;                      // the row with off[row] <= e < off[row + 1]
            while (x < y) {
              const int m = (x + y) >> 1;
              if (sh.off[m + 1] > e) y = m; else x = m + 1;
            }
            at[i] = x;
            wgt[i] = 1u;
            // (32-bit, and none for whole layers: 64-bit divisions cost 32 rows of 1000 0.5 us.  The starts out of shared memory are
            // faster for few rows, one of 1000 5.0 us and 5.3, but cost ties and long rows up to 0.8: 16 rows of 3001 with ties 13.6 and
            // 12.8, 28 of 131072 13.5 and 13.2.)
            const int xl = kFew || hpr == 1 ? x : x / hpr;
            const long long from = kFew ? sh.base[x] : (((long long)xl * Bt + b) * hpr + (x - xl * hpr)) * N + floor;
            key[i] = score_to_key(composite[from + sh.lo[x] + (e - sh.off[x])]);
          }
        }
#pragma unroll
        for (int i = 0; i < kSelItems; ++i)
          if (wgt[i]) { kmin = min(kmin, key[i]); kmax = max(kmax, key[i]); }
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        if (lane == 0) { atomicMin(&sh.kmin, kmin); atomicMax(&sh.kmax, kmax); }
        __syncthreads();
        Bracket A = {sh.kmin, rank, bits_of_range(sh.kmin, sh.kmax), true}, B = {0u, 0u, 0, false};
        for (int level = 0; level < 3 && A.active; ++level) select_level(sh, key, wgt, 1u, false, A, B, 0u);
        const uint32_t T = A.base;
#pragma unroll
        for (int i = 0; i < kSelItems; ++i) {
          const bool lt = wgt[i] && key[i] < T, le = wgt[i] && key[i] <= T;
          const int x0 = __shfl_sync(0xffffffffu, at[i], 0);
          const uint32_t mlt = __ballot_sync(0xffffffffu, lt), mle = __ballot_sync(0xffffffffu, le);
          if (__all_sync(0xffffffffu, at[i] == x0 || !wgt[i])) {        // the whole warp in one row
            if (lane == 0 && mle) { atomicAdd(&sh.clt[x0], __popc(mlt)); atomicAdd(&sh.cle[x0], __popc(mle)); }
          } else {
            if (lt) atomicAdd(&sh.clt[at[i]], 1);
            if (le) atomicAdd(&sh.cle[at[i]], 1);
          }
        }
        __syncthreads();
        if (tid < R) { sh.gt[tid] = sh.lo[tid] + sh.clt[tid]; sh.ge[tid] = sh.lo[tid] + sh.cle[tid]; }
      } else {
        // out of rounds: bisection over the keys, exact counts inside the windows
        uint32_t x = 0u, y = 0xffffffffu;              // T lies in [x, y]
        for (int it = 0; it < 32 && x < y; ++it) {
          const uint32_t mid = x + (y - x) / 2;
          locate_in_windows(composite, sh, R, mid);
          const uint32_t le = (uint32_t)sh.tot_le;
          __syncthreads();
          if (le >= rank) y = mid; else x = mid + 1;
        }
        locate_in_windows(composite, sh, R, x);
      }
    }
  }
  __syncthreads();
  if (tid >= 32) return;
  // the entries equal to T go to the rows in row order until the budget is met; a lane has `per` neighbouring rows
  const int per = (R + 31) / 32, first = tid * per;
  uint32_t gsum = 0, tsum = 0;                             // (below 2^32 over all rows)
  for (int i = 0; i < per; ++i) {
    if (first + i < R) { gsum += (uint32_t)sh.gt[first + i]; tsum += (uint32_t)(sh.ge[first + i] - sh.gt[first + i]); }
  }
  uint32_t gt_incl = gsum, ties_incl = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t g = __shfl_up_sync(0xffffffffu, gt_incl, o), t = __shfl_up_sync(0xffffffffu, ties_incl, o);
    if (tid >= o) { gt_incl += g; ties_incl += t; }
  }
  const long long used = __shfl_sync(0xffffffffu, gt_incl, 31), ties_before = ties_incl - tsum;
  long long rem = budget - used - ties_before;             // what is left when this lane's rows are served
  // (what the rows before this lane's took of the ties follows from the same numbers)
  const long long ties_taken = min(max(budget - used, 0LL), ties_before);
  long long off = (long long)(gt_incl - gsum) + ties_taken + floor * min(first, R);
  for (int i = 0; i < per; ++i) {
    const int rr = first + i;
    if (rr < R) {
      const long long tie = sh.ge[rr] - sh.gt[rr];
      const long long n = floor + sh.gt[rr] + max(0LL, min(tie, rem));
      rem -= tie;
      n_keep[(long long)b * R + rr] = (int32_t)n;
      offsets[(long long)b * (R + 1) + rr] = off;
      off += n;
      if (rr == R - 1) offsets[(long long)b * (R + 1) + R] = off;
    }
  }
}

// Test hooks (see kvc_debug_select_hooks).
std::atomic<int> g_select_path{0};
std::atomic<int> g_select_rounds{-1};

}  // namespace

size_t allocate_workspace_bytes(const Problem& P) {
  return align_up((size_t)P.Bt * 4 * kRadix * sizeof(unsigned int));
}

void set_select_hooks(int path, int max_rounds) {
  g_select_path.store(path);
  g_select_rounds.store(max_rounds);
}

kvc_status launch_allocate(const Problem& P, const float* composite, long long budget, int heads_per_row,
                           long long min_keep, int32_t* n_keep, long long* offsets, void* ws,
                           size_t ws_bytes, cudaStream_t st, SelectPath path) {
  if (ws_bytes < allocate_workspace_bytes(P)) {
    set_error("allocate: workspace too small");
    return KVC_ERR_WORKSPACE;
  }
  const int R = P.L * heads_per_row;
  if (R > kMaxSelectRows) {
    set_error("allocate: %d rows in the pool, at most %d supported", R, kMaxSelectRows);
    return KVC_ERR_UNSUPPORTED;
  }
  if (min_keep < 0 || min_keep > P.N || (long long)R * min_keep > budget) {
    set_error("allocate: per-layer minimum %lld does not fit (N = %lld, rows * minimum <= budget = %lld required)",
              min_keep, P.N, budget);
    return KVC_ERR_INVALID_ARG;
  }
  const long long rest = budget - (long long)R * min_keep;     // handed out beyond the minimum
  if (path == SelectPath::kAuto) {
    const int hook = g_select_path.load();
    if (hook == 1) path = SelectPath::kHistograms;
    if (hook == 2) path = SelectPath::kSortedRows;
  }
  // (with fewer than 8 samples per row a round would hardly cut the windows; the kernel counts in 32 bits)
  if (path != SelectPath::kHistograms && R <= kSelMaxRows && (long long)R * (P.N - min_keep) < (1LL << 32)) {
    const int hook_rounds = g_select_rounds.load();
    const int rounds = hook_rounds >= 0 ? hook_rounds : kSelDefaultRounds;
    KVC_CUDA(launch_dependent(R <= kSelFewRows ? select_sorted_kernel<true> : select_sorted_kernel<false>, dim3(P.Bt), dim3(kSelThreads), 0, st, composite, R, P.Bt,
                              heads_per_row, P.N, min_keep, rest, rounds, n_keep, offsets));
    KVC_LAUNCH_CHECK("select_sorted_kernel");
    return KVC_OK;
  }
  unsigned int* hist = reinterpret_cast<unsigned int*>(ws);
  KVC_CUDA(launch_dependent(select_clear_kernel, dim3(P.Bt), dim3(4 * kRadix), 0, st, hist));
  KVC_LAUNCH_CHECK("select_clear_kernel");
  const long long total = (long long)R * (P.N - min_keep);
  const long long tile = (long long)kHistThreads * kItemsPerThread;
  long long blocks = (total + tile - 1) / tile;
  int dev = 0, sms = 0;
  KVC_CUDA(cudaGetDevice(&dev));
  KVC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (blocks > 4LL * sms) blocks = 4LL * sms;
  if (blocks < 1) blocks = 1;
  if (rest > 0) {
    for (int pass = 0; pass < 4; ++pass) {
      KVC_CUDA(launch_dependent(select_hist_kernel, dim3((unsigned)blocks, P.Bt), dim3(kHistThreads), 0, st,
                                composite, hist, pass, R, P.Bt, heads_per_row, P.N, min_keep, rest));
      KVC_LAUNCH_CHECK("select_hist_kernel");
    }
  }
  KVC_CUDA(launch_dependent(select_finish_kernel, dim3(P.Bt), dim3(1024), (size_t)R * 2 * sizeof(long long), st,
                            composite, hist, R, P.Bt, heads_per_row, P.N, min_keep, rest, n_keep, offsets));
  KVC_LAUNCH_CHECK("select_finish_kernel");
  return KVC_OK;
}

}  // namespace kvc

// Test hook: which way the allocation finds its threshold (0: the library chooses, 1: the histogram
// passes, 2: the sorted-rows kernel wherever the pool has few enough rows) and how many rounds the
// sorted-rows kernel may take before it bisects (< 0: the default; 0: bisect at once).  Process-wide;
// takes effect at the next call.  kvc_allocate_static always takes the histogram passes.
extern "C" __attribute__((visibility("default"))) void kvc_debug_select_hooks(int32_t path, int32_t max_rounds) {
  kvc::set_select_hooks(path, max_rounds);
}
