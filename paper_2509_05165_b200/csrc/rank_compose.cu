// Per-head ranking (Eq. 17), sorted scores (Eq. 18) and composite scores (Eq. 19).
//
// Every (layer, sequence, KV head) is one segment of N (score, position) pairs that must come
// out in descending score order with equal scores in ascending position.  Scores are mapped to
// 32-bit keys whose ascending order is the wanted order.  A segment of up to 32768 elements is
// sorted by one CTA inside its SM's shared memory (a stable least-significant-digit radix sort
// with 4-bit digits, thread-private counters, the permutation updated in place): one launch.  A
// longer segment is cut into such chunks, which are then merged pairwise (merge path), one launch
// per level.
//
// The positions go straight into idx and the sorted keys are left for the composite kernel, which turns them back into scores and reduces over the heads.
#include "kvc_internal.cuh"

#include <mutex>
#include <type_traits>

namespace kvc {
namespace {

// ---------------------------------------------------------------------------------------------
// Segments of at most kSegMaxN elements: one CTA sorts one whole segment inside its SM.
//
// A stable least-significant-digit sort with 4-bit digits.  The keys are read from global memory
// once and stay in shared memory, by position; what moves between the passes is a permutation of
// 16-bit positions, in place.  Thread t owns the places [t * ipt, (t + 1) * ipt) of the current
// order.  A pass:
//   count    every thread walks its places in order: position -> byte of the key -> digit, and a
//            counter of its own per digit (shared memory, one bank per lane): the value it finds
//            is the element's rank among the thread's elements of that digit.  No work crosses
//            lanes, so nothing depends on how the digits are distributed.
//   scan     exclusive prefix over (digit, thread), digits ascending: the first place of every
//            thread's elements of every digit.
//   scatter  position -> place = first place + rank.  Every thread read all of its places
//            before the scan, so the permutation is overwritten in place.
// (thread, place inside the thread) is the order itself, so every pass is stable, and with the
// identity as the first order equal keys stay in ascending position.  The keys are taken relative to the
// segment's smallest, and a digit that none of them has a bit in orders nothing: its pass is left
// out (scores within a factor of 32 differ in 7 of the 8 digits, scores within 2 % in 5: 256 segments of
// 32768 of nearly uniform attention 109 -> 98 us; where no digit falls away the extra step costs
// 1 us).  After the last pass positions and keys go out through the permutation, coalesced.
// Global traffic: scores read once, idx and sorted keys written once; one launch.
constexpr int kSegMaxN = 32768;
constexpr int kSegBatch = 4;                   // key lookups in flight per thread
constexpr int kMaxDevices = 64;

__device__ __forceinline__ uint32_t lds_u8(uint32_t a) { uint32_t v; asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) { uint32_t v; asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) { uint32_t v; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v) { asm volatile("st.shared.u16 [%0], %1;" :: "r"(a), "h"((unsigned short)v) : "memory"); }
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts_v4(uint32_t a, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" :: "r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Shared-memory map of a segment of N elements sorted by T threads (byte offsets).
struct SegLayout {
  int n_pad;            // N rounded up to 32: key_slot and place_slot permute inside aligned blocks of 32
  uint32_t keys;        // uint32[n_pad]: the keys, by position
  uint32_t perm;        // uint16[n_pad]: the key slot (key_slot of the position) at every place
  uint32_t cnt;         // uint16[8][T][2]: thread t's counter of digit d in row d & 7, half d >> 3
  uint32_t wtot;        // uint32[64]: the scan's warp totals; before, the warps' smallest keys and the bits set in theirs
  uint32_t total;
};
__host__ __device__ inline SegLayout seg_layout(long long N, int T) {
  SegLayout s;
  s.n_pad = (int)((N + 31) / 32 * 32);
  s.keys = 0;
  s.perm = 4u * s.n_pad;
  s.cnt = s.perm + 2u * s.n_pad;
  s.wtot = s.cnt + 8u * T * 4u;
  s.total = s.wtot + 256u;
  return s;
}

// Where things sit, to keep the banks apart.  Key of position i: word i ^ ((i >> 5) & 31): the
// threads of a warp start 32 places apart, which in the first pass are 32 positions apart.
// Place j: halfword j ^ (((j >> 6) & 3) << 3): a warp reads 32 stretches of 64 bytes, 16 at a time.
__device__ __forceinline__ uint32_t key_slot(uint32_t i) { return i ^ ((i >> 5) & 31u); }
__device__ __forceinline__ uint32_t place_slot(uint32_t j) { return j ^ (((j >> 6) & 3u) << 3); }

// score_to_key without the branch.
__device__ __forceinline__ uint32_t seg_key(float f) {
  uint32_t b = __float_as_uint(f);
  b = (b == 0x80000000u) ? 0u : b;
  const uint32_t m = (uint32_t)((int32_t)b >> 31) | 0x80000000u;
  return ~(b ^ m);
}

// The thread's keys of the segment, in groups of 4 neighbours: group g holds positions (g * T + tid) * 4 ..  All loads are
// issued before the first use; 16 bytes at a time where the scores are aligned.  Positions behind the end get key 0.
template <int T, int kIpt>
__device__ __forceinline__ void seg_load_keys(const float* s_in, int N, int tid, uint32_t (&k)[kIpt]) {
  constexpr int kGroups = kIpt / 4;
  const bool wide = (reinterpret_cast<uintptr_t>(s_in) & 15u) == 0;
  float v[kIpt];
#pragma unroll
  for (int g = 0; g < kGroups; ++g) {
    const int i = (g * T + tid) * 4;
    if (wide && i + 4 <= N) {
      const float4 w = *reinterpret_cast<const float4*>(s_in + i);
      v[4 * g] = w.x; v[4 * g + 1] = w.y; v[4 * g + 2] = w.z; v[4 * g + 3] = w.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[4 * g + e] = s_in[min(i + e, N - 1)];
    }
  }
#pragma unroll
  for (int j = 0; j < kIpt; ++j) k[j] = (((j >> 2) * T + tid) * 4 + (j & 3)) < N ? seg_key(v[j]) : 0u;
}

// N elements, from `first` on in all three arrays; their positions count from pos0.
template <int T, int kIpt>
__device__ __forceinline__ void segment_sort(const float* __restrict__ scores, uint32_t* __restrict__ keys_out,
                                             int32_t* __restrict__ idx_out, long long first, int N, int pos0) {
  constexpr int kRowShift = T == 1024 ? 12 : T == 512 ? 11 : T == 256 ? 10 : 9;   // log2 of a row of counters in bytes
  static_assert((4 * T) >> kRowShift == 1 && kIpt % 8 == 0 && kIpt <= 32, "rows of counters, groups of places");
  constexpr int kScanWarps = T / 64;                        // the scan runs on the first T / 2 threads
  extern __shared__ __align__(16) unsigned char seg_smem[];
  const SegLayout lay = seg_layout(N, T);
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(seg_smem);
  const uint32_t keys = sbase + lay.keys, perm = sbase + lay.perm, cnt = sbase + lay.cnt, wtot = sbase + lay.wtot;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int j0 = tid * kIpt;
  const int nv = max(0, min(kIpt, N - j0));                  // my places: j0 .. j0 + nv - 1
  const bool full = __all_sync(0xffffffffu, nv == kIpt);     // the warp's decision
  // My counter of digit d: + ((d & 7) << kRowShift) + ((d >> 3) << 1).  Inside a warp's 32 columns, groups
  // of 4 are permuted by the warp number so that the scan's 16-byte reads of neighbouring columns spread
  // over the banks; a lane keeps a bank of its own.
  const uint32_t cbase = cnt + (uint32_t)(tid ^ (((tid >> 5) & 3) << 2)) * 4u;

  grid_dependency_wait();
  const float* s_in = scores + first;

  // ---- the keys, once, relative to the smallest of the segment: scores that lie close together then share their upper
  //      digits, on whichever side of a power of two they lie.  The identity as the first order; which bits are set anywhere
  uint32_t diff = 0, kmin = 0xffffffffu;
  {
    uint32_t k[kIpt];
    seg_load_keys<T, kIpt>(s_in, N, tid, k);
#pragma unroll
    for (int j = 0; j < kIpt; ++j) if ((((j >> 2) * T + tid) * 4 + (j & 3)) < N) kmin = min(kmin, k[j]);
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    if (lane == 0) sts_u32(wtot + warp * 4, kmin);
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < T / 32 ? lds_u32(wtot + lane * 4) : 0xffffffffu);
#pragma unroll
    for (int g = 0; g < kIpt / 4; ++g) {
      const int i = (g * T + tid) * 4;
      if (i < N) {
        const uint32_t sw = ((uint32_t)i >> 5) & 31u;        // the four stay inside their 16 bytes; the table is padded
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t rel = k[4 * g + e] - kmin;
          sts_u32(keys + (((uint32_t)(i + e)) ^ sw) * 4u, rel);
          if (i + e < N) diff |= rel;
        }
      }
    }
    // (the permutation holds key slots, not positions: a lookup needs no translation)
#pragma unroll
    for (int q = 0; q < kIpt / 8; ++q) {
      if (q * 8 < nv) {
        const uint32_t j = (uint32_t)(j0 + q * 8);
        // j is a multiple of 8: the eight slots are (j ^ m's high bits) | (e ^ m's low 3 bits), e = 0..7
        const uint32_t m = (j >> 5) & 31u;
        const uint32_t bb = (j ^ (m & 24u)) * 0x10001u, mm = (m & 7u) * 0x10001u;
        sts_v4(perm + place_slot(j) * 2u, make_uint4(bb | (0x10000u ^ mm), bb | (0x30002u ^ mm),
                                                       bb | (0x50004u ^ mm), bb | (0x70006u ^ mm)));
      }
    }
    diff = __reduce_or_sync(0xffffffffu, diff);
    if (lane == 0) sts_u32(wtot + 128 + warp * 4, diff);
    __syncthreads();
    diff = __reduce_or_sync(0xffffffffu, lane < T / 32 ? lds_u32(wtot + 128 + lane * 4) : 0u);
  }

#pragma unroll 1
  for (int B = 0; B < 4; ++B) {
    const uint32_t kb = keys + (uint32_t)B;                  // byte B of the key in slot s: kb + 4 s
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (((diff >> (8 * B + 4 * h)) & 15u) == 0) continue;  // a digit every key shares orders nothing
      // with an element as  key slot | byte << 16 | rank << 24,  its digit d sits at bit 16 + 4 h
      constexpr uint32_t kRowMask = 7u << kRowShift;
      const int sh_row = 16 + 4 * h - kRowShift, sh_half = 18 + 4 * h;

      // ---- count (warps whose places all exist take the copy without the per-place tests)
#pragma unroll
      for (int d = 0; d < 8; ++d) sts_u32(cbase + ((uint32_t)d << kRowShift), 0u);
      uint32_t packed[kIpt];
      auto count = [&](auto full_tag) {
        constexpr bool kFull = decltype(full_tag)::value;
#pragma unroll
        for (int q = 0; q < kIpt / 8; ++q) {
          if (kFull || q * 8 < nv) {
            const uint4 w = lds_v4(perm + place_slot((uint32_t)(j0 + q * 8)) * 2u);
            packed[q * 8 + 0] = w.x & 0xffffu; packed[q * 8 + 1] = w.x >> 16;
            packed[q * 8 + 2] = w.y & 0xffffu; packed[q * 8 + 3] = w.y >> 16;
            packed[q * 8 + 4] = w.z & 0xffffu; packed[q * 8 + 5] = w.z >> 16;
            packed[q * 8 + 6] = w.w & 0xffffu; packed[q * 8 + 7] = w.w >> 16;
          }
        }
#pragma unroll
        for (int k0 = 0; k0 < kIpt; k0 += kSegBatch) {
          uint32_t b[kSegBatch];
#pragma unroll
          for (int k = 0; k < kSegBatch; ++k) if (kFull || k0 + k < nv) b[k] = lds_u8(kb + packed[k0 + k] * 4u);
#pragma unroll
          for (int k = 0; k < kSegBatch; ++k) {
            if (kFull || k0 + k < nv) {
              const uint32_t pk = packed[k0 + k] | (b[k] << 16);
              const uint32_t a = cbase + (((pk >> sh_row) & kRowMask) | ((pk >> sh_half) & 2u));
              const uint32_t seen = lds_u16(a);
              sts_u16(a, seen + 1u);
              packed[k0 + k] = pk + (seen << 24);
            }
          }
        }
      };
      if (full) count(std::true_type{}); else count(std::false_type{});
      __syncthreads();

      // ---- scan.  Thread s < T / 2 owns 16 neighbouring threads' counters of the digits in its row: the low
      //      halves (digit = row) precede all high halves (digit = row + 8) in the order of the places.
      {
        const uint32_t mine = cnt + (uint32_t)tid * 64u;
        const uint32_t rot = (((uint32_t)tid >> 1) & 3u) << 4;                     // the permutation of cbase, seen from here
        uint32_t lo_sum = 0, hi_sum = 0, lo_incl = 0, hi_incl = 0;
        if (tid < T / 2) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 w = lds_v4(mine + ((q * 16) ^ rot));
            lo_sum += (w.x & 0xffffu) + (w.y & 0xffffu) + (w.z & 0xffffu) + (w.w & 0xffffu);
            hi_sum += (w.x >> 16) + (w.y >> 16) + (w.z >> 16) + (w.w >> 16);
          }
          lo_incl = lo_sum; hi_incl = hi_sum;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, lo_incl, o);
            const uint32_t y = __shfl_up_sync(0xffffffffu, hi_incl, o);
            if (lane >= o) { lo_incl += x; hi_incl += y; }
          }
          if (lane == 31) { sts_u32(wtot + warp * 4, lo_incl); sts_u32(wtot + (kScanWarps + warp) * 4, hi_incl); }
        }
        __syncthreads();
        if (tid < T / 2) {
          const uint32_t x = lane < 2 * kScanWarps ? lds_u32(wtot + lane * 4) : 0u;
          uint32_t e = x;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, e, o);
            if (lane >= o) e += y;
          }
          e -= x;                                                                  // exclusive over the warp totals
          uint32_t lo = __shfl_sync(0xffffffffu, e, warp) + lo_incl - lo_sum;
          uint32_t hi = __shfl_sync(0xffffffffu, e, kScanWarps + warp) + hi_incl - hi_sum;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t a = mine + ((q * 16) ^ rot);
            const uint4 w = lds_v4(a);
            uint4 o4;
            o4.x = lo | (hi << 16); lo += w.x & 0xffffu; hi += w.x >> 16;
            o4.y = lo | (hi << 16); lo += w.y & 0xffffu; hi += w.y >> 16;
            o4.z = lo | (hi << 16); lo += w.z & 0xffffu; hi += w.z >> 16;
            o4.w = lo | (hi << 16); lo += w.w & 0xffffu; hi += w.w >> 16;
            sts_v4(a, o4);
          }
        }
      }
      __syncthreads();

      // ---- scatter (in place: every place was read before the scan)
      auto scatter = [&](auto full_tag) {
        constexpr bool kFull = decltype(full_tag)::value;
#pragma unroll
        for (int k = 0; k < kIpt; ++k) {
          if (kFull || k < nv) {
            const uint32_t pk = packed[k];
            const uint32_t off = lds_u16(cbase + (((pk >> sh_row) & kRowMask) | ((pk >> sh_half) & 2u)));
            sts_u16(perm + place_slot(off + (pk >> 24)) * 2u, pk);
          }
        }
      };
      if (full) scatter(std::true_type{}); else scatter(std::false_type{});
      __syncthreads();
    }
  }

  // ---- out: the positions (a slot's position is key_slot of it: the map is its own inverse), and the keys
  uint32_t* k_out = keys_out + first;
  int32_t* i_out = idx_out + first;
  for (int j = tid; j < N; j += T) {
    const uint32_t q = lds_u16(perm + place_slot((uint32_t)j) * 2u);
    i_out[j] = pos0 + (int32_t)key_slot(q);
    k_out[j] = lds_u32(keys + q * 4u) + kmin;
  }
}

// CTA x sorts chunk x % chunks of segment x / chunks: the positions from chunk * chunk_len on (the chunks of a
// segment of several are merged afterwards).  kShort: the last chunk of a segment is at most half as long as kIpt places
// per thread are made for; with them a few warps would do all of its work (the ranking of 80 segments of 40000: 125 -> 101 us,
// of 32772: 106 -> 93).
template <int T, int kIpt, bool kShort = false>
__global__ void __launch_bounds__(T, 1024 / T)
segment_sort_kernel(const float* __restrict__ scores, uint32_t* __restrict__ keys_out,
                    int32_t* __restrict__ idx_out, long long seg_len, int chunks, int chunk_len) {
  const long long seg = blockIdx.x / (unsigned)chunks;
  const int chunk = (int)(blockIdx.x - seg * chunks), pos0 = chunk * chunk_len;
  const long long first = seg * seg_len + pos0;
  const int N = (int)min((long long)chunk_len, seg_len - pos0);
  if (kShort && N <= T * 8) segment_sort<T, 8>(scores, keys_out, idx_out, first, N, pos0);
  else if (kShort && N <= T * 16) segment_sort<T, 16>(scores, keys_out, idx_out, first, N, pos0);
  else segment_sort<T, kIpt>(scores, keys_out, idx_out, first, N, pos0);
}

// ---------------------------------------------------------------------------------------------
// Segments of several chunks (see chunking): the chunks come sorted from segment_sort_kernel and are merged
// pairwise, level by level (runs of the chunks' length << level).  A CTA produces kMergeTile
// consecutive outputs of one pair of runs A, B: it finds where the tile's first and last output
// split between A and B (the merge path: a binary search over one diagonal each), brings the two
// stretches into shared memory, and every thread merges kMergeItems consecutive outputs from its
// own diagonal.  Equal keys are taken from A first: A holds the smaller positions and both runs
// are stable, so the merged run is in (key, position) order as well.
constexpr int kMergeThreads = 512;
constexpr int kMergeItems = 8;
constexpr int kMergeTile = kMergeThreads * kMergeItems;       // 4096; divides kSegMaxN

// Number of elements taken from A among the first `diag` outputs of merging A (na) and B (nb).
__device__ __forceinline__ int merge_path(int diag, int na, int nb, const uint32_t* a, const uint32_t* b) {
  int lo = max(0, diag - nb), hi = min(diag, na);
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    // A[mid] is among the first diag outputs iff it does not come after B[diag - 1 - mid]
    if (a[mid] <= b[diag - 1 - mid]) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The same by one warp over global memory, 32 probes per round (a round trip per round, not per probe).
__device__ __forceinline__ int merge_path_warp(int diag, int na, int nb, const uint32_t* __restrict__ a,
                                               const uint32_t* __restrict__ b) {
  const int lane = threadIdx.x & 31;
  int lo = max(0, diag - nb), hi = min(diag, na);          // the answer lies in [lo, hi]
  while (hi > lo) {
    const int step = (hi - lo + 31) / 32;
    const int i = lo + (lane + 1) * step - 1;              // this lane's probe
    bool before = false;                                   // "A[i] is among the first diag outputs": true for a prefix of the probes
    if (i < hi) before = a[i] <= b[diag - 1 - i];
    const int n_before = __popc(__ballot_sync(0xffffffffu, before));
    const int new_lo = n_before == 0 ? lo : min(hi, lo + n_before * step);
    const int new_hi = n_before == 32 ? hi : min(hi, lo + (n_before + 1) * step - 1);
    lo = new_lo;
    hi = new_hi;
  }
  return lo;
}

// Bound by the latencies of a tile (split search, loads, merge) at four CTAs per SM; a thread reads one key per output, the
// successor of the one it took.  (Both runs' heads at every step and outputs written to shared memory at a stride of 8:
// the ranking of 28 segments of 131072, two levels, 118 -> 101 us; with 256 threads of 16 outputs 110, with 1024 of 4 109.
// Left to itself the compiler takes 40 registers where kVec is false, and three CTAs fit: 112 segments of 131071 492 us, 458 so.)
// kVec: rows start on 16 bytes (N a multiple of 4, both output arrays aligned): a thread stores its outputs itself, 16 bytes at a time.  Otherwise
// they go through shared memory once more; a tile's element i sits in slot i + i / kMergeItems there, so that the threads'
// stretches begin in different banks.
template <bool kVec>
__global__ void __launch_bounds__(kMergeThreads, 4)
merge_runs_kernel(const uint32_t* __restrict__ keys_in, const int32_t* __restrict__ vals_in,
                  uint32_t* __restrict__ keys_out, int32_t* __restrict__ vals_out, long long seg_len, long long run,
                  int tiles_per_seg) {
  __shared__ uint32_t s_key[kMergeTile + kMergeThreads];
  __shared__ int32_t s_val[kMergeTile + kMergeThreads];
  __shared__ int s_split[2];
  grid_dependency_wait();
  const long long seg = blockIdx.x / (unsigned)tiles_per_seg;
  const long long t0 = (long long)(blockIdx.x - seg * tiles_per_seg) * kMergeTile;    // first output, inside the segment
  const long long pair0 = t0 / (2 * run) * (2 * run);                                  // where this tile's pair of runs starts
  const int na = (int)min(run, seg_len - pair0);
  const int nb = (int)max(0LL, min(run, seg_len - pair0 - run));
  const long long base = seg * seg_len + pair0;
  const uint32_t* ka = keys_in + base;
  const uint32_t* kb = ka + na;
  const int d0 = (int)(t0 - pair0);
  const int d1 = min(d0 + kMergeTile, na + nb);
  const int tid = threadIdx.x;
  if (tid < 64) {                                          // warp 0: the tile's first output; warp 1: one past its last
    const int split = merge_path_warp(tid < 32 ? d0 : d1, na, nb, ka, kb);
    if ((tid & 31) == 0) s_split[tid >> 5] = split;
  }
  __syncthreads();
  const int a0 = s_split[0], a1 = s_split[1];
  const int b0 = d0 - a0, b1 = d1 - a1;
  const int ca = a1 - a0, cb = b1 - b0;                   // this tile's elements of A, then of B, in shared memory
#pragma unroll
  for (int k = 0; k < kMergeItems; ++k) {
    const int i = tid + k * kMergeThreads;
    if (i < ca + cb) {
      const long long src = base + (i < ca ? (long long)a0 + i : (long long)na + b0 + (i - ca));
      s_key[i] = __ldg(keys_in + src);
      s_val[i] = __ldg(vals_in + src);
    }
  }
  __syncthreads();
  const int n_out = d1 - d0;
  const int my0 = min(tid * kMergeItems, n_out);
  int ia = merge_path(my0, ca, cb, s_key, s_key + ca);
  int ib = ca + my0 - ia;                                  // (slot of B's next element)
  const int end_b = ca + cb;
  uint32_t ok[kMergeItems]; int32_t ov[kMergeItems];
  uint32_t xa = ia < ca ? s_key[ia] : 0xffffffffu, xb = ib < end_b ? s_key[ib] : 0xffffffffu;
#pragma unroll
  for (int k = 0; k < kMergeItems; ++k) {
    const bool take_a = ia < ca && (ib >= end_b || xa <= xb);
    ok[k] = take_a ? xa : xb;
    const int at = take_a ? ia : ib;                       // the next element of the run it came from
    ov[k] = at < end_b ? s_val[at] : 0;
    const int nx = at + 1, lim = take_a ? ca : end_b;
    const uint32_t x = nx < lim ? s_key[nx] : 0xffffffffu;
    if (take_a) { ia = nx; xa = x; } else { ib = nx; xb = x; }
  }
  const long long dst = base + d0;
  if (kVec) {
    if (my0 + kMergeItems <= n_out) {
#pragma unroll
      for (int k = 0; k < kMergeItems; k += 4) {
        *reinterpret_cast<uint4*>(keys_out + dst + my0 + k) = make_uint4(ok[k], ok[k + 1], ok[k + 2], ok[k + 3]);
        *reinterpret_cast<int4*>(vals_out + dst + my0 + k) = make_int4(ov[k], ov[k + 1], ov[k + 2], ov[k + 3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < kMergeItems; ++k)
        if (my0 + k < n_out) { keys_out[dst + my0 + k] = ok[k]; vals_out[dst + my0 + k] = ov[k]; }
    }
  } else {
    __syncthreads();                                       // everyone has read its inputs: the buffers take the outputs
    const int slot0 = tid * (kMergeItems + 1);
#pragma unroll
    for (int k = 0; k < kMergeItems; ++k) { s_key[slot0 + k] = ok[k]; s_val[slot0 + k] = ov[k]; }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kMergeItems; ++k) {
      const int i = tid + k * kMergeThreads, slot = i + i / kMergeItems;
      if (i < n_out) { keys_out[dst + i] = s_key[slot]; vals_out[dst + i] = s_val[slot]; }
    }
  }
}

// Eq. 19 over the sorted keys: composite[lb, k] = agg_head_h score(keys[lb, h, k]).
// Mean: heads added in ascending order in fp32, one division at the end.
// blockIdx.y = (layer, sequence), blockIdx.x over the ranks, kE neighbouring ranks per thread (4 with 16-byte accesses where N
// is a multiple of 4: 256 segments of 32768 10.3 -> 7.0 us, 112 of 131072 33 -> 15).  The heads' keys are fetched eight at
// a time before they are added, so that a thread waits for memory once, not once per head.
template <int kE>
__global__ void __launch_bounds__(256)
compose_kernel(const uint32_t* __restrict__ keys, float* __restrict__ composite, int Hkv, long long N, int agg_head) {
  grid_dependency_wait();
  constexpr int kB = 8;
  const long long kk = ((long long)blockIdx.x * 256 + threadIdx.x) * kE;
  if (kk >= N) return;
  const uint32_t* p = keys + (long long)blockIdx.y * Hkv * N + kk;
  float acc[kE];
#pragma unroll
  for (int e = 0; e < kE; ++e) acc[e] = 0.f;
  for (int h0 = 0; h0 < Hkv; h0 += kB) {
    uint32_t v[kB][kE];
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (h0 + j < Hkv) {
        if constexpr (kE == 4) {
          const uint4 w = __ldg(reinterpret_cast<const uint4*>(p + (long long)(h0 + j) * N));
          v[j][0] = w.x; v[j][1] = w.y; v[j][2] = w.z; v[j][3] = w.w;
        } else {
          v[j][0] = __ldg(p + (long long)(h0 + j) * N);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (h0 + j < Hkv) {
#pragma unroll
        for (int e = 0; e < kE; ++e) {
          const float a = key_to_score(v[j][e]);
          if (h0 + j == 0) acc[e] = a;
          else acc[e] = (agg_head == KVC_AGG_MAX) ? fmaxf(acc[e], a) : __fadd_rn(acc[e], a);
        }
      }
    }
  }
  float* out = composite + (long long)blockIdx.y * N + kk;
#pragma unroll
  for (int e = 0; e < kE; ++e) if (agg_head == KVC_AGG_MEAN) acc[e] = __fdiv_rn(acc[e], (float)Hkv);
  if constexpr (kE == 4) *reinterpret_cast<float4*>(out) = make_float4(acc[0], acc[1], acc[2], acc[3]);
  else *out = acc[0];
}

// Eq. 18 as fp32: the sorted keys turned back into scores.
__global__ void __launch_bounds__(256)
sorted_scores_kernel(const uint32_t* __restrict__ keys, float* __restrict__ sorted, long long total) {
  grid_dependency_wait();
  const long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * 4;       // (both arrays start on 256 bytes)
  if (i + 4 <= total) {
    const uint4 k = __ldg(reinterpret_cast<const uint4*>(keys + i));
    *reinterpret_cast<float4*>(sorted + i) = make_float4(key_to_score(k.x), key_to_score(k.y), key_to_score(k.z), key_to_score(k.w));
  } else {
    for (long long j = i; j < total; ++j) sorted[j] = key_to_score(keys[j]);
  }
}

}  // namespace

typedef void (*SegmentSort)(const float*, uint32_t*, int32_t*, long long, int, int);
struct SegmentPlan {
  SegmentSort kernel;
  int threads;
};
// CTA size and places per thread for a segment of N elements.  The number of places is a constant of the kernel and fits
// the segment: all but the last warp take the loops without per-place tests, and no warp idles.  Up to 4096 elements
// few places and more threads (a pass is a chain of look-ups per thread): 256 segments of 1000: 15.0 us with 128 x 8, 15.8
// with 256 x 8, 21.5 with 128 x 16 (23.4 with 256 x 4 of 32 tested places); of 4096: 20.9 with 256 x 16, 23.3 with 512 x 8, 24.3
// with 128 x 32 (31.7 tested).  Beyond, 24 or 32 places, which move the most elements per SM: 1024 segments of 5003: 92 with
// 256 x 24, 108 with 512 x 16, 113 with 256 x 32 (116 before); 256 of 8192: 33.7 with 256 x 32, 35.3 with 512 x 16; of 16384: 60 with
// 512 x 32, of which two fit an SM, 71 with 1024 x 16 (98 before).
static SegmentPlan segment_plan(long long N, bool short_last) {
  if (N <= 1024) return {segment_sort_kernel<128, 8>, 128};
  if (N <= 2048) return {segment_sort_kernel<128, 16>, 128};
  if (N <= 4096) return {segment_sort_kernel<256, 16>, 256};
  if (N <= 6144) return {segment_sort_kernel<256, 24>, 256};
  if (N <= 8192) return {segment_sort_kernel<256, 32>, 256};
  if (N <= 12288) return {segment_sort_kernel<512, 24>, 512};
  if (N <= 16384) return {segment_sort_kernel<512, 32>, 512};
  if (N <= 24576) return {segment_sort_kernel<1024, 24>, 1024};
  if (short_last) return {segment_sort_kernel<1024, 32, true>, 1024};
  return {segment_sort_kernel<1024, 32>, 1024};
}

// Can a segment (or, of several, a chunk) of N elements be sorted inside one SM here?  Sets the shared-memory attribute once
// per device (it is per device), under a lock.
static kvc_status segment_sort_prepare(long long N, bool short_last, SegmentPlan* plan) {
  if (N > kSegMaxN) return KVC_ERR_UNSUPPORTED;
  static std::mutex mu;
  static int optin[kMaxDevices];           // 0: not looked at, else the device's opt-in bytes (or -1)
  int dev = 0;
  KVC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return KVC_ERR_UNSUPPORTED;
  *plan = segment_plan(N, short_last);
  const size_t need = seg_layout(N, plan->threads).total;
  std::lock_guard<std::mutex> lock(mu);
  if (optin[dev] == 0) {
    int bytes = 0;
    KVC_CUDA(cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    for (long long n : {1024LL, 2048LL, 4096LL, 6144LL, 8192LL, 12288LL, 16384LL, 24576LL, (long long)kSegMaxN})
      for (bool s : {false, true})
        KVC_CUDA(cudaFuncSetAttribute(segment_plan(n, s).kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    optin[dev] = bytes > 0 ? bytes : -1;
  }
  if (optin[dev] < 0 || need > (size_t)optin[dev]) return KVC_ERR_UNSUPPORTED;
  return KVC_OK;
}

// How segments are cut into chunks: as few as fit an SM each, but while there are no more chunks than half of the SMs
// (a rank's share of the heads, or a few layers), twice as many, down to 8192 elements: the SMs that would idle take
// part, for one merge level more.  64 segments of 32768: 59 us as they are, 47 in halves; 8 of 131072: 77 -> 61.
// (A constant stands for the SMs: the workspace must not depend on the device.)
struct Chunking {
  long long len;
  int count;
};
static Chunking chunking(const Problem& P) {
  constexpr long long kSms = 148;
  const long long segments = (long long)P.L * P.Bt * P.Hkv;
  long long c = (P.N + kSegMaxN - 1) / kSegMaxN;
  const long long least = c;
  while (segments * c * 2 <= kSms && P.N > c * 8192) c *= 2;
  if (c == least) return {P.N < kSegMaxN ? P.N : (long long)kSegMaxN, (int)c};
  const long long len = ((P.N + c - 1) / c + kMergeTile / 2 - 1) / (kMergeTile / 2) * (kMergeTile / 2);   // pairs of runs hold whole tiles
  return {len, (int)((P.N + len - 1) / len)};
}

// Scratch of the ranking: the sorted keys [L, Bt, Hkv, N] and, for segments of several chunks, one more
// buffer of keys and one of positions for the merge levels to alternate with (keys, idx).
struct SortRegions {
  size_t keys_a, vals_a, keys_b, total;
};
static SortRegions sort_regions(const Problem& P) {
  const size_t region = align_up((size_t)P.L * P.Bt * P.Hkv * P.N * 4);
  SortRegions r;
  if (chunking(P).count == 1) { r.keys_a = r.vals_a = 0; r.keys_b = 0; r.total = region; }
  else { r.keys_a = 0; r.vals_a = region; r.keys_b = 2 * region; r.total = 3 * region; }
  return r;
}

size_t compose_workspace_bytes(const Problem& P) { return sort_regions(P).total; }

kvc_status launch_sorted_scores(const Problem& P, const void* ws, float* sorted, cudaStream_t st) {
  const size_t items = (size_t)P.L * P.Bt * P.Hkv * P.N;
  const uint32_t* keys_b = reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(ws) + sort_regions(P).keys_b);
  KVC_CUDA(launch_dependent(sorted_scores_kernel, dim3((unsigned)((items + 1023) / 1024)), dim3(256), 0, st,
                            keys_b, sorted, (long long)items));
  KVC_LAUNCH_CHECK("sorted_scores_kernel");
  return KVC_OK;
}

kvc_status launch_compose(const Problem& P, const float* scores, int32_t* idx, float* composite,
                          void* ws, size_t ws_bytes, cudaStream_t st) {
  if (ws_bytes < compose_workspace_bytes(P)) {
    set_error("compose: workspace too small");
    return KVC_ERR_WORKSPACE;
  }
  char* w = reinterpret_cast<char*>(ws);
  const SortRegions reg = sort_regions(P);
  uint32_t* const keys_a = reinterpret_cast<uint32_t*>(w + reg.keys_a);
  int32_t* const vals_a = reinterpret_cast<int32_t*>(w + reg.vals_a);
  uint32_t* const keys_b = reinterpret_cast<uint32_t*>(w + reg.keys_b);
  const long long segments = (long long)P.L * P.Bt * P.Hkv;
  SegmentPlan plan;
  const Chunking cut = chunking(P);
  const long long chunk_len = cut.len;
  // (only where it is short: the copy for both takes a percent longer on whole chunks)
  const bool short_last = P.N - (cut.count - 1) * chunk_len <= kSegMaxN / 2;
  const kvc_status seg_state = segment_sort_prepare(chunk_len, short_last, &plan);
  if (seg_state != KVC_OK && seg_state != KVC_ERR_UNSUPPORTED) return seg_state;
  if (seg_state != KVC_OK) {
    set_error("compose: this device cannot give a CTA the %zu bytes of shared memory the ranking needs",
              (size_t)seg_layout(chunk_len, segment_plan(chunk_len, short_last).threads).total);
    return KVC_ERR_UNSUPPORTED;
  }
  {
    // Chunks are sorted inside one SM each: a whole segment in one launch, or,
    // for longer segments, its chunks, which are then merged pairwise, level by level.  The levels
    // alternate between (keys_a, vals_a) and (keys_b, idx); the last one has to end in the latter.
    const long long chunks = cut.count;
    int levels = 0;
    while ((1LL << levels) < chunks) ++levels;
    const long long merge_tiles = (P.N + kMergeTile - 1) / kMergeTile;
    if (segments * chunks >= (1LL << 31) || segments * merge_tiles >= (1LL << 31)) {
      set_error("compose: too many segments");
      return KVC_ERR_UNSUPPORTED;
    }
    bool in_b = (levels % 2) == 0;                 // where the sorted chunks go
    uint32_t* k_cur = in_b ? keys_b : keys_a;
    int32_t* v_cur = in_b ? idx : vals_a;
    const size_t smem = seg_layout(chunk_len, plan.threads).total;
    const unsigned grid = (unsigned)(segments * chunks);
    KVC_CUDA(launch_dependent(plan.kernel, dim3(grid), dim3(plan.threads), smem, st, scores, k_cur, v_cur, P.N, (int)chunks,
                              (int)chunk_len));
    KVC_LAUNCH_CHECK("segment_sort_kernel");
    for (int level = 0; level < levels; ++level) {
      in_b = !in_b;
      uint32_t* k_nxt = in_b ? keys_b : keys_a;
      int32_t* v_nxt = in_b ? idx : vals_a;
      // 16-byte stores where a segment's rows start on 16 bytes; the last level's positions go to the caller's idx, which may
      // start anywhere (the buffers of the workspace start on 256 bytes)
      const bool vec = P.N % 4 == 0 && (reinterpret_cast<uintptr_t>(v_nxt) & 15u) == 0;
      KVC_CUDA(launch_dependent(vec ? merge_runs_kernel<true> : merge_runs_kernel<false>, dim3((unsigned)(segments * merge_tiles)), dim3(kMergeThreads), 0, st,
                                (const uint32_t*)k_cur, (const int32_t*)v_cur, k_nxt, v_nxt, P.N,
                                chunk_len << level, (int)merge_tiles));
      KVC_LAUNCH_CHECK("merge_runs_kernel");
      k_cur = k_nxt;
      v_cur = v_nxt;
    }
  }
  if (composite == nullptr) return KVC_OK;      // ranking only (the unstructured variant has no Eq. 19)
  const bool vec = P.N % 4 == 0 && (reinterpret_cast<uintptr_t>(composite) & 15u) == 0;
  const long long per = vec ? 1024 : 256;
  KVC_CUDA(launch_dependent(vec ? compose_kernel<4> : compose_kernel<1>,
                            dim3((unsigned)((P.N + per - 1) / per), (unsigned)(P.L * P.Bt)), dim3(256), 0, st,
                            (const uint32_t*)keys_b, composite, P.Hkv, P.N, P.agg_head));
  KVC_LAUNCH_CHECK("compose_kernel");
  return KVC_OK;
}

}  // namespace kvc
