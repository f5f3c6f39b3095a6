// Device helpers shared by the selection kernels: order-preserving keys, block scans, histogram
// search, and the generic radix selection that recomputes pooled keys from global memory.
// Not part of the public interface.
#pragma once

#include "common.cuh"

namespace spec {

constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelVec = 4;                       // consecutive positions per thread in the ordered pass of the generic path
constexpr int kSmemLimit = 227 * 1024;

// Monotone map float -> uint32 (larger float <=> larger key), valid for any sign.
__device__ __forceinline__ uint32_t to_key(float v) {
  const uint32_t b = __float_as_uint(v + 0.0f);            // -0.0 + 0.0 = +0.0: the two zeros tie, as they compare equal
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);   // negative: all bits flipped; else: sign bit set
}

// Block-wide exclusive scan of one int per thread; total returned to every thread.
// wsum: kSelWarps ints of shared memory that no thread touches again before the CTA's next
// synchronisation after this call.  One __syncthreads.
__device__ __forceinline__ int block_exclusive_scan(int v, int* wsum, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  // every warp scans the kSelWarps (<= 32) warp totals itself
  int ws = lane < kSelWarps ? wsum[lane] : 0;
  int wincl = ws;
#pragma unroll
  for (int o = 1; o < kSelWarps; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, wincl, o);
    if (lane >= o) wincl += t;
  }
  total = __shfl_sync(0xffffffffu, wincl, kSelWarps - 1);
  const int before = __shfl_sync(0xffffffffu, wincl - ws, warp);
  return before + incl - v;
}

// Finds the bin holding the need-th largest element of a histogram whose bins are spread
// over the threads, bins_per_thread consecutive bins each starting at my_bins (need >= 1).
// Returns the bin and the number of elements in higher bins to every thread; false (outputs
// untouched) when the histogram holds fewer than `need` elements.
__device__ __forceinline__ bool locate_bin(const uint32_t* my_bins, int bins_per_thread, int need, int* wsum, int* out2,
                                           int& bin, int& above) {
  const int b0 = threadIdx.x * bins_per_thread;
  __syncthreads();                                         // histogram complete, wsum free
  if (threadIdx.x == 0) out2[0] = -1;
  int mine = 0;
  for (int i = 0; i < bins_per_thread; ++i) mine += (int)my_bins[i];
  int total;
  const int below = block_exclusive_scan(mine, wsum, total);
  const int over = total - below - mine;                   // elements in bins above my range
  if (over < need && need <= over + mine) {
    int cum = over, b = bins_per_thread - 1;
    for (; b > 0; --b) {
      const int hcount = (int)my_bins[b];
      if (cum + hcount >= need) break;
      cum += hcount;
    }
    out2[0] = b0 + b;
    out2[1] = cum;
  }
  __syncthreads();
  const int found = out2[0];
  const int cum = out2[1];
  __syncthreads();
  if (found < 0) return false;
  bin = found;
  above = cum;
  return true;
}

// Pooled value of position j over the eligible range [0, e).
__device__ __forceinline__ float pooled_at(const float* __restrict__ s, int e, int j, int pool, int k) {
  int lo = j - (k >> 1);
  int hi = lo + k - 1;
  lo = lo < 0 ? 0 : lo;
  hi = hi > e - 1 ? e - 1 : hi;
  if (pool == SPEC_POOL_MAX) {
    float m = s[lo];
    for (int t = lo + 1; t <= hi; ++t) m = fmaxf(m, s[t]);
    return m;
  }
  float a = 0.f;
  for (int t = lo; t <= hi; ++t) a += s[t];
  return a / (float)k;
}

// Key source: shared-memory resident keys, or recomputation from the scores.
struct KeySource {
  const uint32_t* keys;       // non-NULL when resident
  const float* scores;
  int e, pool, k;
  __device__ __forceinline__ uint32_t operator()(int j) const {
    return keys ? keys[j] : to_key(pooled_at(scores, e, j, pool, k));
  }
};

struct SelectScratch {
  uint32_t* hist;             // [kSelWarps][256]
  int* misc;                  // [2*kSelWarps + 8]
};

// Finds the key T of the `need`-th largest element of key(0..e): count(key > T) < need <=
// count(key >= T).  Returns T and need_eq = need - count(key > T) (how many elements equal to
// T belong to the selection).  Requires 1 <= need <= e.  All threads of the CTA must call.
__device__ inline void radix_select(const KeySource& key, int e, int need, const SelectScratch& sc,
                             uint32_t& T_out, int& need_eq_out) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t prefix = 0, mask = 0;
  int remaining = need;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = tid; i < kSelWarps * 256; i += kSelThreads) sc.hist[i] = 0;
    __syncthreads();
    uint32_t* myh = sc.hist + warp * 256;
    int run_d = -1, run_c = 0;
    for (int j = tid; j < e; j += kSelThreads) {
      const uint32_t kk = key(j);
      if ((kk & mask) == prefix) {
        const int dg = (kk >> shift) & 255;
        if (dg == run_d) {
          ++run_c;
        } else {
          if (run_c) atomicAdd(&myh[run_d], (uint32_t)run_c);
          run_d = dg;
          run_c = 1;
        }
      }
    }
    if (run_c) atomicAdd(&myh[run_d], (uint32_t)run_c);
    __syncthreads();
    if (tid < 256) {
      uint32_t tot = 0;
#pragma unroll
      for (int w = 0; w < kSelWarps; ++w) tot += sc.hist[w * 256 + tid];
      sc.hist[tid] = tot;
    }
    __syncthreads();
    if (warp == 0) {
      // lane owns bins [8*lane, 8*lane+8); suffix sums over lanes locate the digit.
      uint32_t b[8], s = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) { b[i] = sc.hist[lane * 8 + i]; s += b[i]; }
      uint32_t suf = s;                                  // inclusive suffix sum over lanes >= lane
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += t;
      }
      const uint32_t above = suf - s;                    // elements in bins of higher lanes
      if (above < (uint32_t)remaining && (uint32_t)remaining <= suf) {
        uint32_t cum = above;
        int dg = 7;
        for (; dg > 0; --dg) {
          if (cum + b[dg] >= (uint32_t)remaining) break;
          cum += b[dg];
        }
        sc.misc[0] = lane * 8 + dg;
        sc.misc[1] = (int)cum;                           // elements strictly above the digit
      }
    }
    __syncthreads();
    const int dg = sc.misc[0];
    remaining -= sc.misc[1];
    prefix |= (uint32_t)dg << shift;
    mask |= 255u << shift;
    __syncthreads();
  }
  T_out = prefix;
  need_eq_out = remaining;
}

// Visits, in ascending position, every selected position j of [0, e): key > T, or key == T and
// fewer than need_eq equal keys precede it.  emit(rank, j) receives the 0-based rank in the
// ascending output.  Returns the number of selected positions.  All threads must call.
template <class Emit>
__device__ inline int ordered_emit(const KeySource& key, int e, uint32_t T, int need_eq, const SelectScratch& sc, Emit emit) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int base_gt = 0, base_eq = 0;
  int* wg = sc.misc + 8;
  int* we = sc.misc + 8 + kSelWarps;
  for (int c0 = 0; c0 < e; c0 += kSelThreads * kSelVec) {
    const int j0 = c0 + tid * kSelVec;
    uint32_t kk[kSelVec];
    int gt = 0, eq = 0;
#pragma unroll
    for (int i = 0; i < kSelVec; ++i) {
      const int j = j0 + i;
      kk[i] = j < e ? key(j) : 0u;
      if (j < e) { gt += kk[i] > T; eq += kk[i] == T; }
    }
    int sgt = gt, seq = eq;                               // inclusive warp scans
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, sgt, o);
      const int b = __shfl_up_sync(0xffffffffu, seq, o);
      if (lane >= o) { sgt += a; seq += b; }
    }
    if (lane == 31) { wg[warp] = sgt; we[warp] = seq; }
    __syncthreads();
    int pre_gt = base_gt + sgt - gt, pre_eq = base_eq + seq - eq, tot_gt = 0, tot_eq = 0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) {
      const int a = wg[w], b = we[w];
      if (w < warp) { pre_gt += a; pre_eq += b; }
      tot_gt += a;
      tot_eq += b;
    }
#pragma unroll
    for (int i = 0; i < kSelVec; ++i) {
      const int j = j0 + i;
      if (j < e) {
        if (kk[i] > T) {
          emit(pre_gt + min(pre_eq, need_eq), j);
          ++pre_gt;
        } else if (kk[i] == T) {
          if (pre_eq < need_eq) emit(pre_gt + pre_eq, j);
          ++pre_eq;
        }
      }
    }
    base_gt += tot_gt;
    base_eq += tot_eq;
    __syncthreads();
  }
  return base_gt + min(base_eq, need_eq);
}

// ------------------------------------------- the CTA-wide steps of the selections -----

constexpr int kStreamBins = 2048;
constexpr int kListMax = 128;                    // members of the threshold's bin that are ranked against one another

__device__ __forceinline__ uint32_t sample_hash(uint32_t unit, uint32_t m) {
  uint32_t h = (unit * 0x9E3779B1u) ^ (m * 0x85EBCA6Bu);
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12;
  return h;
}

// Shared memory of the CTA-wide steps.
struct SelectMem {
  uint32_t hist[kStreamBins];  // all zero between steps
  alignas(16) uint32_t list[kListMax];
  int wsum[32];
  int res[8];
  uint32_t top;                // largest key (zero on entry)
};

// Counts digit dg of the warp's keys that are `in`; neighbouring lanes with equal digits (the
// runs that pooling produces) are merged into one update.
__device__ __forceinline__ void hist_update(uint32_t* hist, bool in, uint32_t dg, int lane) {
  const uint32_t ins = __ballot_sync(0xffffffffu, in);
  if (ins == 0) return;                                    // warp-uniform
  if (__popc(ins) <= 4) {
    if (in) atomicAdd(&hist[dg], 1u);
    return;
  }
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint32_t dg_prev = __shfl_up_sync(0xffffffffu, dg, 1);
  const bool head = in && (lane == 0 || !((ins >> (lane - 1)) & 1u) || dg_prev != dg);
  const uint32_t heads = __ballot_sync(0xffffffffu, head);
  if (head) {
    const uint32_t stop = (heads | ~ins) & ~(lt_mask | (1u << lane));   // next run, or a lane that is out
    atomicAdd(&hist[dg], (uint32_t)((stop ? __ffs(stop) - 1 : 32) - lane));
  }
}

// Finds the bin of the need-th largest element of the histogram, the number of elements in higher bins
// and in the bin itself, and clears the histogram.  False when it holds fewer than `need`.  Called by all
// threads; three synchronisations.
__device__ __forceinline__ bool find_bin(SelectMem& sm, int need, int& bin, int& above, int& count) {
  static_assert(kStreamBins == 4 * kSelThreads, "four bins to a thread");
  const int tid = threadIdx.x;
  __syncthreads();
  uint4* h4 = reinterpret_cast<uint4*>(sm.hist) + tid;
  const uint4 h = *h4;
  *h4 = make_uint4(0u, 0u, 0u, 0u);
  const int mine = (int)(h.x + h.y + h.z + h.w);
  int total;
  const int below = block_exclusive_scan(mine, sm.wsum, total);
  int over = total - below - mine;                         // elements in bins above mine
  if (over < need && need <= over + mine) {
    int b = 3, c = (int)h.w;
    if (over + c < need) { over += c; c = (int)h.z; b = 2;
      if (over + c < need) { over += c; c = (int)h.y; b = 1;
        if (over + c < need) { over += c; c = (int)h.x; b = 0; } } }
    sm.res[0] = 4 * tid + b;
    sm.res[1] = over;
    sm.res[2] = c;
    sm.res[3] = 0;                                         // the length of the list that may be made next
  }
  __syncthreads();
  bin = sm.res[0];
  above = sm.res[1];
  count = sm.res[2];
  return total >= need;
}

// A key that about rho of the sampled keys reach: samples are binned by their distance below the largest,
// 64 bins to a factor of two over 32 factors of two, or, if the rank lies deeper than that, by their
// leading 11 bits.  Scores that differ by a few per cent only (sums over many heads, averages) would crowd into a bin
// or two: the bin is cut again then, or the floor lets through more keys than there is room for (keep set of 1024
// among 32768 tokens whose scores are such sums: 29.6 -> 23.6 us).  0, which all keys reach, when the sample is too small to tell.  `keys`: N samples
// of this thread, 0 = none.  All threads of the CTA call this; the histogram is clear on entry and on return.
struct Floor {
  uint32_t key;
  int reach;                   // samples at or above it
};
template <int N>
__device__ __forceinline__ Floor floor_from_samples(SelectMem& sm, const uint32_t (&keys)[N], int take, int rate_shift) {
  // about take / 2^rate_shift samples lie above the threshold; the floor is taken four standard deviations further down
  const float m_exp = (float)take / (float)(1 << rate_shift);
  const int rho = (int)(m_exp + 4.f * sqrtf(m_exp) + 8.f);
  uint32_t top = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) top = max(top, keys[i]);
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0 && top) atomicMax(&sm.top, top);
  __syncthreads();
  top = sm.top;
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (keys[i]) atomicAdd(&sm.hist[kStreamBins - 1 - min((top - keys[i]) >> 17, (uint32_t)kStreamBins - 1)], 1u);
  int bin, above, count;
  if (!find_bin(sm, rho, bin, above, count)) return {0u, 0x7fffffff};
  if (bin > 0) {
    uint32_t depth = ((uint32_t)(kStreamBins - bin) << 17) - 1u;             // the bin's lower edge
    int higher = 0;
    if (above + count > rho + (rho >> 2) + 8) {            // the bin holds many more samples than were asked for: it is cut again
      const uint32_t upper = depth >> 17;
#pragma unroll
      for (int i = 0; i < N; ++i)
        if (keys[i] && (top - keys[i]) >> 17 == upper) atomicAdd(&sm.hist[kStreamBins - 1 - (((top - keys[i]) >> 6) & (kStreamBins - 1))], 1u);
      higher = above;
      find_bin(sm, rho - higher, bin, above, count);
      depth = (upper << 17) + ((uint32_t)(kStreamBins - bin) << 6) - 1u;
    }
    return {top > depth ? top - depth : 0u, higher + above + count};
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (keys[i]) atomicAdd(&sm.hist[keys[i] >> 21], 1u);
  find_bin(sm, rho, bin, above, count);
  return {(uint32_t)bin << 21, above + count};
}

// The key T of the need-th largest of keys[0..n), all of them in [lo, hi], and how many elements equal to T
// belong to the selection.  The range is cut into 2048 bins as fine as it allows, so that the threshold's
// bin holds a few dozen keys, which are ranked against one another; a fuller bin (ties) is cut again.  Called
// by all threads with the histogram clear.  RUNS: neighbouring keys are often equal (pooling wider than a few
// positions), so that neighbouring lanes' counts are merged first; for width 7 that costs more than it saves
// (64 units of 65536: 23.5 against 21.9 us), for average pooling over 64 it saves half of the step.
template <bool RUNS>
__device__ __forceinline__ void find_threshold(SelectMem& sm, const uint32_t* keys, int n, uint32_t lo, uint32_t hi, int need,
                                               uint32_t& T, int& need_eq) {
  const int tid = threadIdx.x;
  uint32_t span = hi - lo;
  for (;;) {
    const int shift = max(0, 21 - __clz((int)(span | 1u)));
    for (int i0 = 0; i0 < n; i0 += kSelThreads) {
      const uint32_t d = i0 + tid < n ? keys[i0 + tid] - lo : 0u;
      const bool in = i0 + tid < n && d <= span;
      if (RUNS) hist_update(sm.hist, in, d >> shift, tid & 31);
      else if (in) atomicAdd(&sm.hist[d >> shift], 1u);
    }
    int bin, above, count;
    find_bin(sm, need, bin, above, count);
    need -= above;
    lo += (uint32_t)bin << shift;
    if (shift == 0) break;                                 // lo is the key itself
    span = (1u << shift) - 1u;
    if (count > kListMax) continue;
    for (int i = tid; i < n; i += kSelThreads)
      if (keys[i] - lo <= span) sm.list[atomicAdd(&sm.res[3], 1)] = keys[i];
    __syncthreads();
    if (tid < count) {
      const uint32_t mine = sm.list[tid];
      int gt = 0, ge = 0;
      const uint4* l4 = reinterpret_cast<const uint4*>(sm.list);
      for (int j = 0; j < count; j += 4) {
        const uint4 o = l4[j >> 2];
        const int left = count - j;                        // what lies behind the list's end does not count
        gt += (o.x > mine) + (left > 1 && o.y > mine) + (left > 2 && o.z > mine) + (left > 3 && o.w > mine);
        ge += (o.x >= mine) + (left > 1 && o.y >= mine) + (left > 2 && o.z >= mine) + (left > 3 && o.w >= mine);
      }
      if (gt < need && need <= ge) {                       // every holder of the threshold key writes the same
        sm.res[4] = (int)mine;
        sm.res[5] = need - gt;
      }
    }
    __syncthreads();
    lo = (uint32_t)sm.res[4];
    need = sm.res[5];
    break;
  }
  T = lo;
  need_eq = need;
}

// Launches the streaming selection (select_stream.cu) for width-7 max pooling when the caller gave
// a workspace.  Returns SPEC_OK with *done = false when the problem is outside what that path serves.
SPEC_HIDDEN int run_stream_topk(const spec_problem* pr, const float* scores, int c_max, int n_forced_tail, int32_t* idx_out,
                                int32_t* count_out, int n_vert, int32_t* vert_out, int32_t* vert_count_out, void* workspace,
                                size_t workspace_bytes, int32_t* status_word, cudaStream_t st, bool* done);

}  // namespace spec
