// Pooling + top-C selection for the default pooling (Algorithm 1 lines 10, 11 and 13 with the
// hyper-parameter table's Max pool of width 7).
//
// A maximum of seven reaches a floor exactly when one of the seven scores does.  So given a floor that
// lies under the final threshold, the candidates for selection are the positions within three of a
// raw score at or above the floor: a sweep over the scores costs one comparison per score, and
// pooled values are only ever computed for candidates.  A warp holds 1024 scores in registers (eight
// float4 per lane), turns them into hit bits, widens the bits by three positions on either side
// (bit arithmetic on eight nibbles at a time), lists the groups of four positions that hold candidates and
// pools and ranks those, a group to a lane.
//
// Long units take three kernels on the caller's stream, chained as programmatic dependents; no CTA
// ever waits for another:
//   1. sample_floor_kernel, one CTA per (sequence, layer, KV head) unit: pools one 32-byte sector
//      out of every 32..128 positions (a sector holds the whole width-7 window of its fourth
//      score) and takes, from a histogram of the sampled keys below the largest of them, the key a few
//      standard deviations below the rank the budget corresponds to.  That key is a floor under
//      the final threshold with overwhelming probability, and it does not depend on where in the
//      unit the large scores sit.
//   2. stream_sweep_kernel, one warp per chunk of 1024 positions: the scores are read from global
//      memory once, straight into registers (the loads are issued before the floors are waited for);
//      candidates go, as (key, position) pairs in position order, to the chunk's own segment of
//      the unit's candidate array in the workspace.
//   3. stream_finish_kernel, one CTA per unit and budget, or per unit where those are many: the
//      candidates come into shared memory, the exact threshold is found (find_threshold), and the winners
//      are written out as they stand, already in ascending position, ties to the lower position.
// Units of up to 16384 positions skip the workspace and the three launches:
// unit_select_kernel holds a unit in the registers of one CTA and does the same steps.
//
// If the floor was too high or too low (fewer candidates than the budget, or more than the finishing
// CTA holds: only with massively tied scores), the CTA falls back to the generic selection that
// recomputes pooled keys from global memory.  The result is exact in every case.
#include "select_common.cuh"

#include <algorithm>
#include <cmath>

namespace spec {

constexpr int kWarpSteps = 8;                    // 128-position steps a warp holds in registers
constexpr int kWarpSpan = kWarpSteps * 128;
constexpr int kListSlots = kWarpSpan / 4;         // groups of four positions of a warp
constexpr int kMaxSamples = 4096;
constexpr uint32_t kNoSelection = 0xFFFFFFFFu;   // floor value of a unit that keeps everything or nothing

struct StreamParams {
  const float* scores;
  const int32_t* cu;
  int64_t T;
  int n_in, L, H, n_forced, c_max, n_vert;
  int rounds;                 // a sweeping warp's chunk is rounds * kWarpSpan positions
  int chunks_max;             // chunks per unit
  int max_len;                // the host's bound on any sequence length (sizes the grid)
  int held_cap;               // candidates the finishing CTA can hold in shared memory
  int32_t* head;              // [units][head_words]: floor key, three unused, then a candidate count per chunk
  int head_words;
  uint2* cand;                // candidate (key, position) pairs
  int64_t row_entries;        // candidate entries per (layer, KV head) row
  int32_t* idx_out;
  int32_t* count_out;
  int32_t* vert_out;
  int32_t* vert_count_out;
  int32_t* status;
};

struct UnitGeom {
  int begin, n, forced, e;
  bool over;                  // longer than the host's bound: treated as empty and reported
  int take[2];
  const float* src;
  int mis, X;                 // x = position + mis: multiples of four in x are 16-byte boundaries; positions are [mis, X)
  int64_t cand_off;
};

// row = layer * H + head
__device__ __forceinline__ UnitGeom unit_geom_of(const StreamParams& p, int s, int row) {
  UnitGeom g;
  seq_range(p.cu, p.n_in, s, g.begin, g.n);
  g.over = g.n > p.max_len;
  if (g.over) g.n = 0;
  g.forced = min(p.n_forced, g.n);
  g.e = g.n - g.forced;
  g.take[0] = max(min(p.c_max - g.forced, g.e), 0);
  g.take[1] = max(min(p.n_vert, g.e), 0);
  g.src = p.scores + (int64_t)row * p.T + g.begin;
  g.mis = (int)((reinterpret_cast<uintptr_t>(g.src) >> 2) & 3u);
  g.X = g.e + g.mis;
  // even, so that a segment starts on a 16-byte boundary
  g.cand_off = (int64_t)row * p.row_entries + ((g.begin + 1) & ~1) + (int64_t)s * kSelCandSlack;
  return g;
}
__device__ __forceinline__ UnitGeom unit_geom(const StreamParams& p, int unit) {
  const int rows = p.H * p.L;
  return unit_geom_of(p, unit / rows, unit % rows);
}

// The float that a raw score has to reach; everything below the key of -infinity maps to -infinity.
__device__ __forceinline__ float key_to_float(uint32_t key) {
  if (key <= 0x007FFFFFu) return -INFINITY;
  return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}

// Writes the positions of the selected candidates in the order in which they stand: key > T, and the first
// need_eq of key == T.  A warp owns a contiguous run of candidates and writes 32 at a time.
__device__ __forceinline__ void emit_selected(SelectMem& sm, const uint32_t* keys, const uint32_t* pos, int n, uint32_t T, int need_eq,
                                              int32_t* __restrict__ idx) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt_mask = (1u << lane) - 1u;
  const int run = ((n + kSelThreads - 1) / kSelThreads) * 32;
  const int b = min(warp * run, n), e = min(b + run, n);
  int gt = 0, eq = 0;
  for (int i = b + lane; i < e; i += 32) {
    const uint32_t k = keys[i];
    gt += k > T;
    eq += k == T;
  }
  const uint32_t both = __reduce_add_sync(0xffffffffu, (uint32_t)gt | ((uint32_t)eq << 16));    // fewer than 2^15 candidates
  if (lane == 0) sm.wsum[warp] = (int)both;
  __syncthreads();
  const int lower = lane < warp && lane < kSelWarps ? sm.wsum[lane] : 0;
  const uint32_t before = __reduce_add_sync(0xffffffffu, (uint32_t)lower);
  int pre_gt = (int)(before & 0xffffu), pre_eq = (int)(before >> 16);
  for (int i0 = b; i0 < e; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t k = i < e ? keys[i] : 0u;
    const bool is_gt = i < e && k > T, is_eq = i < e && k == T;
    const uint32_t bg = __ballot_sync(0xffffffffu, is_gt), be = __ballot_sync(0xffffffffu, is_eq);
    if (is_gt || is_eq) {
      const int my_gt = pre_gt + __popc(bg & lt_mask), my_eq = pre_eq + __popc(be & lt_mask);
      if (is_gt) idx[my_gt + min(my_eq, need_eq)] = (int32_t)pos[i];
      else if (my_eq < need_eq) idx[my_gt + my_eq] = (int32_t)pos[i];
    }
    pre_gt += __popc(bg);
    pre_eq += __popc(be);
  }
}

// The shared memory of the generic selection, taken from the candidates'.
constexpr size_t kGenericBytes = (size_t)(kSelWarps * 256 + 2 * kSelWarps + 8) * 4;

// The list of one budget of a unit, given its candidates (or `failed`, or too few of them: the generic
// selection, in the shared memory at `scratch`, which is the candidates').  False when they are gone.
__device__ __forceinline__ bool finish_unit(const StreamParams& p, const UnitGeom& g, int unit, int b, SelectMem& sm, const uint32_t* keys,
                                            const uint32_t* pos, int n, bool failed, uint32_t floor_key, uint32_t top, void* scratch) {
  const int tid = threadIdx.x;
  const int width = b == 0 ? p.c_max : p.n_vert;
  int32_t* idx = (b == 0 ? p.idx_out : p.vert_out) + (int64_t)unit * width;
  int32_t* cnt = b == 0 ? p.count_out : p.vert_count_out;
  const int tail = b == 0 ? g.forced : 0;
  const int tk = g.take[b];
  for (int q = tk + tid; q < width; q += kSelThreads) idx[q] = (q - tk < tail) ? g.e + (q - tk) : -1;
  if (cnt && tid == 0) cnt[unit] = tk + tail;
  if (tk >= g.e) {
    for (int q = tid; q < tk; q += kSelThreads) idx[q] = q;        // every eligible position is kept
  } else if (tk > 0) {
    uint32_t T;
    int need_eq;
    if (!failed && n >= tk) {
      find_threshold<false>(sm, keys, n, floor_key, top, tk, T, need_eq);
      emit_selected(sm, keys, pos, n, T, need_eq, idx);
    } else {
      __syncthreads();
      SelectScratch sc;
      sc.hist = reinterpret_cast<uint32_t*>(scratch);
      sc.misc = reinterpret_cast<int*>(sc.hist + kSelWarps * 256);
      KeySource key;
      key.scores = g.src;
      key.e = g.e; key.pool = SPEC_POOL_MAX; key.k = 7;
      key.keys = nullptr;
      radix_select(key, g.e, tk, sc, T, need_eq);
      ordered_emit(key, g.e, T, need_eq, sc, [&](int rank, int j) { idx[rank] = j; });
      return false;
    }
  }
  return true;
}
// The list of budget b of a unit, or (BOTH) of its two.
template <bool BOTH>
__device__ __forceinline__ void finish_budgets(const StreamParams& p, const UnitGeom& g, int unit, int b, SelectMem& sm, const uint32_t* keys,
                                               const uint32_t* pos, int n, bool failed, uint32_t floor_key, uint32_t top, void* scratch) {
  if constexpr (BOTH) {
#pragma unroll 1
    for (b = 0; b < 2; ++b)
      if (!finish_unit(p, g, unit, b, sm, keys, pos, n, failed, floor_key, top, scratch)) failed = true;
  } else {
    finish_unit(p, g, unit, b, sm, keys, pos, n, failed, floor_key, top, scratch);
  }
}
__device__ __forceinline__ bool cuts(const UnitGeom& g, int b) { return g.take[b] > 0 && g.take[b] < g.e; }

// -------------------------------------------------------- a warp's scores in registers --

// n_steps (0..8, warp-uniform) steps of 128 scores from x0 on, four per lane and step, and the three scores
// before and after them (lanes 0..2).  Slots that are not positions of the unit hold -infinity.
struct WarpScores {
  float4 v[kWarpSteps];
  float before, after;
  int x0, n_steps;
};

__device__ __forceinline__ float score_at(const UnitGeom& g, int x) {
  return (x >= g.mis && x < g.X) ? __ldcg(g.src + (x - g.mis)) : -INFINITY;
}
__device__ __forceinline__ void load_scores(const UnitGeom& g, int x0, int n_steps, int lane, WarpScores& w) {
  w.x0 = x0;
  w.n_steps = n_steps;
  if (n_steps == kWarpSteps && x0 - 4 >= g.mis && x0 + kWarpSpan + 4 <= g.X) {    // warp-uniform: full, with neighbours on both sides
    const float* at = g.src + (x0 - g.mis);
#pragma unroll
    for (int k = 0; k < kWarpSteps; ++k) w.v[k] = __ldcg(reinterpret_cast<const float4*>(at) + k * 32 + lane);
    w.before = __ldcg(at - 3 + min(lane, 2));
    w.after = __ldcg(at + kWarpSpan + min(lane, 2));
    return;
  }
#pragma unroll
  for (int k = 0; k < kWarpSteps; ++k) {
    w.v[k] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (k < n_steps) {
      const int x = x0 + k * 128 + lane * 4;
      if (x >= g.mis && x + 4 <= g.X) w.v[k] = __ldcg(reinterpret_cast<const float4*>(g.src + (x - g.mis)));
      else w.v[k] = make_float4(score_at(g, x), score_at(g, x + 1), score_at(g, x + 2), score_at(g, x + 3));
    }
  }
  w.before = lane < 3 ? score_at(g, x0 - 3 + lane) : -INFINITY;
  w.after = lane < 3 ? score_at(g, x0 + n_steps * 128 + lane) : -INFINITY;
}

// Candidate bits of this lane (bit 4k + u: its position u of step k), and how many the warp has.
struct WarpCandidates {
  uint32_t mask;
  int total;
};

// Sets `bit` if v >= floor_f, in two instructions; written in C++, the bit is selected first and costs a third.
__device__ __forceinline__ void set_if_reached(uint32_t& bits, float v, float floor_f, uint32_t bit) {
  asm("{\n.reg .pred p;\nsetp.ge.f32 p, %1, %2;\n@p or.b32 %0, %0, %3;\n}" : "+r"(bits) : "f"(v), "f"(floor_f), "r"(bit));
}
__device__ __forceinline__ WarpCandidates find_candidates(const UnitGeom& g, const WarpScores& w, float floor_f, int lane) {
  constexpr uint32_t ones = 0x11111111u;
  uint32_t hit = 0;
#pragma unroll
  for (int k = 0; k < kWarpSteps; ++k) {
    set_if_reached(hit, w.v[k].x, floor_f, 1u << (4 * k));
    set_if_reached(hit, w.v[k].y, floor_f, 2u << (4 * k));
    set_if_reached(hit, w.v[k].z, floor_f, 4u << (4 * k));
    set_if_reached(hit, w.v[k].w, floor_f, 8u << (4 * k));
  }
  const uint32_t near_l = __ballot_sync(0xffffffffu, w.before >= floor_f) & 7u;
  const uint32_t near_r = __ballot_sync(0xffffffffu, w.after >= floor_f) & 7u;
  WarpCandidates c;
  c.mask = 0;
  c.total = 0;
  if (!__any_sync(0xffffffffu, hit != 0) && near_l == 0 && near_r == 0) return c;
  // the nibbles to the left and to the right of each of mine: neighbouring lanes, or the neighbouring step
  uint32_t left = __shfl_up_sync(0xffffffffu, hit, 1), right = __shfl_down_sync(0xffffffffu, hit, 1);
  const uint32_t of31 = __shfl_sync(0xffffffffu, hit, 31), of0 = __shfl_sync(0xffffffffu, hit, 0);
  if (lane == 0) left = (of31 << 4) | (near_l << 1);
  if (lane == 31) right = (of0 >> 4) | (near_r << (4 * max(w.n_steps - 1, 0)));
  uint32_t any = hit | (hit >> 1);
  any = (any | (any >> 2)) & ones;
  const uint32_t l1 = (left >> 1) & ones, l2 = (left >> 2) & ones, l3 = (left >> 3) & ones;
  const uint32_t r0 = right & ones, r1 = (right >> 1) & ones, r2 = (right >> 2) & ones;
  c.mask = (any | l1 | l2 | l3) | ((any | l2 | l3 | r0) << 1) | ((any | l3 | r0 | r1) << 2) | ((any | r0 | r1 | r2) << 3);
  if (w.n_steps < kWarpSteps) c.mask &= (1u << (4 * w.n_steps)) - 1u;
  if (w.x0 < g.mis || w.x0 + w.n_steps * 128 > g.X) {      // only positions of the unit
#pragma unroll
    for (int k = 0; k < kWarpSteps; ++k) {
      const int lo = g.mis - (w.x0 + k * 128 + lane * 4), hi = g.X - (w.x0 + k * 128 + lane * 4);   // valid u: lo <= u < hi
      const uint32_t ok = (0xfu << min(max(lo, 0), 4)) & (hi >= 4 ? 0xfu : (1u << max(hi, 0)) - 1u) & 0xfu;
      c.mask &= ~((ok ^ 0xfu) << (4 * k));
    }
  }
  c.total = (int)__reduce_add_sync(0xffffffffu, (uint32_t)__popc(c.mask));
  return c;
}

// Calls put(rank, key, position) for every candidate of the warp, rank in position order from `base` on.  The groups of
// four positions that hold candidates (a dozen of 256, as a rule) are listed in position order in
// shared memory; every lane takes one from the list, pools its four positions from the twelve scores around
// them, read again from L2, and ranks them by a scan over the list.  (The sweep is bound by the instructions that it
// issues.  With every lane walking its own groups, two to four turns of the loop for the warp, it took 674 per
// 1024 positions and 35.6 us for 256 units of 131072; with this, a short path for chunks inside a unit and two
// instructions per score in find_candidates, 530 and 27.4.  Leaving out steps without candidates, or a persistent
// sweep that copies its chunks ahead into shared memory, was slower.)
template <class Put>
__device__ __forceinline__ void pool_candidates(const UnitGeom& g, const WarpScores& w, const WarpCandidates& c, int base, int lane, uint16_t* list, Put put) {
  if (c.total == 0) return;                                // warp-uniform
  const uint32_t lt_mask = (1u << lane) - 1u;
  int count = 0;
#pragma unroll
  for (int k = 0; k < kWarpSteps; ++k) {
    const uint32_t nib = (c.mask >> (4 * k)) & 15u;
    const uint32_t has = __ballot_sync(0xffffffffu, nib != 0);
    if (nib) list[count + __popc(has & lt_mask)] = (uint16_t)(nib | ((uint32_t)(k * 32 + lane) << 4));
    count += __popc(has);
  }
  __syncwarp();
#pragma unroll 1
  for (int i0 = 0; i0 < count; i0 += 32) {
    const uint32_t entry = i0 + lane < count ? list[i0 + lane] : 0u;
    const uint32_t nib = entry & 15u;
    const int x0 = w.x0 + (int)(entry >> 4) * 4;
    float4 pv, cv, nv;
    if (nib != 0) {
      if (x0 - 4 >= g.mis && x0 + 8 <= g.X) {
        const float4* at = reinterpret_cast<const float4*>(g.src + (x0 - g.mis));
        pv = __ldcg(at - 1); cv = __ldcg(at); nv = __ldcg(at + 1);
      } else {
        pv = make_float4(0.f, score_at(g, x0 - 3), score_at(g, x0 - 2), score_at(g, x0 - 1));
        cv = make_float4(score_at(g, x0), score_at(g, x0 + 1), score_at(g, x0 + 2), score_at(g, x0 + 3));
        nv = make_float4(score_at(g, x0 + 4), score_at(g, x0 + 5), score_at(g, x0 + 6), 0.f);
      }
    }
    const int mine = __popc(nib);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      asm volatile("{\n.reg .pred p;\n.reg .b32 t;\nshfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n@p add.s32 %0, %0, t;\n}" : "+r"(incl) : "r"(o));
    }
    const int at = base + incl - mine;
    base += __shfl_sync(0xffffffffu, incl, 31);
    if (nib != 0) {
      // the four windows share the middle four; neighbouring windows share a pair on either side
      const float mid = fmax3(cv.x, cv.y, fmaxf(cv.z, cv.w)), l12 = fmaxf(pv.z, pv.w), r78 = fmaxf(nv.x, nv.y);
      const uint32_t k4[4] = {to_key(fmax3(mid, pv.y, l12)), to_key(fmax3(mid, l12, nv.x)), to_key(fmax3(mid, pv.w, r78)), to_key(fmax3(mid, r78, nv.z))};
      const int j0 = x0 - g.mis;
      int to[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) to[u] = at + __popc(nib & ((1u << u) - 1u));
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (nib & (1u << u)) put(to[u], k4[u], j0 + u);
    }
  }
  __syncwarp();                                            // the list is free again
}

// ---------------------------------------------------------------- 1. the floor -------

// One sample per 2^shift positions of a unit (of the eligible ones; extent: with the slots before the first).
__host__ __device__ inline int sample_shift(int eligible, int extent) {
  int shift = eligible >= 65536 ? 7 : eligible >= 16384 ? 6 : 5;
  while (((extent >> shift) + 1) > kMaxSamples) ++shift;
  return shift;
}

__global__ void __launch_bounds__(kSelThreads) sample_floor_kernel(const StreamParams p) {
  __shared__ __align__(16) SelectMem sm;
  const int unit = blockIdx.x, tid = threadIdx.x;
  reinterpret_cast<uint4*>(sm.hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) sm.top = 0;
  // The sweep may start as soon as every CTA of this grid knows that the scores are complete: its warps issue
  // their loads and wait for this grid before they read the floor.
  wait_for_previous_grid();
  launch_dependents();
  const UnitGeom g = unit_geom(p, unit);
  const int tk = max(g.take[0], g.take[1]);
  const bool selects = (g.take[0] > 0 && g.take[0] < g.e) || (g.take[1] > 0 && g.take[1] < g.e);
  uint32_t floor_key = kNoSelection;
  if (selects) {
    // x = position + mis8 puts every multiple of eight on a 32-byte boundary of global memory
    const int mis8 = (int)((reinterpret_cast<uintptr_t>(g.src) >> 2) & 7u);
    const int X = g.e + mis8;
    const int shift = sample_shift(g.e, X);
    const int spg = 1 << (shift - 3);                                // sectors per sample group
    const int n_sectors = (X + 7) >> 3;
    const int n_groups = (n_sectors + spg - 1) / spg;                // <= kMaxSamples
    uint32_t keys[kMaxSamples / kSelThreads];
#pragma unroll
    for (int i = 0; i < kMaxSamples / kSelThreads; ++i) {
      const int m = tid + i * kSelThreads;
      keys[i] = 0;                                                   // 0: no sample here
      if (m >= n_groups) continue;
      const int q = m * spg + (int)(sample_hash((uint32_t)unit, (uint32_t)m) % (uint32_t)min(spg, n_sectors - m * spg));
      const int p0 = q * 8 - mis8;                                   // position of the sector's first score
      const int centre = p0 + 3;
      if (centre < 0 || centre >= g.e) continue;
      float v[7];
      if (p0 >= 0 && p0 + 8 <= g.e) {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(g.src + p0));
        const float4 b = __ldcg(reinterpret_cast<const float4*>(g.src + p0 + 4));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z;
      } else {
#pragma unroll
        for (int u = 0; u < 7; ++u) v[u] = (p0 + u >= 0 && p0 + u < g.e) ? __ldcg(g.src + p0 + u) : -INFINITY;
      }
      keys[i] = to_key(fmax3(fmax3(v[0], v[1], v[2]), fmax3(v[3], v[4], v[5]), v[6]));   // pooled value of the centre
    }
    __syncthreads();
    floor_key = floor_from_samples(sm, keys, tk, shift).key;
  }
  if (tid == 0) {
    if (g.over) report(p.status, SPEC_ERR_BAD_ARG);
    p.head[(int64_t)unit * p.head_words] = (int32_t)floor_key;
  }
}

// ---------------------------------------------------------------- 2. the sweep -------

constexpr int kSweepThreads = 128, kSweepCtas = 8;        // 6 CTAs to an SM: 135.0 us for selection and gather of 256 units of 131072, 8: 133.0, 10: 136.1
constexpr int kSweepWarps = kSweepThreads / 32;

// One warp per chunk; warps never meet.  A lane's eight 16-byte loads are in flight at once.  The finishing kernel is not let
// in early: its CTAs would take the first SMs that the sweep leaves, two to each, and run there in each other's way, while
// other SMs have none (64 units of 131072: 24.3 -> 22.0 us; 64 units of 65536 with all scores tied, where a CTA works for
// 200 us, 366 -> 272).
__global__ void __launch_bounds__(kSweepThreads, kSweepCtas) stream_sweep_kernel(const StreamParams p) {
  __shared__ uint16_t lists[kSweepWarps][kListSlots];
  const int lane = threadIdx.x & 31;
  const int chunk_id = blockIdx.x * kSweepWarps + (threadIdx.x >> 5);
  const int row = blockIdx.y, s = blockIdx.z;
  const UnitGeom g = unit_geom_of(p, s, row);
  const int chunk = p.rounds * kWarpSpan;
  const int c0 = chunk_id * chunk;
  WarpScores w;
  if (c0 < g.X) load_scores(g, c0, min(kWarpSteps, (g.X - c0 + 127) >> 7), lane, w);
  wait_for_previous_grid();                                // the floors are written by the grid before this one
  if (c0 >= g.X) return;
  int32_t* hd = p.head + ((int64_t)s * (p.H * p.L) + row) * p.head_words;
  const uint32_t floor_key = (uint32_t)__ldcg(hd);
  if (floor_key == kNoSelection) return;
  const float floor_f = key_to_float(floor_key);
  uint2* dst = p.cand + g.cand_off + (int64_t)chunk_id * chunk;
  int n = 0;
  for (int r = 0;; ++r) {
    const WarpCandidates c = find_candidates(g, w, floor_f, lane);
    pool_candidates(g, w, c, n, lane, lists[threadIdx.x >> 5], [&](int at, uint32_t key, int j) {
      *reinterpret_cast<uint2*>(reinterpret_cast<char*>(dst) + (uint32_t)at * 8u) = make_uint2(key, (uint32_t)j);
    });
    n += c.total;
    const int x = c0 + (r + 1) * kWarpSpan;
    if (r + 1 >= p.rounds || x >= g.X) break;
    load_scores(g, x, min(kWarpSteps, (g.X - x + 127) >> 7), lane, w);
  }
  if (lane == 0) hd[4 + chunk_id] = n;                     // a segment is as long as the chunk: it cannot overflow
}

// ------------------------------------------------------------- 3. the finishing CTA --

static size_t held_bytes(int held_cap) { return std::max((size_t)held_cap * 8, kGenericBytes); }

// One CTA per unit and budget while all of them are on the GPU at once, two to an SM; BOTH: one per unit for its two budgets, which
// then cost a second threshold and emission but no second copy of the candidates (148 units of 17001, 384 and 400 kept:
// 15.5 us with two CTAs to a unit, 17.1 with one; 2048 units 137 and 118).  CTAS: three to an SM with 40 registers a thread for
// units in several waves whose candidates leave the memory (2048 units of 3000, 428 kept: 83 -> 73 us; 256 units of 131072,
// all there at once, 47.0 -> 48.2).  The next kernel is not let in early
// either: the floor CTAs of a selection that follows would crowd on the few SMs with room beside two finishing CTAs, and
// the sweep behind them waits for the slowest (256 units of 131072, one selection after the other: 70.4 -> 46.9 us each).
template <int CTAS, bool BOTH>
__global__ void __launch_bounds__(kSelThreads, CTAS) stream_finish_kernel(const StreamParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ __align__(16) SelectMem sm;
  __shared__ int chunk_at[kSelThreads], chunk_n[kSelThreads];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int unit = blockIdx.x, b = BOTH ? 0 : blockIdx.y;
  reinterpret_cast<uint4*>(sm.hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) sm.top = 0;
  wait_for_previous_grid();                                // the candidates are written by the grid before this one
  const UnitGeom g = unit_geom(p, unit);
  const int32_t* hd = p.head + (int64_t)unit * p.head_words;
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* pos = keys + p.held_cap;
  const bool selects = cuts(g, b) || (BOTH && cuts(g, 1));
  int n = 0;
  bool failed = false;
  uint32_t floor_key = 0, top = 0;
  if (selects) {
    floor_key = (uint32_t)__ldcg(hd);
    const int chunk = p.rounds * kWarpSpan;
    const int n_chunks = (g.X + chunk - 1) / chunk;        // <= kSelThreads, checked on the host
    const int cnt = tid < n_chunks ? __ldcg(hd + 4 + tid) : 0;
    chunk_at[tid] = block_exclusive_scan(cnt, sm.wsum, n);
    chunk_n[tid] = cnt;
    failed = n > p.held_cap;
    __syncthreads();
    if (!failed) {
      // the segments one after the other: a warp takes every 16th, four at a time, two pairs per lane and load
      const uint2* segs = p.cand + g.cand_off;
      for (int c0 = warp; c0 < n_chunks; c0 += 4 * kSelWarps) {
        uint4 v[4];
        int cn[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = c0 + u * kSelWarps;
          cn[u] = c < n_chunks ? chunk_n[c] : 0;
          if (2 * lane < cn[u]) v[u] = __ldcg(reinterpret_cast<const uint4*>(segs + (int64_t)c * chunk) + lane);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (cn[u] == 0) continue;                        // warp-uniform
          const int c = c0 + u * kSelWarps, at = chunk_at[c];
          for (int i = 2 * lane; i < cn[u]; i += 64) {
            if (i >= 64) v[u] = __ldcg(reinterpret_cast<const uint4*>(segs + (int64_t)c * chunk) + (i >> 1));
            keys[at + i] = v[u].x;
            pos[at + i] = v[u].y;
            top = max(top, v[u].x);
            if (i + 1 < cn[u]) {
              keys[at + i + 1] = v[u].z;
              pos[at + i + 1] = v[u].w;
              top = max(top, v[u].z);
            }
          }
        }
      }
      __syncwarp();
      top = __reduce_max_sync(0xffffffffu, top);
      if (lane == 0) atomicMax(&sm.top, top);
    }
    __syncthreads();
    top = sm.top;
  }
  finish_budgets<BOTH>(p, g, unit, b, sm, keys, pos, n, failed, floor_key, top, smem_raw);
}

// --------------------------------------------------- short units: all steps in one CTA --

constexpr int kUnitSlots = kSelWarps * kWarpSpan;          // 16384
constexpr int kUnitSampleShift = 4;                        // the floor's sample: one position in 16

// One CTA per unit and budget, or BOTH in one as above (256 units of 16384, 384 and 400 kept: 20.8 us with two CTAs to a unit,
// 14.7 with one): the unit's scores in the registers of 16 warps, the floor from a sample of them, the candidates in shared memory.
template <bool BOTH>
__global__ void __launch_bounds__(kSelThreads, 2) unit_select_kernel(const StreamParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ __align__(16) SelectMem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int unit = blockIdx.x, b = BOTH ? 0 : blockIdx.y;
  reinterpret_cast<uint4*>(sm.hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) sm.top = 0;
  wait_for_previous_grid();
  launch_dependents();
  const UnitGeom g = unit_geom(p, unit);
  if (tid == 0 && b == 0 && g.over) report(p.status, SPEC_ERR_BAD_ARG);
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* pos = keys + p.held_cap;
  int n = 0;
  bool failed = false;
  uint32_t floor_key = 0, top = 0;
  if (cuts(g, b) || (BOTH && cuts(g, 1))) {
    const int n_steps = (g.X + 127) >> 7;                  // <= kSelWarps * kWarpSteps, checked on the host
    const int per_warp = (n_steps + kSelWarps - 1) / kSelWarps;
    const int s0 = warp * per_warp;
    WarpScores w;
    load_scores(g, s0 * 128, max(0, min(per_warp, n_steps - s0)), lane, w);
    // ---- the floor: in every step, one lane in four pools its first or its last position
    uint32_t samples[kWarpSteps];
#pragma unroll
    for (int k = 0; k < kWarpSteps; ++k) {
      samples[k] = 0;
      if (k >= w.n_steps) continue;                        // warp-uniform
      const float4 v = w.v[k];
      const int u = k & 1 ? 3 : 0;
      float q0, q1, q2;
      if (u == 0) {
        q0 = __shfl_up_sync(0xffffffffu, v.y, 1); q1 = __shfl_up_sync(0xffffffffu, v.z, 1); q2 = __shfl_up_sync(0xffffffffu, v.w, 1);
      } else {
        q0 = __shfl_down_sync(0xffffffffu, v.x, 1); q1 = __shfl_down_sync(0xffffffffu, v.y, 1); q2 = __shfl_down_sync(0xffffffffu, v.z, 1);
      }
      const int x = w.x0 + k * 128 + lane * 4 + u;
      const bool mine = (int)(sample_hash((uint32_t)unit, (uint32_t)((s0 + k) * 8 + (lane >> 2))) & 3u) == (lane & 3);
      if (mine && x >= g.mis && x < g.X) samples[k] = to_key(fmax3(fmax3(v.x, v.y, v.z), fmax3(v.w, q0, q1), q2));
    }
    __syncthreads();
    floor_key = floor_from_samples(sm, samples, BOTH ? max(g.take[0], g.take[1]) : g.take[b], kUnitSampleShift).key;
    // ---- the candidates
    const WarpCandidates c = find_candidates(g, w, key_to_float(floor_key), lane);
    __syncthreads();                                       // the scan's memory is free; everyone has the sample's largest key
    if (lane == 0) sm.wsum[warp] = c.total;
    if (tid == 0) sm.top = 0;
    __syncthreads();
    const int wt = lane < kSelWarps ? sm.wsum[lane] : 0;
    n = (int)__reduce_add_sync(0xffffffffu, (uint32_t)wt);
    const int base = (int)__reduce_add_sync(0xffffffffu, (uint32_t)(lane < warp ? wt : 0));
    failed = n > p.held_cap;
    if (!failed) {
      pool_candidates(g, w, c, base, lane, reinterpret_cast<uint16_t*>(pos + p.held_cap) + warp * kListSlots, [&](int at, uint32_t key, int j) {
        keys[at] = key;
        pos[at] = (uint32_t)j;
        top = max(top, key);
      });
      __syncwarp();
      top = __reduce_max_sync(0xffffffffu, top);
      if (lane == 0) atomicMax(&sm.top, top);
    }
    __syncthreads();
    top = sm.top;
  }
  finish_budgets<BOTH>(p, g, unit, b, sm, keys, pos, n, failed, floor_key, top, smem_raw);
}

// ------------------------------------------------------------------ host side ---------

// Two budgets of a unit in one CTA: where a CTA for each would not all be on the GPU at once.
static bool both_budgets(const StreamParams& p, int64_t n_units) { return p.n_vert > 0 && n_units > sm_count(); }

// The one-CTA selection of short units.  *done = false: the shapes do not fit it.
static int run_unit_topk(const spec_problem* pr, StreamParams p, cudaStream_t st, bool* done) {
  *done = false;
  // A unit is held from the 16-byte boundary at or below its first score: up to three more slots,
  // none when every unit is known to start on such a boundary.
  const bool aligned = !pr->cu_seqlens && (reinterpret_cast<uintptr_t>(p.scores) & 15u) == 0 && pr->total_tokens % 4 == 0;
  if (p.max_len < 1 || p.max_len + (aligned ? 0 : 3) > kUnitSlots) return SPEC_OK;
  const int64_t n_units = (int64_t)pr->n_seq * pr->n_layers * pr->n_kv_heads;
  if (n_units < 1 || n_units > 0x7fffffff) return SPEC_OK;
  // The floor, from one sample in 16, lets through 1.4 (budget 2048) to 2.5 (256) times the budget.  For units in several waves
  // of up to 8192 positions there is room for all of them, so that ties never need the generic selection (2048 units of 3000 of
  // five values 178 -> 68 us).  Not for longer units, where it costs more (2048 units of 16384 with room for 12000 94 -> 105 us),
  // nor for fewer, where a kernel that follows starts later beside that memory (64 units of 4164 with their gather 14.0 -> 15.8).
  const bool room_for_all = n_units > 2 * sm_count() && p.max_len <= 8192;
  p.held_cap = ((room_for_all ? p.max_len : std::min(5 * std::max(p.c_max, p.n_vert) / 2 + 1024, p.max_len)) + 3) & ~3;
  const size_t smem = held_bytes(p.held_cap) + kSelWarps * kListSlots * sizeof(uint16_t);
  if (smem > (size_t)kSmemLimit - 16 * 1024) return SPEC_OK;
  static int set[64] = {0};
  int dev = 0;
  SPEC_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SPEC_OK;
  if (!__atomic_load_n(&set[dev], __ATOMIC_ACQUIRE)) {
    SPEC_CUDA_OK(cudaFuncSetAttribute(unit_select_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - 16 * 1024));
    SPEC_CUDA_OK(cudaFuncSetAttribute(unit_select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - 16 * 1024));
    __atomic_store_n(&set[dev], 1, __ATOMIC_RELEASE);
  }
  const bool both = both_budgets(p, n_units);
  SPEC_CUDA_OK(launch_dependent(both ? unit_select_kernel<true> : unit_select_kernel<false>, dim3((unsigned)n_units, p.n_vert > 0 && !both ? 2 : 1),
                                kSelThreads, smem, st, p));
  *done = true;
  return SPEC_OK;
}

int run_stream_topk(const spec_problem* pr, const float* scores, int c_max, int n_forced_tail, int32_t* idx_out,
                    int32_t* count_out, int n_vert, int32_t* vert_out, int32_t* vert_count_out, void* workspace,
                    size_t workspace_bytes, int32_t* status_word, cudaStream_t st, bool* done) {
  *done = false;
  const int64_t n_units = (int64_t)pr->n_seq * pr->n_layers * pr->n_kv_heads;
  StreamParams p = {};
  p.scores = scores; p.cu = pr->cu_seqlens; p.T = pr->total_tokens; p.n_in = pr->n_in;
  p.L = pr->n_layers; p.H = pr->n_kv_heads; p.n_forced = n_forced_tail; p.c_max = c_max; p.n_vert = n_vert;
  p.max_len = max_seq_len(pr);
  p.idx_out = idx_out; p.count_out = count_out; p.vert_out = vert_out; p.vert_count_out = vert_count_out;
  p.status = status_word;
  // Short units: one CTA does all of it, however many they are (256 units of 16384, a 7th kept, 15 us and 24 streamed; 592 of
  // 5000 19.9 and 31.2; 4096 of 1500, a 40th kept, 100 and 102; 16384 of 300 355 and 354).
  const int rc = run_unit_topk(pr, p, st, done);
  if (rc != SPEC_OK || *done) return rc;
  if (!workspace) return SPEC_OK;
  const WorkspacePlan wp = plan_workspace(pr);
  if (workspace_bytes < wp.total) return SPEC_OK;
  if (p.max_len < 1 || pr->n_layers * pr->n_kv_heads > 65535) return SPEC_OK;   // rows are a grid dimension of the sweep
  // One chunk per warp and one count per finishing thread: longer units take two rounds per warp.
  const int64_t per_round = (int64_t)kSelThreads * kWarpSpan;
  p.rounds = (int)(((int64_t)p.max_len + 3 + per_round - 1) / per_round);
  if (p.rounds * kWarpSpan > kSelChunkMax) return SPEC_OK;
  static_assert(kWarpSpan == kSelChunkMin, "the workspace has a count per kSelChunkMin positions");
  p.chunks_max = (int)(((int64_t)p.max_len + 3 + p.rounds * kWarpSpan - 1) / (p.rounds * kWarpSpan));
  const int largest = std::max(c_max, n_vert);
  const int64_t room = ((int64_t)kSmemLimit - 16 * 1024) / 8;
  p.held_cap = (int)(std::min<int64_t>(4 * (int64_t)largest + 4096, room) & ~(int64_t)3);
  if (p.held_cap < 2 * (int64_t)largest + 2048) return SPEC_OK;                 // too large a budget for the finishing CTA
  // The floor is about the rho-th of the samples, rho = m + 4 sqrt(m) + 8 and m = budget / rate, rate = 32 to 128 positions
  // per sample; a full bin lets r = 1.25 rho + 8 samples in at most.  With room for rate * (r + 5 sqrt(r) + 12) candidates a
  // unit overflows less than once in 10^7 (Poisson), and for 2048 of 131072 with 4 * budget + 4096 less than once in 10^5 (with
  // 3 * budget + 2048 one unit in 100 did, and one generic selection costs more than the other 255 units together).  Memory
  // beyond that only keeps a second CTA off the SM: 2048 units of 16384, 2730 kept, 214 us with 4 * budget + 4096, 153 so.
  const int rate = 1 << sample_shift(p.max_len, p.max_len + 7);
  const double m = (double)largest / rate, r = 1.25 * (m + 4.0 * std::sqrt(m) + 8.0) + 8.0;
  const int64_t enough = std::min<int64_t>((int64_t)(rate * (r + 5.0 * std::sqrt(r) + 12.0)), p.max_len);
  p.held_cap = (int)std::min<int64_t>(p.held_cap, (enough + 3) & ~(int64_t)3);
  uint8_t* ws = workspace_base(workspace);
  p.head = reinterpret_cast<int32_t*>(ws + wp.sel_head_off);
  p.head_words = wp.sel_head_words;
  p.cand = reinterpret_cast<uint2*>(ws + wp.sel_cand_off);
  p.row_entries = wp.sel_row_entries;

  typedef void (*FinishKernel)(const StreamParams);
  static const FinishKernel finish[4] = {stream_finish_kernel<2, false>, stream_finish_kernel<2, true>, stream_finish_kernel<3, false>, stream_finish_kernel<3, true>};
  static int set[64] = {0};
  int dev = 0;
  SPEC_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SPEC_OK;
  if (!__atomic_load_n(&set[dev], __ATOMIC_ACQUIRE)) {
    for (const FinishKernel f : finish) SPEC_CUDA_OK(cudaFuncSetAttribute((const void*)f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit - 16 * 1024));
    __atomic_store_n(&set[dev], 1, __ATOMIC_RELEASE);
  }
  SPEC_CUDA_OK(launch_dependent(sample_floor_kernel, dim3((unsigned)n_units), kSelThreads, 0, st, p));
  const dim3 sweep_grid((unsigned)((p.chunks_max + kSweepWarps - 1) / kSweepWarps), (unsigned)(pr->n_layers * pr->n_kv_heads), (unsigned)pr->n_seq);
  SPEC_CUDA_OK(launch_dependent(stream_sweep_kernel, sweep_grid, kSweepThreads, 0, st, p));
  const bool both = both_budgets(p, n_units);
  const bool three = n_units > 2 * sm_count() && held_bytes(p.held_cap) <= (size_t)(228 * 1024 / 3 - 14 * 1024);   // 13 KB and 1 KB beside them
  SPEC_CUDA_OK(launch_dependent(finish[2 * three + both], dim3((unsigned)n_units, n_vert > 0 && !both ? 2 : 1), kSelThreads, held_bytes(p.held_cap), st, p));
  *done = true;
  return SPEC_OK;
}

}  // namespace spec
