// Lookahead importance scoring (Eq. 1; Algorithm 1 lines 8-9) on tcgen05 tensor cores.
//
// score[j] = reduce_i softmax_j(scale * q_i . k_j) over the M = G*R query rows that share a
// KV head.  The M x n probability matrix never leaves the SM:
//   pass 1   S = Q K^T per 128-key tile (query rows on TMEM lanes): sum-exp over a
//            reference per row, kept per thread, written per (CTA, unit) segment;
//   pass 2   first combines the segments' statistics into one constant per row,
//            c_i = log2e*scale*m_i + log2 Z_i - log2 w_i; then S^T = K Q^T per tile (keys on TMEM lanes,
//            query rows on columns): p = exp2(scale*log2e*S - c_i), reduced over columns
//            thread-locally, one reduction per key and warpgroup.
// Both passes are persistent, warp-specialised kernels: warp 0 feeds K tiles (and the unit's Q)
// with TMA into a shared-memory ring, two warps issue tcgen05.mma into TMEM, and four epilogue
// warpgroups (16 warps, four per SM sub-partition) drain the accumulators with tcgen05.ld and
// do the exponentials.  Every warpgroup owns one 128-column TMEM buffer.  A work item is
// 128 x 128 logits: 128 query rows x the 128 keys of a tile in pass 1, the 128 keys of a tile x
// a chunk of 128 query rows in pass 2.  Key tiles alternate between the two pairs of
// warpgroups (each pair has its own issuing warp); within a pair the items of a tile
// alternate between its two warpgroups, which start alternately from tile to tile where that evens out their work.  A
// warpgroup drains an item whole, four 32-column loads with the arithmetic in between (two
// blocks in registers: the other roles give up registers for that), and hands the buffer back
// after the last load, so the four warps that share an SM sub-partition run out of step with one
// another.
// The exponential is the scarce resource (16 MUFU results per clock per SM against 32 logits per
// clock from the tensor cores), so a fixed share of the elements is evaluated on the FMA pipes
// instead (range reduction + quartic polynomial, relative error up to 5.3e-6), and the surrounding
// arithmetic uses the packed two-lane fp32 instructions to halve its issue slots.  Warpgroups
// never synchronise inside a unit: pass 1 writes their statistics as separate partials; in
// pass 2 a key tile belongs to one pair, whose two warpgroups add their per-key sums (over the
// chunks each of them drained) into the zero-filled output with one reduction each (two
// addends, so the result does not depend on their order).  More query rows than fit in shared
// memory are scored in several launches over groups of rows (ScoreParams::row0), each adding
// into the same output.
// The global key-tile space (layer, KV head, sequence, tile) is cut into equal contiguous
// ranges, one per CTA; units of one length, few to a GPU, are cut among CTAs of their own.
//
// What bounds it: long calls run at the board's power limit, so that their time is the energy of a logit (tensor
// core, TMEM read, two packed FMA-pipe operations, the exponential), whatever the clock: 32 layers of 131072 keys,
// 640 rows of head_dim 128, 12.32 -> 11.41 ms for the step in a loop, at 1582 MHz; of 16384 keys, 384 rows, at full
// clock 0.94 -> 0.865 ms.  Short calls are bound by the way into each pass: one layer of 12345 keys (36 us) waits 3.4 us
// for its queries and 1.5 for the first accumulators in pass 1, which ends at 18, and in pass 2 from 18 to 23.5 for the
// last CTA of pass 1, the statistics (2.5 us) and the constants.
//
// Every wait on an mbarrier is bounded in time; on expiry the CTA passes the named barriers that are left, without the
// items (kReturnBarrier), reports SPEC_ERR_TIMEOUT through the status word, lets its copies land, frees its TMEM and returns.
#include <cuda.h>

#include "common.cuh"
#include <algorithm>

namespace spec {

constexpr int kEpilogueWarpgroups = 4;
constexpr int kEpilogueThreads = kEpilogueWarpgroups * 128;
constexpr int kThreads = 128 + kEpilogueThreads;        // one more warpgroup: TMA producer, two MMA issuers, an idle warp
// Registers per thread: at launch (the most that five warps per SM sub-partition leave), and after the
// warpgroups have divided them; the epilogue needs two blocks of 32 accumulator columns at a time.
constexpr int kLaunchRegs = 96, kIssueRegs = 64, kEpilogueRegs = 104;
static_assert(128 * kIssueRegs + kEpilogueThreads * kEpilogueRegs <= kThreads * kLaunchRegs, "the warpgroups' shares must fit what the block is launched with");
// Of the 16 element pairs in a 32-element block, evaluated on the FMA pipes.  Sustained time of 8 layers at 128K
// (640 rows) for 2, 3, 4, 5 pairs: 3.120, 3.068, 3.033, 3.030 ms (6 was 2 % slower than 5).
constexpr int kPolyPairs = 5;
// minimax quartic of 2^f on [-1/2, 1/2], from the lowest coefficient
constexpr float kExpC0 = 0.9999992614f, kExpC1 = 0.6931218147f, kExpC2 = 0.2402474482f, kExpC3 = 0.0559178603f, kExpC4 = 0.0095701019f;
constexpr int kBufCols = 128;                 // TMEM columns of an accumulator buffer, one per epilogue warpgroup
constexpr int kTileKeys = 128;
constexpr int kMaxStages = 8;
constexpr int kMaxMTiles = 10;
constexpr int kNumBars = 2 * kMaxStages + 2 + 4;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
constexpr uint32_t kSuspendHintNs = 100000;

struct ScoreParams {
  const int32_t* cu;
  const float* row_weight;
  float* partial;       // [n_units + n_ctas][4 warpgroups][M][2]  (max in log2 domain, sum-exp)
  float* scores;        // [L, Hkv, T]
  int32_t* status;
  long long T;
  int n_in, n_seq, L, Hq, Hkv, G, R, M, M_pad, d;   // M, M_pad: the query rows of this launch, rows [row0, row0 + M) of every unit
  int row0;
  int pieces;            // CTAs per unit, each of which has a share of that unit only (0: equal shares of the whole tile space)
  int n_window;          // causal kernels: window row r sees keys up to position n - n_window + r only
  int merge_slots;       // threads that share the merging of a unit's statistics when there are fewer rows than threads (0: none do)
  int n_stages, n_chunks, cw_last;   // pass 2: chunks of 128 query rows, the last of cw_last (a multiple of 16)
  int n_full, rem_cols;  // pass 1: blocks of 128 query rows on lanes, and 16..48 remaining rows on columns (0: none)
  int turn;             // 1: the warpgroups of a pair begin a tile in turn, 0: the first always does
  float a;              // softmax_scale * log2(e)
  uint32_t q_bytes, stage_bytes;
};

// ------------------------------------------------------------------ PTX wrappers ------

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// A buffer's return from its warpgroup to the warp that issues into it: a named barrier, on which the four epilogue warps
// arrive and the issuing warp waits.  An mbarrier's arrivals and tests stand in one queue with the exponentials, and the issuing
// warp saw a buffer's return some 900 cycles late; where pass 2 has no exponentials (MAX), that is the time of its items.  With it,
// and with issuing warps that see their own pair's key tiles only, 8 layers of 16384, 260 rows of head_dim 64: MAX 137.2 -> 128.5 us,
// SUM 158.7 -> 155.0; 384 rows of head_dim 128: 187.9 -> 184.4 and 210.2 -> 209.2.
// A buffer has two such barriers, which its returns take in turn; the parity of their number is also that of the item's phase.  A
// barrier counts arrivals and does not know whose they are: an epilogue warp that has given up waiting for items goes on to
// the next return at once, and with one barrier, where the issuing warp has not taken the one before yet (it may be waiting
// for keys), that would count as its fifth arrival, and every phase from then on lack one, for good.  It waits at that next
// return, so it is never further ahead.
constexpr int kReturnBarrier = 6, kReturnThreads = 128 + 32;
static_assert(kReturnBarrier % 2 == 0 && kReturnBarrier + 2 * kEpilogueWarpgroups <= 16, "the low bit is the parity, and a CTA has sixteen barriers");
__device__ __forceinline__ void return_arrive(uint32_t ret) { asm volatile("bar.arrive %0, %1;" ::"r"(ret), "n"(kReturnThreads) : "memory"); }
__device__ __forceinline__ void return_sync(uint32_t ret) { asm volatile("bar.sync %0, %1;" ::"r"(ret), "n"(kReturnThreads) : "memory"); }
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait.  Returns false when another role has given up or the time limit passed.  The
// suspend-time hint lets the hardware park the thread until the phase completes instead of
// spinning in the issue slots the epilogue warps need.
__device__ __forceinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  const uint32_t addr = smem_u32(bar);
  unsigned long long t0 = 0;
  for (uint32_t it = 1;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(addr), "r"(parity), "r"(kSuspendHintNs) : "memory");
    if (ok) return true;
    if ((it & 7u) == 0) {                                   // every failed wait already lasted up to the hint
      if (*abort_flag) return false;
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
}

// The common case, a phase that has already completed, costs one non-blocking test inline.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_test(bar, parity) || mbar_wait_slow(bar, parity, abort_flag);
}
// The same for a whole warp: every lane gets the same answer, and the branches that depend on it do not
// diverge as far as the compiler can see.  The vote on the test comes before the slow path, not behind both: 16 layers of
// 32768, 512 rows of head_dim 64, 917 -> 900 us.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, abort_flag));
}
// True in exactly one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e != 0;
}
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}
// Key tiles give way first in L2: each is read once per pass, and what they would push out (the instructions and small
// buffers of the kernels that follow) comes from DRAM again otherwise: one layer of 64K, the selection 14 us later,
// 139 -> 131 us for the step; the keep set with the paper's settings 546 -> 538.
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  return policy;
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar)), "l"(policy) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulation, issued by one thread.
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}

// 32 (16) consecutive fp32 columns of this thread's TMEM lane; not to be read before tmem_wait.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// Waits for this thread's TMEM loads.  The registers of the load go through the statement, so that
// no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :: "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Shared-memory matrix descriptor: K-major operand, rows of 64 bf16 (128 bytes) with the
// 128-byte swizzle TMA writes; 8-row groups are 1024 bytes apart.  Only the start address
// (bits 0-13, in 16-byte units) differs between the operands of this kernel, so the issuing
// thread keeps the low word per operand and adds offsets to it; the high word is constant.
constexpr uint32_t kDescHi = (uint32_t)(1024 >> 4)        // stride byte offset between 8-row groups
                             | (1u << 14)                 // descriptor version of this architecture
                             | (2u << 29);                // 128-byte swizzle
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) {
  return ((saddr & 0x3FFFFu) >> 4) | (1u << 16);          // leading byte offset (unused for swizzled K-major)
}
__device__ __forceinline__ uint64_t desc_at(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128.
__device__ __forceinline__ uint32_t make_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// ------------------------------------------------------------- work decomposition -----

struct Seg {
  int unit;        // ordinal (layer*Hkv + head)*n_seq + seq
  int s, l, h;
  int begin, n;    // token range of the sequence
  int t0, nt;      // first key tile of the unit handled here, number of tiles
};

struct SegIter {
  long long g, g_end, per_cta, n_tiles;
  int TT, s;              // s: sequence of the last segment
  // Whether a unit that ends before tile `end` is the last one that CTA `cta` worked on.
  __device__ __forceinline__ bool last_segment(int cta, long long end) const {
    const long long range_end = (cta + 1) * per_cta;
    return end >= (range_end < n_tiles ? range_end : n_tiles);
  }
};

// Tile-count prefix over sequences, tp[0..n_seq].
__device__ void build_tile_prefix(const ScoreParams& p, int* tp) {
  int acc = 0;
  tp[0] = 0;
  for (int s = 0; s < p.n_seq; ++s) {
    int b, n;
    seq_range(p.cu, p.n_in, s, b, n);
    acc += (n + kTileKeys - 1) / kTileKeys;
    tp[s + 1] = acc;
  }
}

__device__ __forceinline__ SegIter seg_begin(const ScoreParams& p, const int* tp, int n_ctas, int cta) {
  SegIter it;
  it.TT = tp[p.n_seq];
  it.s = -2;                                               // none
  const long long N = (long long)p.L * p.Hkv * it.TT;
  it.n_tiles = N;
  if (p.pieces > 0) {                                      // every unit cut evenly among as many CTAs of its own
    const int unit = cta / p.pieces, i = cta - unit * p.pieces;
    const int base = it.TT / p.pieces, extra = it.TT - base * p.pieces;
    it.per_cta = 0;
    it.g = it.g_end = 0;
    if (unit < p.L * p.Hkv) {
      it.g = (long long)unit * it.TT + i * base + min(i, extra);
      it.g_end = it.g + base + (i < extra);
    }
    return it;
  }
  const long long P = (N + n_ctas - 1) / n_ctas;
  it.per_cta = P;
  it.g = P * cta;
  it.g_end = it.g + P < N ? it.g + P : N;
  return it;
}

// The next segment of the range: pass 1 goes through it forwards, pass 2 backwards, tile by tile, so that pass 2 begins
// with the keys that pass 1 has just left in L2 (one layer of 64K, 134 MB of keys: 118.6 -> 115.0 us).
template <int PASS, bool RAGGED>
__device__ bool seg_next(SegIter& it, const ScoreParams& p, const int* tp, Seg& sg) {
  if (it.g >= it.g_end) return false;
  const long long at = PASS == 1 ? it.g : it.g_end - 1;
  const int lh = (int)(at / it.TT);
  const int rem = (int)(at % it.TT);
  // the sequence that the tile belongs to, the last one with tp[lo] <= rem: as a rule the neighbour of the last segment's
  int lo = PASS == 1 ? it.s + 1 : it.s - 1, hi = p.n_seq;
  if (!RAGGED || lo < 0 || lo >= hi || tp[lo] > rem || tp[lo + 1] <= rem) {
    lo = 0;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (tp[mid] <= rem) lo = mid; else hi = mid;
    }
  }
  it.s = lo;
  sg.s = lo;
  sg.l = lh / p.Hkv;
  sg.h = lh % p.Hkv;
  sg.unit = lh * p.n_seq + lo;
  const long long left = it.g_end - it.g;
  const int in_unit = PASS == 1 ? tp[lo + 1] - rem : rem - tp[lo] + 1;
  sg.nt = left < in_unit ? (int)left : in_unit;
  sg.t0 = PASS == 1 ? rem - tp[lo] : rem - tp[lo] - sg.nt + 1;
  seq_range(p.cu, p.n_in, lo, sg.begin, sg.n);
  if (PASS == 1) it.g += sg.nt; else it.g_end -= sg.nt;
  return true;
}
// The t-th key tile of a segment in the pass's order.
template <int PASS>
__device__ __forceinline__ int seg_tile(const Seg& sg, int t) { return sg.t0 + (PASS == 1 ? t : sg.nt - 1 - t); }

// ------------------------------------------------------------------ epilogue math -----

// The packed fp32 instructions (two lanes per instruction) through the float2 intrinsics.
__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }

// 2^x for both lanes on the MUFU unit.
__device__ __forceinline__ float2 ex2_mufu2(float2 x) {
  return make_float2(ex2(x.x), ex2(x.y));
}
// 2^x for both lanes without the MUFU unit, x = s*a + c held in [-B, 128 - B]: in units of 128,
// y = (x + B) / 128 is one multiply-add that saturates to [0, 1] for nothing, so that neither end of the
// range needs a clamp of its own.  Adding 1.5 * 2^16 rounds y to a multiple of 1/128 and leaves
// n = round(128 y) in the low mantissa bits; 2^f of the rest, |f| <= 1/2, is a quartic, and n goes into the exponent
// field.  Relative error: 2.6e-6 of the quartic, and as much of the rounding of y to 2^-25, together up to 5.3e-6.  a128 = a / 128, c128 = (c + B) / 128.
template <int B>
__device__ __forceinline__ float2 ex2_poly2(float s0, float s1, float a128, float2 c128) {
  constexpr float k = B == 64 ? 5.421010862427522e-20f : 2.350988701644575e-38f;   // 2^-B
  static_assert(B == 64 || B == 125, "the scale of the coefficients");
  const float2 y = make_float2(__saturatef(fmaf(s0, a128, c128.x)), __saturatef(fmaf(s1, a128, c128.y)));
  const float2 yr = __fadd2_rn(y, splat2(98304.f));
  const float2 n = __fadd2_rn(yr, splat2(-98304.f));
  const float2 f = __fadd2_rn(y, make_float2(-n.x, -n.y));
  float2 q = __ffma2_rn(f, splat2(k * 268435456.f * kExpC4), splat2(k * 2097152.f * kExpC3));
  q = __ffma2_rn(q, f, splat2(k * 16384.f * kExpC2));
  q = __ffma2_rn(q, f, splat2(k * 128.f * kExpC1));
  q = __ffma2_rn(q, f, splat2(k * kExpC0));
  return make_float2(__uint_as_float(__float_as_uint(q.x) + (__float_as_uint(yr.x) << 23)),
                     __uint_as_float(__float_as_uint(q.y) + (__float_as_uint(yr.y) << 23)));
}
// Pair i (0..15) of a 32-element block: NP of them, evenly spread, avoid the MUFU unit.
template <int NP>
__host__ __device__ constexpr bool is_poly(int i) { return (i * NP) / 16 != ((i + 1) * NP) / 16; }

// Pass 1: fold logits of one row into the running statistics (m, z): z sums 2^(a*s - m).  m is not the
// running maximum but a reference, the maximum of the first block the row saw: fp32 holds sums of
// terms up to 2^62 above it and loses nothing below it that a sum of at least 1 would show, so
// the maximum (a third of an instruction per logit, and a chain in front of every exponential) is
// only taken again by the rare row whose block exceeds the reference by 2^62.
// The general form: only the first `valid` logits count, the reference becomes the maximum so far.
__device__ __forceinline__ void stats_general(const uint32_t (&r)[32], int valid, float a, float& m, float& z) {
  float g = -INFINITY;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i < valid) g = fmaxf(g, __uint_as_float(r[i]));
  const float mn = fmaxf(m, g * a);                        // a > 0
  if (!(mn > -INFINITY)) return;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (i < valid) s += ex2(fmaf(__uint_as_float(r[i]), a, -mn));
  z = z * ex2(m - mn) + s;                                 // first block: 0 * 2^-inf = 0
  m = mn;
}
// 32 logits that all count.
__device__ __forceinline__ void stats_update(const uint32_t (&r)[32], float a, float& m, float& z) {
  const float2 a2 = splat2(a), neg2 = splat2(-m);
  const float a128 = a * (1.f / 128.f);
  const float2 c128 = splat2(fmaf(m, -1.f / 128.f, 0.5f));
  float2 s0 = splat2(0.f), s1 = splat2(0.f);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float x0 = __uint_as_float(r[2 * i]), x1 = __uint_as_float(r[2 * i + 1]);
    const float2 e = is_poly<kPolyPairs>(i) ? ex2_poly2<64>(x0, x1, a128, c128) : ex2_mufu2(__ffma2_rn(make_float2(x0, x1), a2, neg2));
    if (i & 1) s1 = __fadd2_rn(s1, e); else s0 = __fadd2_rn(s0, e);
  }
  const float s = (s0.x + s0.y) + (s1.x + s1.y);
  if (s < 4.6e18f) z += s;                                 // 2^62; also false for the row's first block (m = -inf: infinite terms)
  else stats_general(r, 32, a, m, z);
}

// Pass 1, the rows that remain behind the last full block of 128: up to 48 of them would leave most lanes of
// a block idle, so they are scored the other way round, keys on lanes and rows on columns, and the
// sums over the lanes are taken by a butterfly that halves the columns at every step: lane l ends up
// with column l of a 32-column block (of 16 columns: l & 15).  With the butterfly a block of 32 costs
// about 0.4 of a block of 128 lanes, one of 16 about 0.2.
template <int COLS, bool MAX>
__device__ __forceinline__ float reduce_lanes(float (&e)[COLS], int lane) {
#pragma unroll
  for (int o = COLS / 2; o >= 1; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float got = __shfl_xor_sync(0xffffffffu, up ? e[i] : e[i + o], o);
      const float kept = up ? e[i + o] : e[i];
      e[i] = MAX ? fmaxf(kept, got) : kept + got;
    }
  }
  if (COLS == 16) {
    const float got = __shfl_xor_sync(0xffffffffu, e[0], 16);
    e[0] = MAX ? fmaxf(e[0], got) : e[0] + got;
  }
  return e[0];
}
// One block of a warp's remaining rows: z belongs to this lane's column, ref holds the references of the
// block's columns in the form that each column's exponential wants.  False, with nothing changed, when a sum
// is 2^62 above its reference or more (stats_update).
template <int COLS>
__device__ __forceinline__ bool rem_update(const uint32_t (&r)[32], float a, int lane, const float* ref, float& z) {
  const float a128 = a * (1.f / 128.f);
  const float2 a2 = splat2(a);
  const float4* c4 = reinterpret_cast<const float4*>(ref);
  float e[COLS];
#pragma unroll
  for (int i = 0; i < COLS / 2; ++i) {
    const float4 c = c4[i >> 1];
    const float2 cc = i & 1 ? make_float2(c.z, c.w) : make_float2(c.x, c.y);
    const float x0 = __uint_as_float(r[2 * i]), x1 = __uint_as_float(r[2 * i + 1]);
    const float2 v = is_poly<kPolyPairs>(i) ? ex2_poly2<64>(x0, x1, a128, cc) : ex2_mufu2(__ffma2_rn(make_float2(x0, x1), a2, cc));
    e[2 * i] = v.x;
    e[2 * i + 1] = v.y;
  }
  const float s = reduce_lanes<COLS, false>(e, lane);
  if (__any_sync(0xffffffffu, !(s < 4.6e18f))) return false;
  z += s;
  return true;
}
// The same for a block with keys that not every row sees, or rows without a reference: the columns of
// `visible` see this lane's key.  References become the maxima so far.
template <int COLS>
__device__ __noinline__ void rem_general(uint32_t taddr, uint32_t visible, float a, int lane, float* ref, float& m, float& z) {
  uint32_t r[32];
  if (COLS == 32) tmem_ld32(taddr, r); else tmem_ld16(taddr, r);
  tmem_wait(r);
  float v[COLS];
#pragma unroll
  for (int i = 0; i < COLS; ++i) v[i] = (visible >> i) & 1u ? __uint_as_float(r[i]) * a : -INFINITY;
  const float mn = fmaxf(m, reduce_lanes<COLS, true>(v, lane));
  if (mn > -INFINITY) z *= ex2(m - mn);
  m = mn;
  __syncwarp();                                            // the references are no longer read
  if (lane < COLS) ref[lane] = !(mn > -INFINITY) ? 0.f : is_poly<kPolyPairs>(lane >> 1) ? fmaf(mn, -1.f / 128.f, 0.5f) : -mn;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < COLS; ++i) {
    const float mi = __shfl_sync(0xffffffffu, mn, i);
    v[i] = (visible >> i) & 1u ? ex2(fmaf(__uint_as_float(r[i]), a, -mi)) : 0.f;
  }
  const float s = reduce_lanes<COLS, false>(v, lane);
  if (mn > -INFINITY) z += s;
}
template <int COLS>
__device__ __forceinline__ void rem_block(uint32_t taddr, bool general, uint32_t visible, float a, int lane, float* ref, float& m, float& z) {
  if (!general) {
    uint32_t r[32];
    if (COLS == 32) tmem_ld32(taddr, r); else tmem_ld16(taddr, r);
    tmem_wait(r);
    if (rem_update<COLS>(r, a, lane, ref, z)) return;
  }
  rem_general<COLS>(taddr, visible, a, lane, ref, m, z);
}

// Pass 2: COLS (16 or 32) query rows for this thread's key, reduced into acc.  SUM: two packed partial sums of the
// probabilities; the row constants come in the form that each column's exponential wants (row_const).
// MAX: four maxima of the exponents a*s - c_i, for the largest probability is the one with the largest
// exponent: one exponential per key, at the end, instead of one per logit (16 layers of 32768, 260 rows of
// head_dim 64: pass 2 284 -> 195 us; 8 layers of 32768, 640 rows of head_dim 128: 330 -> 245 us).
template <bool MAXRED>
__device__ __forceinline__ float row_const(int row, float negc) {
  return !MAXRED && is_poly<kPolyPairs>((row & 31) >> 1) ? (negc + 125.f) * (1.f / 128.f) : negc;
}
// hidden (MASKED): the columns that do not see this thread's key.
template <bool MAXRED, int COLS, bool MASKED = false>
__device__ __forceinline__ void prob_accumulate(const uint32_t (&r)[32], const float* __restrict__ rowc, float2 a2, float a128, float2 (&acc)[2],
                                                uint32_t hidden = 0) {
  const float4* c4 = reinterpret_cast<const float4*>(rowc);
#pragma unroll
  for (int i = 0; i < COLS / 4; ++i) {
    const float4 c = c4[i];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float x0 = __uint_as_float(r[4 * i + 2 * u]), x1 = __uint_as_float(r[4 * i + 2 * u + 1]);
      float2 cc = u == 0 ? make_float2(c.x, c.y) : make_float2(c.z, c.w);
      if (MASKED) {
        if ((hidden >> (4 * i + 2 * u)) & 1u) cc.x = -INFINITY;
        if ((hidden >> (4 * i + 2 * u + 1)) & 1u) cc.y = -INFINITY;
      }
      if (MAXRED) {
        const float2 x = __ffma2_rn(make_float2(x0, x1), a2, cc);
        float& m = i & 1 ? acc[u].y : acc[u].x;            // four chains, merged at the end
        m = fmax3(m, x.x, x.y);
      } else {
        const float2 e = is_poly<kPolyPairs>(2 * i + u) ? ex2_poly2<125>(x0, x1, a128, cc) : ex2_mufu2(__ffma2_rn(make_float2(x0, x1), a2, cc));
        acc[u] = __fadd2_rn(acc[u], e);
      }
    }
  }
}

// The columns from row0 on (bit i: row0 + i) that may not see key position `key` of a sequence of n: window row
// r < n_window does not when the key lies after the row's own position n - n_window + r, that is,
// when r < key - (n - n_window).
__device__ __forceinline__ uint32_t hidden_columns(int row0, int R, int n_window, int n, int key) {
  const int lim = key > 0 ? min(max(key - (n - n_window), 0), n_window) : 0;
  uint32_t hidden = 0;
  if (lim > 0) {
    for (int b = -(row0 % R); b < 32; b += R) {
      const int lo = max(b, 0), hi = min(b + lim, 32);       // columns lo .. hi - 1
      if (hi > lo) hidden |= (0xffffffffu >> (32 - (hi - lo))) << lo;
    }
  }
  return hidden;
}

// Combines the statistics that pass 1 left for a unit (`n` partials of M rows each: one from each of the n_last + 1 CTAs
// that worked on it, at every fourth place from `part`, or four from the last of them) into minus the softmax constant of every row, in
// shared memory.  Called by all epilogue threads.  Every CTA of pass 2 does this for each of its
// segments: a unit's partials are read from L2 by the few CTAs that share the unit, which takes
// about a microsecond, where a kernel of its own between the passes took 4 to 22 (one layer of 64K:
// 80 partials per row in a serial loop) plus two launch gaps.  When there are fewer rows than half
// the threads and more partials than a thread loads at once, several threads take a share of a row's partials each and
// meet in shared memory.  Short sequences have a few partials in hundreds of segments per CTA, where the meeting and 16
// exponentials for four partials cost more than all else (see RAGGED below).
__device__ __forceinline__ void fold_stats(float& m, float& z, float pm, float pz) {
  const float mn = fmaxf(m, pm);
  if (mn > -INFINITY) z = z * exp2f(m - mn) + pz * exp2f(pm - mn);
  m = mn;
}

constexpr int kMergeLoads = 16;       // in flight per thread; with 8, one layer of 12K (72 partials per row) spent 8 us here

template <bool MAXRED, bool RAGGED>
__device__ __forceinline__ void row_constants(const ScoreParams& p, const float2* __restrict__ part, int n_last, int n, int et, float scale_log2, float* c_sm, float2* merge_sm) {
  const int Mr = (p.M + 31) & ~31;
  const int slices = p.merge_slots > 0 && n > kMergeLoads ? p.merge_slots / Mr : 1;
  for (int i0 = 0; i0 < p.M_pad; i0 += kEpilogueThreads) {
    const int sl = slices > 1 ? et / Mr : 0;
    const int i = slices > 1 ? et - sl * Mr : i0 + et;
    float m = -INFINITY, z = 0.f;
    auto partial_at = [&](int c) { return __ldcg(part + (size_t)(min(c, n_last) * kEpilogueWarpgroups + max(c - n_last, 0)) * p.M + i); };
    if (RAGGED && n <= 4) {
      if (i < p.M) {
        float2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = u < n ? partial_at(u) : make_float2(-INFINITY, 0.f);
        m = fmaxf(fmaxf(v[0].x, v[1].x), fmaxf(v[2].x, v[3].x));
        if (m > -INFINITY) {
#pragma unroll
          for (int u = 0; u < 4; ++u) z += v[u].y * exp2f(v[u].x - m);
        }
      }
    } else if (i < p.M && sl < slices) {
      for (int c0 = sl; c0 < n; c0 += kMergeLoads * slices) {
        float2 v[kMergeLoads];
        float mx = m;
#pragma unroll
        for (int u = 0; u < kMergeLoads; ++u) {
          const int c = c0 + u * slices;
          v[u] = c < n ? partial_at(c) : make_float2(-INFINITY, 0.f);
        }
#pragma unroll
        for (int u = 0; u < kMergeLoads; ++u) mx = fmaxf(mx, v[u].x);
        if (mx > -INFINITY) {
          z *= exp2f(m - mx);
#pragma unroll
          for (int u = 0; u < kMergeLoads; ++u) z += v[u].y * exp2f(v[u].x - mx);
        }
        m = mx;
      }
    }
    if (slices > 1) {
      if (sl < slices) merge_sm[et] = make_float2(m, z);
      asm volatile("bar.sync 1, 512;" ::: "memory");
      if (et < p.M) {
        for (int s = 1; s < slices; ++s) {
          const float2 v = merge_sm[s * Mr + et];
          fold_stats(m, z, v.x, v.y);
        }
      }
    }
    if (sl == 0 && i < p.M_pad) {
      float c = -INFINITY;                                     // rows that pad the last tile weigh nothing
      if (i < p.M) {
        c = m + log2f(z);
        if (p.row_weight) c -= log2f(p.row_weight[(p.row0 + i) % p.R]) - scale_log2;
        c = -c;
      }
      c_sm[i] = row_const<MAXRED>(i, c);
    }
    if (slices > 1) {                                          // the padding rows beyond the slices' reach
      for (int j = Mr + et; j < p.M_pad; j += kEpilogueThreads) c_sm[j] = -INFINITY;
      break;
    }
  }
}

// ------------------------------------------------------------------ the kernel --------

// FLAG: pass 1, whether remaining rows are scored on columns (a variant of its own: the registers that it needs
// slowed the other one down by 4 to 20 %); pass 2, whether the reduction is the maximum.  CAUSAL: the causal window,
// likewise apart (its masks cost the other kernels 1 to 2 % in registers).  RAGGED: many sequences,
// dozens of segments to a CTA.  What a segment costs beside its tiles counts there (1024 sequences of 100 to 199 keys, 2
// layers of 8 heads, 32 rows: 925 us with the other kernels, 661 so; 128 sequences of 1000, 28 units to a CTA, 405 and 396),
// and the code for it cost one layer of 12345 keys 0.4 of 52.8 us, one of two sequences 1 of 27.
template <int PASS, bool FLAG, bool CAUSAL, bool RAGGED>
__global__ void __launch_bounds__(kThreads, 1)
score_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const ScoreParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr int BUFCOLS = kBufCols;
  constexpr bool REM = PASS == 1 && FLAG, MAXRED = PASS == 2 && FLAG;

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  uint8_t* k_sm = smem;
  uint8_t* q_sm = smem + (size_t)p.n_stages * p.stage_bytes;
  float* c_sm = reinterpret_cast<float*>(q_sm + p.q_bytes);
  float2* merge_sm = reinterpret_cast<float2*>(c_sm + p.M_pad);            // pass 2, units of few rows: see row_constants
  float* rem_sm = reinterpret_cast<float*>(merge_sm + p.merge_slots);      // pass 1: [16 warps][rem_cols] references, then as many sums
  int* tp = reinterpret_cast<int*>(rem_sm + (REM ? 2 * 16 * p.rem_cols : 0));
  uint64_t* bars = reinterpret_cast<uint64_t*>((reinterpret_cast<uintptr_t>(tp + p.n_seq + 1) + 7) & ~(uintptr_t)7);
  uint64_t* k_full = bars;
  uint64_t* k_empty = bars + kMaxStages;
  uint64_t* q_full = bars + 2 * kMaxStages;
  uint64_t* q_empty = q_full + 1;
  uint64_t* t_full = q_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* scale_sm = reinterpret_cast<float*>(tmem_slot + 2);

  if ((smem_u32(smem) & 1023u) != 0) {      // the swizzled tiles need 1024-byte alignment
    if (tid == 0) report(p.status, SPEC_ERR_ALIGNMENT);
    return;
  }
  if (tid == 0) {
    *abort_flag = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_q) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_k) : "memory");
  }
  // Every wait tells two phases of a key stage apart by their parity, so that a phase may be waited for only once the one before it
  // has completed.  With an even number of stages, a stage has tiles of one pair only within a segment, whose issuing warp takes
  // them all.  From one segment to the next pairs and stages may change places (a segment of an odd number of tiles); there
  // the producer's wait for q_empty keeps the phases apart: q_full of a segment is armed when both issuing warps have taken and
  // handed back all their tiles of the segment before.  With an odd number of stages, a stage has tiles of both pairs in turn, and both warps wait for
  // every tile and hand it back.
  const bool both_take = (p.n_stages & 1) != 0;
  if (tid == 32) {
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1 + both_take); }
    mbar_init(q_full, 1);
    mbar_init(q_empty, 2);
    for (int i = 0; i < 4; ++i) mbar_init(&t_full[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // Pass 1 may be launched while whatever fills its inputs still runs; pass 2 while pass 1 still does, but
  // every CTA of pass 1 is past its wait by then, so that only what pass 1 writes has to be waited for (below).
  if (PASS == 1) {
    wait_for_previous_grid();
    launch_dependents();
  }
  if (tid == 0) build_tile_prefix(p, tp);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = (uint32_t)uniform((int)*tmem_slot);
  const int n_kh = p.d / 64;                               // 64-element halves of the contraction
  const uint32_t q_half_bytes = (uint32_t)p.M_pad * 128u;
  // K ring: [64-element half of the contraction][stage][128 keys x 128 bytes]
  const uint32_t k_half_bytes = (uint32_t)p.n_stages * (128u * 128u);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
    if (warp == 0) {
      // ------------------------------------------------ TMA producer ----
      if (lane == 0) {
        SegIter it = seg_begin(p, tp, gridDim.x, blockIdx.x);
        Seg sg;
        const uint64_t policy = evict_first_policy();
        uint32_t kit = 0, nseg = 0;
        bool ok = true;
        while (ok && seg_next<PASS, RAGGED>(it, p, tp, sg)) {
          if (nseg > 0) ok = mbar_wait(q_empty, (nseg - 1) & 1, abort_flag);   // previous segment's MMAs retired, its key stages' phases complete (both_take)
          if (!ok) break;
          ++nseg;
          mbar_expect_tx(q_full, p.q_bytes);
          const int qrow0 = ((sg.s * p.L + sg.l) * p.Hq + sg.h * p.G) * p.R;
          for (int kh = 0; kh < n_kh; ++kh)
            for (int rb = 0; rb < p.M_pad / 128; ++rb)
              tma_load_2d(q_sm + kh * q_half_bytes + rb * (128 * 128), &tm_q, kh * 64, qrow0 + p.row0 + rb * 128, q_full);
          for (int t = 0; t < sg.nt; ++t, ++kit) {
            const int stage = kit % p.n_stages;
            const uint32_t par = (kit / p.n_stages) & 1;
            ok = mbar_wait(&k_empty[stage], par ^ 1, abort_flag);
            if (!ok) break;
            mbar_expect_tx(&k_full[stage], p.stage_bytes);
            uint8_t* dst = k_sm + (size_t)stage * (128 * 128);
            const int row = sg.begin + seg_tile<PASS>(sg, t) * kTileKeys;
            for (int kh = 0; kh < n_kh; ++kh)
              tma_load_4d(dst + kh * k_half_bytes, &tm_k, kh * 64, row, sg.h, sg.l, &k_full[stage], policy);
          }
        }
      }
    } else if (warp <= 2) {
      // ------------------------------------------------ MMA issuers -----
      // Two issuing warps, one per warpgroup pair: warp s feeds the buffers of that pair's two
      // warpgroups, and hands the pair's key tiles back.
      // The whole warp runs the loops, and one elected lane issues: in converged code the descriptors stay in
      // the uniform registers that tcgen05.mma reads them from.  Issued from a branch that one lane had
      // taken, the eight instructions of an item took 1400 cycles among the epilogue warps (512 on the
      // tensor pipe), and the epilogue waited for them; this form takes 1000 with the pipe shared by two.  A
      // single issuing warp for all four buffers was slower (32 layers at 16K: 1.02 against 0.98 ms).
      const int strm = warp - 1;
      SegIter it = seg_begin(p, tp, gridDim.x, blockIdx.x);
      Seg sg;
      uint32_t nseg = 0, kit = 0;                              // segments, key tiles of the segments before
      uint32_t ret[2] = {0, 0};                                // my pair's two buffers: the barrier of the next return (0: no item issued yet)
      bool ok = true;
      const uint32_t idesc_full = make_idesc(128);
      const uint32_t idesc_last = make_idesc(PASS == 2 ? p.cw_last : REM ? p.rem_cols : 128);
      const int n_sub = PASS == 1 ? p.n_full + REM : p.n_chunks;
      const uint32_t q_lo0 = desc_lo(smem_u32(q_sm)), k_lo0 = desc_lo(smem_u32(k_sm));
      const uint32_t q_half16 = q_half_bytes >> 4;
      const uint32_t k_half16 = k_half_bytes >> 4;
      const int t_first = both_take ? 0 : strm, t_step = both_take ? 1 : 2;
      // Every item passes its buffer's barrier, also after a wait has given up, so that no warp is left waiting there (kReturnBarrier).
      for (;;) {
        const bool more = seg_next<PASS, RAGGED>(it, p, tp, sg);
        const int nt = uniform(more ? sg.nt : 0);
        if (nt == 0) break;
        ok = ok && mbar_wait_warp(q_full, nseg & 1, abort_flag);
        ++nseg;
        tc_fence_after();
        // A key tile belongs to the pair with the parity of its index in the segment; within the
        // pair, sub-item `sub` (a block of 128 query rows) of the pair's k-th tile goes to the
        // warpgroup (sub + k * turn) & 1, whose private 128-column buffer receives it.
        int stage = (int)((kit + t_first) % p.n_stages);
        uint32_t k_par = ((kit + t_first) / p.n_stages) & 1;
        kit += nt;
        for (int t = t_first; t < nt; t += t_step) {
          ok = ok && mbar_wait_warp(&k_full[stage], k_par, abort_flag);
          tc_fence_after();
          const uint32_t k_lo = k_lo0 + stage * ((128 * 128) >> 4);
          if ((t & 1) == strm) {
            for (int sub = 0; sub < n_sub; ++sub) {
              const int h = (sub + (t >> 1) * p.turn) & 1;
              const int buf = strm * 2 + h;
              const uint32_t back = h ? ret[1] : ret[0];
              if (back) return_sync(back);
              const uint32_t next = back ? back ^ 1 : kReturnBarrier + 2 * buf;
              if (h) ret[1] = next; else ret[0] = next;
              tc_fence_after();
              const uint32_t d_tmem = tmem_base + buf * BUFCOLS;
              const uint32_t q_lo = q_lo0 + sub * ((128 * 128) >> 4);
              const uint32_t idesc = (PASS == 2 || REM) && sub == n_sub - 1 ? idesc_last : idesc_full;
              const bool rows_on_lanes = PASS == 1 && (!REM || sub < p.n_full);
              const uint32_t a_lo = rows_on_lanes ? q_lo : k_lo, a_half16 = rows_on_lanes ? q_half16 : k_half16;
              const uint32_t b_lo = rows_on_lanes ? k_lo : q_lo, b_half16 = rows_on_lanes ? k_half16 : q_half16;
              if (ok && elect_one()) {
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {
                  if (kh < n_kh) {
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                      tc_mma(d_tmem, desc_at(a_lo + kh * a_half16 + ks * 2), desc_at(b_lo + kh * b_half16 + ks * 2), idesc, (kh | ks) != 0);
                    }
                  }
                }
                tc_commit(&t_full[buf]);
              }
              __syncwarp();
            }
          }
          if (ok && elect_one()) tc_commit(&k_empty[stage]);        // arrives once my MMAs on this stage (if any) retire
          __syncwarp();
          stage += t_step;
          if (stage >= p.n_stages) { stage -= p.n_stages; k_par ^= 1; }
        }
        if (ok && elect_one()) tc_commit(q_empty);
        __syncwarp();
      }
      if (ret[0]) return_sync(ret[0]);                           // of the last items
      if (ret[1]) return_sync(ret[1]);
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpilogueRegs));
    // ------------------------------------------------ epilogue --------
    const int wg = (warp - 4) >> 2;                        // warpgroup 0..3
    const int pair = wg >> 1;                              // pairs take alternate key tiles
    const int half = wg & 1;                               // column half of the pair's buffer
    const int quarter = warp & 3;                          // TMEM lane quarter this warp may read
    const int row_in_tile = quarter * 32 + lane;
    const int et = tid - 128;                              // 0..511 among epilogue threads
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    SegIter it = seg_begin(p, tp, gridDim.x, blockIdx.x);
    Seg sg;
    bool ok = true;
    uint32_t ra[32], rb[32];
    uint32_t ret = kReturnBarrier + 2 * wg;                  // the barrier of my buffer's next return, whose parity is that of its next item
    const uint32_t my_taddr = lane_base + wg * BUFCOLS;
    if (PASS == 1) {
      // Work item = 128 query rows (on lanes) x the 128 keys of a tile, all of it mine.
      // The scores are zeroed here, tile by tile, for pass 2 to add into: tokens of a sequence by the CTA that has
      // their tile, tokens that no sequence covers by whole rows in turn.
      const bool clears = p.row0 == 0;
      if (clears) {
        const long long lo = p.cu ? p.cu[0] : 0, hi = p.cu ? p.cu[p.n_seq] : p.n_in;
        if (lo > 0 || hi < p.T) {
          for (int r = blockIdx.x; r < p.L * p.Hkv; r += gridDim.x) {
            float* row = p.scores + (long long)r * p.T;
            for (long long j = et; j < lo; j += kEpilogueThreads) row[j] = 0.f;
            for (long long j = hi + et; j < p.T; j += kEpilogueThreads) row[j] = 0.f;
          }
        }
      }
      const int n_full = p.n_full, n_sub = n_full + REM;
      float mrun[kMaxMTiles], zrun[kMaxMTiles];
      float* my_ref = rem_sm + (warp - 4) * p.rem_cols;
      // Every epilogue thread passes the barriers of every segment, also after a wait has given up.
      while (seg_next<PASS, RAGGED>(it, p, tp, sg)) {
        float rem_m[2] = {-INFINITY, -INFINITY}, rem_z[2] = {0.f, 0.f};
        float* out = p.scores + ((long long)sg.l * p.Hkv + sg.h) * p.T + sg.begin;
#pragma unroll
        for (int i = 0; i < kMaxMTiles; ++i) { mrun[i] = -INFINITY; zrun[i] = 0.f; }
        for (int t = pair; t < sg.nt; t += 2) {
          const int key0 = seg_tile<PASS>(sg, t) * kTileKeys;                                // first key of the tile
          const int nv = min(kTileKeys, sg.n - key0);                              // valid keys of the tile
          const bool in_window = CAUSAL && key0 + kTileKeys > sg.n - p.n_window;    // warp-uniform
          const bool plain = nv >= kTileKeys && !in_window;
          if (clears && half == 0 && row_in_tile < nv) out[key0 + row_in_tile] = 0.f;
          for (int mt = ((t >> 1) * p.turn + half) & 1; mt < n_sub; mt += 2) {
            ok = ok && mbar_wait_warp(&t_full[wg], ret & 1, abort_flag);
            if (!ok) { return_sync(ret); ret ^= 1; continue; }
            ret ^= 1;                                           // the item's own is now ret ^ 1
            tc_fence_after();
            if (REM && mt == n_full) {
              // the remaining rows, on columns; this lane's key is key0 + row_in_tile
              const int cols = p.rem_cols;
              // warp-uniform: not every key is seen by every row, or a row has not seen any key yet
              const bool general = !plain || !__all_sync(0xffffffffu, rem_m[0] > -INFINITY && (cols <= 32 || rem_m[1] > -INFINITY));
              uint32_t seen = row_in_tile < nv ? 0xffffffffu : 0u, seen1 = seen;
              if (in_window) {
                int rr = (p.row0 + n_full * 128) % p.R;
#pragma unroll 1
                for (int i = 0; i < cols; ++i) {
                  if (rr < p.n_window && key0 + row_in_tile > max(sg.n - p.n_window + rr, 0)) {
                    if (i < 32) seen &= ~(1u << i); else seen1 &= ~(1u << (i - 32));
                  }
                  if (++rr == p.R) rr = 0;
                }
              }
              if (cols >= 32) rem_block<32>(my_taddr, general, seen, p.a, lane, my_ref, rem_m[0], rem_z[0]);
              else rem_block<16>(my_taddr, general, seen, p.a, lane, my_ref, rem_m[0], rem_z[0]);
              if (cols > 32) rem_block<16>(my_taddr + 32, general, seen1, p.a, lane, my_ref + 32, rem_m[1], rem_z[1]);
              __syncwarp();
              tc_fence_before();
              return_arrive(ret ^ 1);
              continue;
            }
            float m = mrun[mt], z = zrun[mt];
            if (plain) {
              // Every row sees all 128 keys: no masks, no per-row arithmetic.  The next block of columns is on its way
              // while one is worked on; the last two are both in registers when the buffer is given
              // back, whose refill takes about as long as their arithmetic.
              tmem_ld32(my_taddr, ra);
              tmem_wait(ra);
              tmem_ld32(my_taddr + 32, rb);
              stats_update(ra, p.a, m, z);
              tmem_wait(rb);
              tmem_ld32(my_taddr + 64, ra);
              stats_update(rb, p.a, m, z);
              tmem_ld32(my_taddr + 96, rb);
              tmem_wait(ra);
              tmem_wait(rb);
              tc_fence_before();
              return_arrive(ret ^ 1);
              stats_update(ra, p.a, m, z);
              stats_update(rb, p.a, m, z);
            } else {
              int vis = nv;                                    // keys of the tile that this thread's row may see
              if (in_window) {
                const int rr = (p.row0 + mt * 128 + row_in_tile) % p.R;
                if (rr < p.n_window) vis = min(nv, max(sg.n - p.n_window + rr, 0) + 1 - key0);
              }
#pragma unroll 1
              for (int c = 0; c < 4; ++c) {
                if (c * 32 >= nv) break;                                    // warp-uniform
                tmem_ld32(my_taddr + c * 32, ra);
                tmem_wait(ra);
                if (__all_sync(0xffffffffu, vis - c * 32 >= 32)) stats_update(ra, p.a, m, z);
                else if (vis - c * 32 > 0) stats_general(ra, min(vis - c * 32, 32), p.a, m, z);
              }
              __syncwarp();
              tc_fence_before();
              return_arrive(ret ^ 1);
            }
            mrun[mt] = m;
            zrun[mt] = z;
          }
        }
        // The statistics of a CTA's last segment are combined here, in the memory of the key ring, which nobody reads any
        // more once every warpgroup has seen its last accumulator; those of the segments before it go out per
        // warpgroup.  In a short call every segment is a last one, and pass 2 has a quarter of the partials
        // to read (one layer of 12K: 72 -> 21 per row, spec_score 43.4 -> 39.1 us).
        const bool last = it.g >= it.g_end;
        float2* part = reinterpret_cast<float2*>(p.partial) + (size_t)(sg.unit + blockIdx.x) * kEpilogueWarpgroups * p.M;
        float2* mine = (last ? reinterpret_cast<float2*>(k_sm) : part) + (size_t)wg * p.M;
        if (last) asm volatile("bar.sync 1, 512;" ::: "memory");
        if (ok) {
          for (int mt = 0; mt < n_full; ++mt) {
            const int row = mt * 128 + row_in_tile;
            if (row < p.M) mine[row] = make_float2(mrun[mt], zrun[mt]);
          }
        }
        if (REM) {
          // the four warps of the warpgroup saw different keys: their (reference, sum) meet in shared memory
          float* sums = rem_sm + 16 * p.rem_cols;
          const int b1 = p.rem_cols - 32;                       // columns of the second block, if positive
          if (lane < min(p.rem_cols, 32)) { my_ref[lane] = rem_m[0]; sums[(warp - 4) * p.rem_cols + lane] = rem_z[0]; }
          if (lane < b1) { my_ref[32 + lane] = rem_m[1]; sums[(warp - 4) * p.rem_cols + 32 + lane] = rem_z[1]; }
          asm volatile("bar.sync %0, 128;" ::"r"(2 + wg) : "memory");
          const int row = n_full * 128 + row_in_tile;
          if (row_in_tile < p.rem_cols && row < p.M && ok) {
            float m = -INFINITY, z = 0.f;
            for (int w = 0; w < 4; ++w) {
              const int o = (wg * 4 + w) * p.rem_cols + row_in_tile;
              fold_stats(m, z, rem_sm[o], sums[o]);
            }
            mine[row] = make_float2(m, z);
          }
          asm volatile("bar.sync %0, 128;" ::"r"(2 + wg) : "memory");
        }
        if (last) {
          asm volatile("bar.sync 1, 512;" ::: "memory");
          const float2* of = reinterpret_cast<const float2*>(k_sm);
          for (int row = et; row < p.M && ok; row += kEpilogueThreads) {
            float2 v = of[row];
#pragma unroll
            for (int w = 1; w < kEpilogueWarpgroups; ++w) fold_stats(v.x, v.y, of[(size_t)w * p.M + row].x, of[(size_t)w * p.M + row].y);
            part[row] = v;
          }
        }
      }
    } else {
      // Work item = one key tile (keys on lanes) x one chunk of 128 query rows, all of it mine; the
      // chunks of a tile alternate between the two warpgroups of the pair.
      const float2 a2 = splat2(p.a);
      const float a128 = p.a * (1.f / 128.f);
      const long long per_cta = it.per_cta;
      // Weighted probabilities above 8 would leave the range of the polynomial exponential: with larger weights
      // everything is scaled down by a power of two, and the scores up again as they are written.
      float scale_log2 = 0.f;
      if (!MAXRED && p.row_weight) {
        float w = 0.f;
        for (int i = lane; i < p.R; i += 32) w = fmaxf(w, __ldg(p.row_weight + i));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w = fmaxf(w, __shfl_xor_sync(0xffffffffu, w, o));
        scale_log2 = fminf(fmaxf(floorf(log2f(w)) - 1.f, 0.f), 126.f);
      }
      if (et == 0) *scale_sm = exp2f(scale_log2);               // read after the barriers below
      bool waited = false;
      // Every epilogue thread passes the barriers of every segment, also after a wait has
      // given up, so that no warp is left waiting at them.
      while (seg_next<PASS, RAGGED>(it, p, tp, sg)) {
        // the CTAs of pass 1 that worked on this unit: its tiles are u0 .. u0 + n_tiles - 1 of the global tile space
        int b0 = sg.unit * p.pieces, b1 = b0 + p.pieces - 1, n_part = p.pieces;
        if (p.pieces == 0) {
          const long long u0 = (long long)(sg.l * p.Hkv + sg.h) * it.TT + tp[sg.s];
          const int n_tiles = tp[sg.s + 1] - tp[sg.s];
          b0 = b1 = (int)blockIdx.x;
          if (sg.nt < n_tiles) {                                // other CTAs had a part of it, too
            b0 = (int)(u0 / per_cta);
            b1 = (int)((u0 + n_tiles - 1) / per_cta);
          }
          n_part = b1 - b0 + (it.last_segment(b1, u0 + n_tiles) ? 1 : kEpilogueWarpgroups);
        }
        if (!waited) {
          waited = true;
          wait_for_previous_grid();                             // pass 1: statistics and zeroed scores
          launch_dependents();
        }
        asm volatile("bar.sync 1, 512;" ::: "memory");          // previous unit's constants no longer read
        row_constants<MAXRED, RAGGED>(p, reinterpret_cast<const float2*>(p.partial) + (size_t)(sg.unit + b0) * kEpilogueWarpgroups * p.M,
                              b1 - b0, n_part, et, scale_log2, c_sm, merge_sm);
        asm volatile("bar.sync 1, 512;" ::: "memory");
        float* out = p.scores + ((long long)sg.l * p.Hkv + sg.h) * p.T + sg.begin;
        for (int t = pair; t < sg.nt; t += 2) {
          float2 acc[2] = {splat2(MAXRED ? -INFINITY : 0.f), splat2(MAXRED ? -INFINITY : 0.f)};
          const int key = seg_tile<PASS>(sg, t) * kTileKeys + row_in_tile;
          const bool in_window = CAUSAL && (seg_tile<PASS>(sg, t) + 1) * kTileKeys > sg.n - p.n_window;   // warp-uniform
          bool any = false;
          for (int ch = ((t >> 1) * p.turn + half) & 1; ch < p.n_chunks; ch += 2) {
            // causal: the vote behind both, without which these kernels spill (one layer of 12345 keys 34.9 and 34.6 us)
            ok = ok && (CAUSAL ? __all_sync(0xffffffffu, mbar_wait(&t_full[wg], ret & 1, abort_flag)) : mbar_wait_warp(&t_full[wg], ret & 1, abort_flag));
            if (!ok) { return_sync(ret); ret ^= 1; continue; }
            ret ^= 1;                                           // the item's own is now ret ^ 1
            any = true;
            tc_fence_after();
            const int cw = ch == p.n_chunks - 1 ? p.cw_last : 128;            // my columns
            const float* rowc = c_sm + ch * 128;
            const int row0 = p.row0 + ch * 128;                 // query row of my first column
            if (in_window) {
#pragma unroll 1
              for (int c = 0; c < cw; c += 32) {
                const uint32_t hidden = hidden_columns(row0 + c, p.R, p.n_window, sg.n, key);
                if (c + 32 <= cw) {
                  tmem_ld32(my_taddr + c, ra);
                  tmem_wait(ra);
                  prob_accumulate<MAXRED, 32, true>(ra, rowc + c, a2, a128, acc, hidden);
                } else {
                  tmem_ld16(my_taddr + c, ra);
                  tmem_wait(ra);
                  prob_accumulate<MAXRED, 16, true>(ra, rowc + c, a2, a128, acc, hidden);
                }
              }
              __syncwarp();
              tc_fence_before();
              return_arrive(ret ^ 1);
              continue;
            }
            if (cw == 128) {                                    // look-ahead as in pass 1
              tmem_ld32(my_taddr, ra);
              tmem_wait(ra);
              tmem_ld32(my_taddr + 32, rb);
              prob_accumulate<MAXRED, 32>(ra, rowc, a2, a128, acc);
              tmem_wait(rb);
              tmem_ld32(my_taddr + 64, ra);
              prob_accumulate<MAXRED, 32>(rb, rowc + 32, a2, a128, acc);
              tmem_ld32(my_taddr + 96, rb);
              tmem_wait(ra);
              tmem_wait(rb);
              tc_fence_before();
              return_arrive(ret ^ 1);
              prob_accumulate<MAXRED, 32>(ra, rowc + 64, a2, a128, acc);
              prob_accumulate<MAXRED, 32>(rb, rowc + 96, a2, a128, acc);
            } else {
              // a last chunk of 16 to 112 rows, the odd half block first
              const int n32 = cw >> 5;
              if (cw & 16) {
                tmem_ld16(my_taddr + n32 * 32, rb);
                tmem_wait(rb);
                if (n32 == 0) { tc_fence_before(); return_arrive(ret ^ 1); }
                prob_accumulate<MAXRED, 16>(rb, rowc + n32 * 32, a2, a128, acc);
              }
#pragma unroll 1
              for (int c = 0; c < n32; ++c) {
                tmem_ld32(my_taddr + c * 32, ra);
                tmem_wait(ra);
                if (c == n32 - 1) { tc_fence_before(); return_arrive(ret ^ 1); }
                prob_accumulate<MAXRED, 32>(ra, rowc + c * 32, a2, a128, acc);
              }
            }
          }
          if (ok && any && key < sg.n) {
            // The output was zero-filled; the two warpgroups of the pair contribute once per key.
            const float v0 = acc[0].x, v1 = acc[0].y, v2 = acc[1].x, v3 = acc[1].y;
            if (MAXRED) {
              const float v = ex2(fmaxf(fmaxf(v0, v1), fmaxf(v2, v3)));
              asm volatile("red.global.max.u32 [%0], %1;" ::"l"(out + key), "r"(__float_as_uint(v)) : "memory");
            } else {
              const float v = ((v0 + v1) + (v2 + v3)) * *scale_sm;
              asm volatile("red.global.add.f32 [%0], %1;" ::"l"(out + key), "f"(v) : "memory");
            }
          }
        }
      }
      if (!waited) {                                            // nothing to do: the grid still ends after the one before it
        wait_for_previous_grid();
        launch_dependents();
      }
    }
  }

  if (*abort_flag) {
    if (tid == 0) report(p.status, SPEC_ERR_TIMEOUT);
    __nanosleep(200000);                                     // let copies already in flight land
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
}

// ------------------------------------------------------------------ host side ---------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qr) == cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// The tensor map of a bf16 array.  A driver call, which wants a context on the calling thread; the runtime binds one where it
// needs it itself, and on a thread whose first call this is it has not yet.
static CUresult encode_map(EncodeTiledFn encode, CUtensorMap* map, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                           const cuuint32_t* box) {
  const cuuint32_t es[4] = {1, 1, 1, 1};
  auto call = [&]() {
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = call();
  int dev = 0;
  if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = call();
  return r;
}

}  // namespace spec

SPEC_EXPORT int32_t spec_score(const spec_problem* pr, const void* q, const void* k, const float* row_weight,
                               int32_t reduce, int32_t causal_window, float* scores_out, void* workspace,
                               size_t workspace_bytes, int32_t* status_word, void* stream) {
  using namespace spec;
  int rc = check_problem(pr);
  if (rc != SPEC_OK) return rc;
  if (!q || !k || !scores_out) return fail(SPEC_ERR_BAD_ARG, "q, k and scores_out must not be NULL");
  if (reduce != SPEC_REDUCE_SUM && reduce != SPEC_REDUCE_MAX) return fail(SPEC_ERR_BAD_ARG, "reduce=%d is not a spec_reduce value", reduce);
  if (causal_window != 0 && causal_window != 1) return fail(SPEC_ERR_BAD_ARG, "causal_window=%d must be 0 or 1", causal_window);
  if (!(pr->softmax_scale > 0.f) || !(pr->softmax_scale < 1e30f)) return fail(SPEC_ERR_BAD_ARG, "softmax_scale must be positive and finite");
  if (!aligned16(q) || !aligned16(k)) return fail(SPEC_ERR_ALIGNMENT, "q and k must be 16-byte aligned");
  const int d = pr->head_dim;
  if (pr->k_stride_token < d || pr->k_stride_head < d || pr->k_stride_layer < d ||
      (pr->k_stride_token * 2) % 16 || (pr->k_stride_head * 2) % 16 || (pr->k_stride_layer * 2) % 16)
    return fail(SPEC_ERR_ALIGNMENT, "K strides must be multiples of 8 elements and at least head_dim");
  const int R = pr->n_lookahead + pr->n_window;
  const int G = pr->n_q_heads / pr->n_kv_heads;
  const int M = G * R;
  // The query rows of a unit stay resident in shared memory, in blocks of 128, beside two key stages and what grows with
  // them and with the number of sequences (from 78 sequences on, 512 instead of 640 rows of head_dim 128); more than fit
  // are scored in several launches over groups of as many blocks as the largest needs, whose contributions add up in scores_out.
  const int smem_max = 227 * 1024;
  auto small_bytes = [&](int rows) {                       // all but queries and keys
    const int Mr = (rows + 31) & ~31, rows_pad = (rows + 127) / 128 * 128;
    const int slots = 2 * Mr <= kEpilogueThreads ? kEpilogueThreads / Mr * Mr : 0;
    return rows_pad * 4 + slots * 8 + (pr->n_seq + 1) * 4 + 8 + kNumBars * 8 + 16;
  };
  int rows_max = std::min(81920 / d, kMaxMTiles * 128) / 128 * 128;
  while (rows_max > 128 && rows_max * d * 2 + 2 * kTileKeys * d * 2 + small_bytes(rows_max) > smem_max) rows_max -= 128;
  const int n_groups = (M + rows_max - 1) / rows_max;
  const int rows_group = ((M + n_groups - 1) / n_groups + 127) / 128 * 128;
  const WorkspacePlan wp = plan_workspace(pr);
  if (!workspace || workspace_bytes < wp.total)
    return fail(SPEC_ERR_WORKSPACE, "workspace of %zu bytes given, %zu needed", workspace_bytes, wp.total);
  rc = check_device();
  if (rc != SPEC_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t tokens = pr->cu_seqlens ? pr->total_tokens : pr->n_in;
  if (tokens == 0) {                                       // nothing to score: the whole output reads as 0
    const size_t out_bytes = (size_t)pr->n_layers * pr->n_kv_heads * (size_t)pr->total_tokens * sizeof(float);
    if (out_bytes) SPEC_CUDA_OK(cudaMemsetAsync(scores_out, 0, out_bytes, st));
    return SPEC_OK;
  }

  EncodeTiledFn encode = encode_fn();
  if (!encode) return fail(SPEC_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");

  CUtensorMap tm_q, tm_k;
  {
    const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)pr->n_seq * pr->n_layers * pr->n_q_heads * R};
    const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
    const cuuint32_t box[2] = {64, 128};
    const CUresult r = encode_map(encode, &tm_q, q, 2, dims, strides, box);
    if (r != CUDA_SUCCESS) return fail(SPEC_ERR_CUDA, "tensor map for q could not be encoded (CUresult %d)", (int)r);
  }
  {
    const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)pr->total_tokens, (cuuint64_t)pr->n_kv_heads, (cuuint64_t)pr->n_layers};
    const cuuint64_t strides[3] = {(cuuint64_t)pr->k_stride_token * 2, (cuuint64_t)pr->k_stride_head * 2, (cuuint64_t)pr->k_stride_layer * 2};
    const cuuint32_t box[4] = {64, 128, 1, 1};
    const CUresult r = encode_map(encode, &tm_k, k, 4, dims, strides, box);
    if (r != CUDA_SUCCESS) return fail(SPEC_ERR_CUDA, "tensor map for k could not be encoded (CUresult %d)", (int)r);
  }

  ScoreParams p;
  p.cu = pr->cu_seqlens;
  p.row_weight = row_weight;
  uint8_t* ws = workspace_base(workspace);
  p.partial = reinterpret_cast<float*>(ws + wp.partial_off);
  p.scores = scores_out;
  p.status = status_word;
  p.T = pr->total_tokens;
  p.n_in = pr->n_in; p.n_seq = pr->n_seq; p.L = pr->n_layers; p.Hq = pr->n_q_heads; p.Hkv = pr->n_kv_heads;
  p.G = G; p.R = R; p.d = d;
  p.n_window = pr->n_window;
  p.a = (float)((double)pr->softmax_scale * 1.4426950408889634);
  p.stage_bytes = (uint32_t)kTileKeys * d * 2;

  const int n_ctas = wp.score_ctas;
  typedef void (*ScoreKernel)(const CUtensorMap, const CUtensorMap, const ScoreParams);
  static const ScoreKernel kernels[2][2][2][2] = {          // [ragged][pass][flag][causal]
      {{{score_kernel<1, false, false, false>, score_kernel<1, false, true, false>}, {score_kernel<1, true, false, false>, score_kernel<1, true, true, false>}},
       {{score_kernel<2, false, false, false>, score_kernel<2, false, true, false>}, {score_kernel<2, true, false, false>, score_kernel<2, true, true, false>}}},
      {{{score_kernel<1, false, false, true>, score_kernel<1, false, true, true>}, {score_kernel<1, true, false, true>, score_kernel<1, true, true, true>}},
       {{score_kernel<2, false, false, true>, score_kernel<2, false, true, true>}, {score_kernel<2, true, false, true>, score_kernel<2, true, true, true>}}}};
  const bool ragged = pr->n_seq > 1 && (int64_t)pr->n_seq * pr->n_layers * pr->n_kv_heads > 16 * (int64_t)n_ctas;
  // The kernels may use all of an SM's shared memory; the attribute is set once per device (it is per
  // function and context, so setting it per call would race between host threads).
  {
    static int set[64] = {0};
    int dev = 0;
    SPEC_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(SPEC_ERR_UNSUPPORTED, "device ordinal %d is not supported", dev);
    if (!__atomic_load_n(&set[dev], __ATOMIC_ACQUIRE)) {
      for (int i = 0; i < 16; ++i) {
        const void* f = (const void*)kernels[i >> 3][(i >> 2) & 1][(i >> 1) & 1][i & 1];
        SPEC_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        // The warpgroups divide the registers that the block was launched with: a build that launches with fewer
        // would wait for registers that do not exist.
        cudaFuncAttributes at;
        SPEC_CUDA_OK(cudaFuncGetAttributes(&at, f));
        if (at.numRegs < kLaunchRegs) return fail(SPEC_ERR_UNSUPPORTED, "the scoring kernel was built with %d registers per thread, %d needed", at.numRegs, kLaunchRegs);
      }
      __atomic_store_n(&set[dev], 1, __ATOMIC_RELEASE);
    }
  }
  // A CTA whose share spans two units pays for a second set of queries and constants (5 us of a short call), so units
  // of one length, few to a GPU, are cut each among CTAs of its own, if that costs no CTA more than two tiles.
  p.pieces = 0;
  if (!pr->cu_seqlens) {
    const int64_t units = (int64_t)pr->n_layers * pr->n_kv_heads, tiles_unit = (pr->n_in + kTileKeys - 1) / kTileKeys;
    const int64_t pieces = std::min(n_ctas / units, tiles_unit);
    if (pieces >= 2 && (tiles_unit + pieces - 1) / pieces <= (units * tiles_unit + n_ctas - 1) / n_ctas + 2) p.pieces = (int)pieces;
  }
  for (int g = 0; g < n_groups; ++g) {
    p.row0 = g * rows_group;
    p.M = std::min(rows_group, M - p.row0);
    p.M_pad = (p.M + 127) / 128 * 128;
    p.n_chunks = (p.M + 127) / 128;
    p.cw_last = (p.M - (p.n_chunks - 1) * 128 + 15) / 16 * 16;
    p.q_bytes = (uint32_t)p.M_pad * d * 2;
    const int Mr = (p.M + 31) & ~31;
    p.merge_slots = 2 * Mr <= kEpilogueThreads ? kEpilogueThreads / Mr * Mr : 0;
    const int small = small_bytes(p.M);
    int stages = std::min((smem_max - (int)p.q_bytes - small) / (int)p.stage_bytes, kMaxStages);
    // Up to 48 rows behind the last full block are scored on columns, from as many key tiles per CTA on as that needs: the first
    // tile of a segment, which sets the references, takes the general form, and a block of columns costs more the wider it
    // is.  Blocks of rows against columns (128 units of head_dim 64, us): 8 rows 22.3 and 21.7 at 8 tiles, 58 and 51 at 48;
    // 136 rows 39.4 and 41.0 at 12, 60 and 58 at 24; 152 rows 62 and 67 at 24, 107 and 104 at 48; 168 rows 107 and 119 at 48,
    // 212 and 208 at 96.  Not where the memory for it would leave fewer than three key stages.
    p.n_full = p.M_pad / 128;
    // An odd number of items to a tile, or a short last one, evens out over the tiles when the warpgroups begin in turn. With an even
    // number of equal items that gives a warpgroup two items in a row, for which its one buffer makes it wait: 8 layers of
    // 32768, SUM, in turns and without: head_dim 128, 256 rows 308 and 295 us, 512 rows 546 and 527 (of head_dim 64 475 and 472); odd
    // numbers: 128 rows 181 and 199, 352 rows 399 and 412, 640 rows 651 and 657.  The line lies at full blocks.  An even number with a
    // short last one is left in turns, although many of these do better without: 160 rows 238 and 235, 192 rows 281 and 272,
    // 240 rows 314 and 288, 496 rows 545 and 521; of head_dim 64, 160 rows 193 and 199, 192 rows 229 and 232, 240 rows 252 and 249.
    p.turn = p.M % 128 != 0 || p.n_full % 2 != 0;
    p.rem_cols = 0;
    int rem_bytes = 0;
    const int rem_cols = (p.M % 128 + 15) / 16 * 16;
    const int64_t tiles = (int64_t)pr->n_layers * pr->n_kv_heads * ((tokens + kTileKeys - 1) / kTileKeys);
    const int min_tiles = rem_cols == 16 ? (p.M < 128 ? 0 : 16) : rem_cols == 32 ? 32 : 96;
    if (rem_cols >= 16 && rem_cols <= 48 && tiles >= (int64_t)min_tiles * n_ctas) {
      const int bytes = 2 * 16 * rem_cols * 4;
      const int left = std::min((smem_max - (int)p.q_bytes - small - bytes) / (int)p.stage_bytes, kMaxStages);
      if (left >= std::min(stages, 3)) {
        stages = left;
        rem_bytes = bytes;
        p.n_full = p.M / 128;
        p.rem_cols = rem_cols;
      }
    }
    if (stages < 2) return fail(SPEC_ERR_UNSUPPORTED, "not enough shared memory for two key stages (%d rows, head_dim=%d)", p.M, d);
    p.n_stages = stages;
    int smem = stages * (int)p.stage_bytes + (int)p.q_bytes + small + rem_bytes;
    if (smem < 120 * 1024) smem = 120 * 1024;             // one CTA per SM: each CTA owns the whole TMEM
    SPEC_CUDA_OK(launch_dependent(kernels[ragged][0][p.rem_cols > 0][causal_window], dim3(n_ctas), kThreads, smem, st, tm_q, tm_k, p));
    SPEC_CUDA_OK(launch_dependent(kernels[ragged][1][reduce == SPEC_REDUCE_MAX][causal_window], dim3(n_ctas), kThreads, smem, st, tm_q, tm_k, p));
  }
  return SPEC_OK;
}
