// Modified CMRS (Section 6.6): strips rearranged into 32-item warp passes that
// hold at most M contiguous items of any one row (M = slots, 1..8; the
// paper's is 8), filled with zero items, so that the SpMV kernel can add
// each product into slot (lane mod M) of its row's buffer without two lanes
// of a pass meeting in one slot.  With M = 1 and height 32 every pass holds
// exactly one item (or zero item) of each row, row r at lane r.
//
// One warp per strip, lane r owning row r.  Each pass is planned from the
// items each row has left: C = max(ceil(total / 32), ceil(longest / M))
// passes remain; every row first takes max(0, left - M (C - 1)) items (what
// the remaining C - 1 passes cannot hold), free room then goes to the rows
// with most items left (ties: lower row) up to min(left, M) each, and room
// still free becomes zero items, rows 0 upwards, each row topped up to M.
// Inside a pass the rows appear in ascending order, each one run.
//
// The plan always ends after exactly C0 = max(ceil(T / 32), ceil(L / M))
// passes (T the strip's items, L its longest row), the fewest any arrangement
// can have: with C passes left every row holds at most M C items, so each
// forced take max(0, left - M (C - 1)) is at most left / C and together they
// fit in one pass; the pass then takes min(32, sum of min(left, M)) items,
// which is at least total - 32 (C - 1) because left - min(left, M) <=
// left (C - 1) / C; so after it both the total and the longest row fit in
// C - 1 passes.  The layout pass therefore counts C0 per strip from T and L
// alone; a scan turns the counts into the padded StripPtr; the fill pass runs
// the plan and writes, never more passes than the layout gave the strip.
#include <algorithm>

#include "common.cuh"
#include "scan.cuh"
#include "stage.cuh"

namespace cmrs {
namespace {

constexpr int kPadWarps = 8;
constexpr uint32_t kFull = 0xffffffffu;
constexpr uint32_t ST_PAD_PLAN = 2u;

__device__ __forceinline__ int warp_excl_scan(int v, int lane) {
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  return incl - v;
}

// First item of row `lane` of strip [sa, sb) (RowInStrip is non-decreasing
// in an unsorted strip) and its item count; lanes at or past the height get 0.
__device__ __forceinline__ int row_span(int sa, int sb, int height, uint32_t mask,
                                        const uint32_t *__restrict__ packed, int lane, int *first) {
  int start = sa;
  if (lane > 0 && lane < height) {
    int lo = sa, hi = sb;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((packed[mid] & mask) < (uint32_t)lane) lo = mid + 1;
      else hi = mid;
    }
    start = lo;
  }
  int end = __shfl_down_sync(kFull, start, 1);
  if (lane == height - 1) end = sb;
  *first = start;
  return lane < height ? end - start : 0;
}

// Sum of v (0..kM) over the lanes below this one.  For M = 2 by two votes,
// which do not wait for each other as a shuffle scan's five steps do.
template <int kM>
__device__ __forceinline__ int small_scan(int v, int lane) {
  if (kM > 2) return warp_excl_scan(v, lane);
  const unsigned lt = (1u << lane) - 1;
  return __popc(__ballot_sync(kFull, v & 1) & lt) + 2 * __popc(__ballot_sync(kFull, v & 2) & lt);
}

// One pass of the plan in its general form, for the passes k_pad_fill's short
// form does not cover: `left` items per row, C passes left (this one
// included).  Writes the pass at out (32 items) and takes it off left and
// next; returns false, with nothing written, if the pass would overflow
// (never for a valid unsorted strip).
template <typename S, bool kSplit, int kM>
__device__ __forceinline__ bool pad_pass(int &left, int &next, int C, int height,
                                         const uint32_t *__restrict__ cp, const S *__restrict__ vh,
                                         const S *__restrict__ vl, uint32_t *__restrict__ pk_out,
                                         S *__restrict__ vo_h, S *__restrict__ vo_l) {
  const int lane = threadIdx.x & 31;
  int take = max(0, left - kM * (C - 1));
  int room = 32 - (int)__reduce_add_sync(kFull, (unsigned)take);
  if (room < 0 || __any_sync(kFull, take > kM)) return false;
  // free room: rows with most items left first, lower row on ties
  const int want = min(left, kM) - take;
  const int wanted = (int)__reduce_add_sync(kFull, (unsigned)max(want, 0));
  int extra;
  if (wanted <= room) {
    extra = max(want, 0);  // every row gets what it wants
  } else {
    // before = the want of the rows ranked ahead (more items left, or as
    // many and a lower row), one distinct count of items left at a time,
    // largest first, until the free room is given out
    const int lv = want > 0 ? left - take : 0;  // >= 1 for a row that wants
    unsigned rem = __ballot_sync(kFull, want > 0);
    int before = room, done = 0;
    while (rem && done < room) {
      const int v = (int)__reduce_max_sync(kFull, (rem >> lane) & 1u ? (unsigned)lv : 0u);
      const unsigned g = __ballot_sync(kFull, ((rem >> lane) & 1u) && lv == v);
      const int wg = (g >> lane) & 1u ? want : 0;
      const int below = small_scan<kM>(wg, lane);  // want of the group's lower rows
      if ((g >> lane) & 1u) before = done + below;
      done += (int)__reduce_add_sync(kFull, (unsigned)wg);
      rem &= ~g;
    }
    extra = want > 0 ? max(0, min(want, room - before)) : 0;
  }
  take += extra;
  room -= (int)__reduce_add_sync(kFull, (unsigned)extra);
  // zero items: rows 0 upwards, each topped up to M
  const int zcap = lane < height ? kM - take : 0;
  const int zero = max(0, min(zcap, room - small_scan<kM>(zcap, lane)));
  const int len = take + zero;
  const int off = small_scan<kM>(len, lane);
#pragma unroll
  for (int j = 0; j < kM; ++j) {
    if (j < take) {
      pk_out[off + j] = cp[next + j];
      vo_h[off + j] = vh[next + j];
      if (kSplit) vo_l[off + j] = vl[next + j];
    } else if (j < len) {
      pk_out[off + j] = (uint32_t)lane;  // column 0, this row
      vo_h[off + j] = S(0);
      if (kSplit) vo_l[off + j] = S(0);
    }
  }
  next += take;
  left -= take;
  return true;
}

// An item read from the stage, or from global memory by a load that may pass
// the stores before it (the compiler cannot tell that they do not alias).
template <bool kStaged, typename T>
__device__ __forceinline__ T item(const T *p) {
  if constexpr (kStaged) return *p;
  return __ldg(p);
}

// Runs the plan of one strip and writes its `limit` passes from out0 on.  The
// strip's items are cp[next..], lane r's row starting at `next` with `left`
// items; map: this warp's 2 x 32 words of shared memory.
//
// The passes left are limit - p throughout (the plan takes exactly the
// minimum, see the top of the file), so a pass needs neither the total nor
// the longest row.  With t the items left such that rows above t all go and
// rows at t go lowest first until 32 / M rows do, a pass with t >= M is
// exactly those 32 / M rows, M items each, and no zero item: every chosen row
// holds M items, and a forced row (left > M (C - 1)) ranks at M (C - 1), so
// it goes in full whenever t lies below that, or no row is forced at all.  t
// only falls from pass to pass, so it is found by stepping down from the last
// pass's, a vote a step.  Lane j then reads item j % M of the (j / M)-th
// chosen row, whose next item is passed through `map`; the pass is read and
// stored while the next one is planned, so that the votes do not wait for the
// two reads (M < 8).  On rows of 4..60 items (height 32, M = 2) 94% of the
// passes take this form.  k_pad_fill on 2,097,152 such rows (67M FP32
// entries): 1,149 us when every pass ran the general form, 316 us with each
// pass read as it was planned, 290 us so; reading and writing the items
// once is 163 us.  What is left: fixed latencies (votes, their use; a quarter
// as many waits for shared memory) at 20 warps per SM (the stage's shared
// memory), issue 62% of an SM's active cycles, and SMs that have run out of
// strips while others work (524,288 such rows, 5.4 strips a warp: active 81% of
// the elapsed cycles, issue 50%).  Forms with small stages are bound by
// registers instead: 48 (10 CTAs per SM) against the compiler's 56 leave rows
// of power-law lengths 10% faster, 40 spill and are 4-17% slower.
template <typename S, bool kSplit, int kM, bool kStaged>
__device__ __forceinline__ void pad_strip_fill(int left, int next, int height, long long limit, uint32_t *map,
                                               const uint32_t *__restrict__ cp, const S *__restrict__ vh,
                                               const S *__restrict__ vl, long long out0,
                                               uint32_t *__restrict__ pk_out, S *__restrict__ vo_h,
                                               S *__restrict__ vo_l) {
  constexpr int K = 32 / kM;  // rows of a full pass
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1;
  uint32_t *po = pk_out + out0;
  S *ho = vo_h + out0, *lo = kSplit ? vo_l + out0 : nullptr;
  if (limit <= 0) return;
  int t = (int)__reduce_max_sync(kFull, (unsigned)left);
  po += lane;
  ho += lane;
  lo += kSplit ? lane : 0;
  // passes left after this one (below 2^31 / 32).  The last pass never takes
  // the short form: every item left is forced then.
  int src = 0;        // this position's item in the pass planned last,
  bool held = false;  // which is copied while the next one is planned
  for (int D = (int)limit - 1; D > 0; --D, po += 32, ho += 32, lo += kSplit ? 32 : 0) {
    uint32_t c;
    S h, l;
    if (held) {
      c = cp[src];
      h = vh[src];
      if (kSplit) l = vl[src];
    }
    unsigned gt = __ballot_sync(kFull, left > t), ge = __ballot_sync(kFull, left >= t);
    if (__popc(ge) < K) {
      gt = ge;
      ge = __ballot_sync(kFull, left >= --t);  // the next lower count, usually
      while (__popc(ge) < K) {                 // ends: at t = 0 every lane votes
        gt = ge;
        t = (int)__reduce_max_sync(kFull, left < t ? (unsigned)left : 0u);
        ge = __ballot_sync(kFull, left >= t);
      }
    }
    if (t >= kM && (t < kM * D || !__any_sync(kFull, left > kM * D))) {
      const bool sel = left > t || (left == t && __popc(ge & ~gt & lt) < K - __popc(gt));
      const unsigned sm = __ballot_sync(kFull, sel);
      uint32_t *mp = map + ((D & 1) << 5);  // alternate halves: one warp barrier a pass
      if (sel) {
        mp[__popc(sm & lt)] = (uint32_t)next;
        next += kM;
        left -= kM;
      }
      if (held) {
        po[-32] = c;
        ho[-32] = h;
        if (kSplit) lo[-32] = l;
      }
      __syncwarp();
      src = (int)mp[lane / kM] + (lane & (kM - 1));
      if (kM == 8) {  // four rows a pass: few passes in a row take this form, and holding one cost 5-8%
        *po = cp[src];
        *ho = vh[src];
        if (kSplit) *lo = vl[src];
        continue;
      }
      held = true;
      continue;
    }
    if (held) {
      po[-32] = c;
      ho[-32] = h;
      if (kSplit) lo[-32] = l;
    }
    held = false;
    const unsigned some = __ballot_sync(kFull, left > 0);
    const int same = __popc(some) > K ? 0 : min(D, (int)__reduce_min_sync(kFull, left > 0 ? (unsigned)left / kM : ~0u >> 1));
    __syncwarp();
    if (same > 1) {
      // 32 / M rows or fewer have items left, so each takes min(left, M) of them
      // every pass; until one holds fewer than M the passes are alike: M items
      // of each, the same zero items.  The pass's layout once -- each position's
      // row, and where its items lie -- then `same` passes of copies.  (A strip
      // with one row of 2,000 items, M = 8: 250 passes of 2 us each before.)
      const int take = left > 0 ? kM : 0;
      const int zcap = lane < height ? kM - take : 0;
      const int zero = max(0, min(zcap, 32 - kM * __popc(some) - small_scan<kM>(zcap, lane)));
      const int len = take + zero, off = small_scan<kM>(len, lane);
      const unsigned rows = __ballot_sync(kFull, len > 0);
      const unsigned starts = __reduce_or_sync(kFull, len > 0 ? 1u << off : 0u);
      if (len > 0) {
        const int k = __popc(rows & lt);
        map[k] = (uint32_t)next;
        map[32 + k] = (uint32_t)(off | take << 8 | lane << 16);
      }
      __syncwarp();
      const int k = __popc(starts << (31 - lane)) - 1;  // the run of this position
      const uint32_t in = map[32 + k];
      const int at = lane - (int)(in & 255);
      const bool real = at < (int)((in >> 8) & 255);
      const int src = (int)map[k] + at;
      const uint32_t filler = in >> 16;  // a zero item: column 0, this row
      __syncwarp();
#pragma unroll(kStaged && kM < 8 ? 2 : 4)
      for (int p = 0; p < same; ++p) {
        po[32 * (long long)p] = real ? item<kStaged>(cp + src + kM * p) : filler;
        ho[32 * (long long)p] = real ? item<kStaged>(vh + src + kM * p) : S(0);
        if (kSplit) lo[32 * (long long)p] = real ? item<kStaged>(vl + src + kM * p) : S(0);
      }
      next += take * same;
      left -= take * same;
      D -= same - 1;
      po += 32 * (long long)(same - 1);
      ho += 32 * (long long)(same - 1);
      lo += kSplit ? 32 * (long long)(same - 1) : 0;
    } else {
      if (!pad_pass<S, kSplit, kM>(left, next, D + 1, height, cp, vh, vl, po - lane, ho - lane,
                                   kSplit ? lo - lane : nullptr))
        return;
    }
  }
  if (held) {
    po[-32] = cp[src];
    ho[-32] = vh[src];
    if (kSplit) lo[-32] = vl[src];
  }
  pad_pass<S, kSplit, kM>(left, next, 1, height, cp, vh, vl, po - lane, ho - lane, kSplit ? lo - lane : nullptr);
}

// Passes of each strip: max(ceil(T / 32), ceil(L / M)), 0 for an empty strip.
__global__ void __launch_bounds__(kPadWarps * 32) k_pad_count(int strips, int height, int bits, int slots,
                                                             const int32_t *__restrict__ sp,
                                                             const uint32_t *__restrict__ packed,
                                                             int32_t *__restrict__ counts, uint32_t *status) {
  const int nw = gridDim.x * kPadWarps;
  const int lane = threadIdx.x & 31;
  const uint32_t mask = (1u << bits) - 1;
  for (int s = blockIdx.x * kPadWarps + (threadIdx.x >> 5); s < strips; s += nw) {
    const int sa = sp[s], sb = sp[s + 1];
    int first;
    const int len = row_span(sa, sb, height, mask, packed, lane, &first);
    const bool bad = __any_sync(kFull, len < 0) || sb < sa;
    const int longest = (int)__reduce_max_sync(kFull, (unsigned)max(len, 0));
    if (lane == 0) {
      if (bad) atomicOr(status, ST_PAD_PLAN);
      const long long T = bad ? 0 : sb - sa;
      const long long c = std::max((T + 31) / 32, ((long long)longest + slots - 1) / slots);
      counts[s] = bad ? 0 : (int32_t)std::min<long long>(c, 0x7fffffffLL);
    }
  }
}

// height x M = 32 (M = 1: height 32): every row with items left takes
// min(items left, M) per pass (together at most 32, so the free room never
// turns one away) and zero items top it up to M, so row r has positions r M ..
// r M + M - 1 of every pass, and the strip has max(ceil(row length / M))
// passes.  No plan to run: lane j copies every M-th item of row j / M,
// U passes' loads in flight.  16.8M FP32 entries in rows of 4..60 at
// height 16, M = 2: 151 us by the plan, 62 us so; M = 1 (twice the items,
// most of them zero) 60 us either way.
template <typename S, bool kSplit, int kM>
__device__ __forceinline__ void pad_strip_fill_even(int left, int next, long long limit,
                                                    const uint32_t *__restrict__ cp, const S *__restrict__ vh,
                                                    const S *__restrict__ vl, long long out0,
                                                    uint32_t *__restrict__ pk_out, S *__restrict__ vo_h,
                                                    S *__restrict__ vo_l) {
  constexpr int U = kM == 1 ? 8 : 4;
  const int lane = threadIdx.x & 31, row = lane / kM;
  const int items = __shfl_sync(kFull, left, row) - (lane & (kM - 1));  // of this position's row, from its first here
  const int first = __shfl_sync(kFull, next, row) + (lane & (kM - 1));
  const int passes = (int)limit;  // below 2^31 / 32
  for (int p = 0; p < passes; p += U) {
    uint32_t c[U];
    S h[U], l[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      c[u] = (uint32_t)row;  // a zero item: column 0, this row
      h[u] = S(0);
      l[u] = S(0);
      const int k = (p + u) * kM;
      if (k < items) {
        c[u] = cp[first + k];
        h[u] = vh[first + k];
        if (kSplit) l[u] = vl[first + k];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (p + u < passes) {
        const long long o = out0 + (p + u) * 32LL + lane;
        pk_out[o] = c[u];
        vo_h[o] = h[u];
        if (kSplit) vo_l[o] = l[u];
      }
  }
}

// Strip [sa, sb) whose item k is at cp[k - base].
template <typename S, bool kSplit, int kM, bool kStaged>
__device__ __forceinline__ void pad_strip(int sa, int sb, int base, int height, int bits, long long limit,
                                          uint32_t *map, const uint32_t *__restrict__ cp, const S *__restrict__ vh,
                                          const S *__restrict__ vl, long long out0, uint32_t *__restrict__ pk_out,
                                          S *__restrict__ vo_h, S *__restrict__ vo_l) {
  int next;
  int left = row_span(sa - base, sb - base, height, (1u << bits) - 1, cp, threadIdx.x & 31, &next);
  if (left < 0) left = 0;  // a corrupt strip, which the layout pass reports
  if (kM == 1 || height * kM == 32)
    pad_strip_fill_even<S, kSplit, kM>(left, next, limit, cp, vh, vl, out0, pk_out, vo_h, vo_l);
  else
    pad_strip_fill<S, kSplit, kM, kStaged>(left, next, height, limit, map, cp, vh, vl, out0, pk_out, vo_h, vo_l);
}

// Asks for the lines of [a, b) in L2, a line per lane and step.
template <typename T>
__device__ __forceinline__ void prefetch_l2(const T *a, const T *b) {
  constexpr int kLine = 128 / sizeof(T);
  for (const T *p = a + (threadIdx.x & 31) * kLine; p < b; p += 32 * kLine)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// One strip per warp.  The strip's items are copied into the warp's own
// shared-memory stage by one bulk copy per stream (the plan then reads them M
// at a time from 32 / M rows, which from global memory touches as many lines
// per load); a strip longer than the stage is read from global memory.  The
// stage also serves the row-start searches.  Should a copy's bounded wait
// give up, the warp reads this and its later strips from global memory, so
// the result does not depend on it, and waits (bounded) once more before it
// leaves.
constexpr int kFillWarps = 4;
constexpr int kFillCap = 2048;    // most items per stage
constexpr int kFillAhead = 2048;  // most items of a longer strip asked for in L2
template <int DT, int kM>
__global__ void __launch_bounds__(kFillWarps * 32, kM == 1 ? 8 : 10) k_pad_fill(int strips, int height, int bits, int cap, int nnz,
                                                             const int32_t *__restrict__ sp,
                                                             const uint32_t *__restrict__ packed,
                                                             const typename Form<DT>::Stored *__restrict__ vh,
                                                             const typename Form<DT>::Stored *__restrict__ vl,
                                                             const int32_t *__restrict__ sp_out,
                                                             uint32_t *__restrict__ pk_out,
                                                             typename Form<DT>::Stored *__restrict__ vo_h,
                                                             typename Form<DT>::Stored *__restrict__ vo_l) {
  typedef typename Form<DT>::Stored S;
  constexpr bool kSplit = DT == CMRS_BF16X2;
  extern __shared__ __align__(128) char smem[];
  __shared__ uint64_t bars[kFillWarps];
  __shared__ StageInfo info[kFillWarps];
  __shared__ uint32_t maps[kFillWarps][64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  char *stg = smem + (size_t)w * (cap ? Stage<DT>::bytes(cap) : 0);
  if (lane == 0) {
    mbar_init(&bars[w], 1);
    fence_barrier_init();
  }
  __syncwarp();
  uint64_t pol = 0;
  if (lane == 0) pol = policy_evict_first();
  uint32_t phase = 0;
  bool stages = cap > 0;
  const int nw = gridDim.x * kFillWarps;
  for (int s = blockIdx.x * kFillWarps + w; s < strips; s += nw) {
    const int sa = sp[s], sb = sp[s + 1];
    bool staged = stages && sb > sa && sb - sa <= cap;
    if (staged && lane == 0) issue_stage<DT>(sa, sb, nnz, packed, vh, vl, stg, cap, &bars[w], pol, &info[w]);
    if (!staged) {
      // read from global memory below, a few passes' loads at a time: from L2,
      // the strip's first kFillAhead items (power-law rows of 1M, M = 8 at
      // height 16: 250 -> 129 us with the reads of passes alike by item<>).
      // Should every warp of the largest launch (6,080) ask for that many at
      // once, FP64's 149 MB would pass the 129 MB of L2, FP32's 100 MB not.
      const int to = sb - sa > kFillAhead ? sa + kFillAhead : sb;
      prefetch_l2(packed + sa, packed + to);
      prefetch_l2(vh + sa, vh + to);
      if (kSplit) prefetch_l2(vl + sa, vl + to);
    }
    const long long o0 = sp_out[s], o1 = sp_out[s + 1];
    const long long limit = o1 > o0 ? (o1 - o0) / 32 : 0;
    if (staged) {
      if (__all_sync(kFull, mbar_wait_bounded(&bars[w], phase))) {
        phase ^= 1;
      } else {
        staged = stages = false;
      }
    }
    // compiled twice, so that the staged walk's reads are shared-memory loads
    if (staged) {
      const char *sh = stg + Stage<DT>::colp_bytes(cap);
      pad_strip<S, kSplit, kM, true>(sa, sb, (int)info[w].a8, height, bits, limit, maps[w],
                               reinterpret_cast<const uint32_t *>(stg), reinterpret_cast<const S *>(sh),
                               reinterpret_cast<const S *>(sh + Stage<DT>::val_bytes(cap)), o0, pk_out, vo_h, vo_l);
    } else {
      pad_strip<S, kSplit, kM, false>(sa, sb, 0, height, bits, limit, maps[w], packed, vh, vl, o0, pk_out, vo_h, vo_l);
    }
    __syncwarp();  // every lane is done with the stage before the next copy lands in it
  }
  if (cap > 0 && !stages) mbar_wait_bounded(&bars[w], phase);  // the late copy lands before the warp leaves
}

size_t pad_ws_bytes(int strips) { return 256 + scan_ws_bytes(strips); }

int slots_log2(int slots) {
  for (int k = 0; k <= 3; ++k)
    if (slots == (1 << k)) return k;
  return -1;
}

int check_pad_input(const cmrs_matrix *A, int slots) {
  if (slots_log2(slots) < 0) return CMRS_ERR_ARG;
  if (!A) return CMRS_ERR_ARG;
  if (A->rows < 0 || A->cols < 0 || A->nnz < 0) return CMRS_ERR_ARG;
  const int bits = cmrs_bits_for_height(A->height);
  if (bits < 0) return CMRS_ERR_HEIGHT;
  if (A->bits != bits || A->strips != ceil_div(A->rows, A->height)) return CMRS_ERR_ARG;
  if (A->dtype < CMRS_F64 || A->dtype > CMRS_BF16X2) return CMRS_ERR_ARG;
  if (A->flags & ~(CMRS_SORTED | CMRS_PADDED | CMRS_PAD_SLOTS_MASK)) return CMRS_ERR_ARG;
  if (A->flags) return CMRS_ERR_UNSUPPORTED;  // sorted strips, or already padded
  if (A->height * slots < 32) return CMRS_ERR_HEIGHT;
  if (A->rows > 0 && !A->strip_ptr) return CMRS_ERR_ARG;
  if (A->nnz > 0 && (!A->col_packed || !A->val)) return CMRS_ERR_ARG;
  return CMRS_OK;
}

int pad_grid(int strips) {
  static int sms = 0;
  if (sms == 0) sms = sm_count();
  return (int)std::min<long long>(ceil_div(strips, kPadWarps), (long long)sms * 8);
}

template <int DT, int kM>
int launch_fill_m(const cmrs_matrix *A, const int32_t *sp_out, int nnz_padded, uint32_t *pk_out, void *val_out,
                  cudaStream_t st) {
  typedef typename Form<DT>::Stored S;
  constexpr bool kSplit = DT == CMRS_BF16X2;
  const S *vh = reinterpret_cast<const S *>(A->val);
  const S *vl = kSplit ? vh + cmrs_pad8(A->nnz) : nullptr;
  S *oh = reinterpret_cast<S *>(val_out);
  S *ol = kSplit ? oh + cmrs_pad8(nnz_padded) : nullptr;
  // stage: 1.25x an average strip, so that most strips fit and short ones
  // leave shared memory for more warps; none where the arrays' alignment does
  // not allow bulk copies, and none where the strips are longer than any stage:
  // it would stay empty and cost the warps that hide the reads' latency (rows
  // of 200, height 32, M = 1, 12M FP64 entries: 279 us with an empty stage, 89
  // without).
  const bool aligned = ((reinterpret_cast<uintptr_t>(A->col_packed) | reinterpret_cast<uintptr_t>(A->val)) & 15) == 0;
  const long long avg = A->nnz / A->strips;
  const int cap = aligned && avg <= kFillCap ? (int)std::min<long long>(kFillCap, (avg + avg / 4) / 32 * 32 + 64) : 0;
  const size_t smem = cap ? (size_t)kFillWarps * Stage<DT>::bytes(cap) : 0;
  const size_t smem_max = (size_t)kFillWarps * Stage<DT>::bytes(kFillCap);
  CMRS_CUDA_TRY(cudaFuncSetAttribute(k_pad_fill<DT, kM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max));
  int per_sm = 0;
  CMRS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pad_fill<DT, kM>, kFillWarps * 32, smem));
  const int grid = (int)std::min<long long>(ceil_div(A->strips, kFillWarps), (long long)std::max(1, per_sm) * sm_count());
  k_pad_fill<DT, kM><<<grid, kFillWarps * 32, smem, st>>>(A->strips, A->height, A->bits, cap, A->nnz, A->strip_ptr,
                                                          A->col_packed, vh, vl, sp_out, pk_out, oh, ol);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

template <int DT>
int launch_fill(const cmrs_matrix *A, int slots, const int32_t *sp_out, int nnz_padded, uint32_t *pk_out,
                void *val_out, cudaStream_t st) {
  switch (slots) {
    case 1: return launch_fill_m<DT, 1>(A, sp_out, nnz_padded, pk_out, val_out, st);
    case 2: return launch_fill_m<DT, 2>(A, sp_out, nnz_padded, pk_out, val_out, st);
    case 4: return launch_fill_m<DT, 4>(A, sp_out, nnz_padded, pk_out, val_out, st);
    default: return launch_fill_m<DT, 8>(A, sp_out, nnz_padded, pk_out, val_out, st);
  }
}

}  // namespace
}  // namespace cmrs

using namespace cmrs;

extern "C" int cmrs_pad_workspace(const cmrs_matrix *A, int slots, size_t *bytes) {
  if (!bytes) return CMRS_ERR_ARG;
  const int rc = check_pad_input(A, slots);
  if (rc) return rc;
  *bytes = pad_ws_bytes(A->strips);
  return CMRS_OK;
}

extern "C" int cmrs_pad_layout(const cmrs_matrix *A, int slots, int32_t *strip_ptr_padded, int32_t *nnz_padded,
                               void *workspace, size_t workspace_bytes, void *stream) {
  CMRS_TRACE();
  int rc = check_pad_input(A, slots);
  if (rc) return rc;
  if (!strip_ptr_padded || !nnz_padded) return CMRS_ERR_ARG;
  if (!workspace || workspace_bytes < pad_ws_bytes(A->strips) || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return CMRS_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  char *ws = reinterpret_cast<char *>(workspace);
  uint32_t *status = reinterpret_cast<uint32_t *>(ws);
  int32_t *counts = reinterpret_cast<int32_t *>(ws + 256);
  CMRS_CUDA_TRY(cudaMemsetAsync(status, 0, 4, st));
  const int S = A->strips;
  if (S == 0) {
    CMRS_CUDA_TRY(cudaMemsetAsync(strip_ptr_padded, 0, 4, st));
    *nnz_padded = 0;
    CMRS_CUDA_TRY(cudaStreamSynchronize(st));
    return CMRS_OK;
  }
  k_pad_count<<<pad_grid(S), kPadWarps * 32, 0, st>>>(S, A->height, A->bits, slots, A->strip_ptr, A->col_packed,
                                                      counts, status);
  CMRS_LAUNCH_CHECK();
  rc = scan_counts(S, ws + 256, 32, strip_ptr_padded, status, st);
  if (rc) return rc;
  uint32_t host[2] = {0, 0};  // status, padded item count
  CMRS_CUDA_TRY(cudaMemcpyAsync(host, status, 8, cudaMemcpyDeviceToHost, st));
  CMRS_CUDA_TRY(cudaStreamSynchronize(st));
  if (host[0] & ST_PAD_PLAN) return CMRS_ERR_CSR_INVALID;
  if (host[0] & ST_SCAN_OVERFLOW) return CMRS_ERR_ARG;
  *nnz_padded = (int32_t)host[1];
  return CMRS_OK;
}

extern "C" int cmrs_pad_fill(const cmrs_matrix *A, int slots, const int32_t *strip_ptr_padded, int32_t nnz_padded,
                             uint32_t *col_packed_out, void *val_out, void *stream, cmrs_matrix *out) {
  CMRS_TRACE();
  int rc = check_pad_input(A, slots);
  if (rc) return rc;
  if (!out || nnz_padded < 0 || (nnz_padded & 31)) return CMRS_ERR_ARG;
  if (A->rows > 0 && !strip_ptr_padded) return CMRS_ERR_ARG;
  if (nnz_padded > 0 && (!col_packed_out || !val_out)) return CMRS_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(col_packed_out) | reinterpret_cast<uintptr_t>(val_out)) & 15) return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  if (A->strips > 0 && nnz_padded > 0) {
    switch (A->dtype) {
      case CMRS_F64: rc = launch_fill<CMRS_F64>(A, slots, strip_ptr_padded, nnz_padded, col_packed_out, val_out, st); break;
      case CMRS_F32: rc = launch_fill<CMRS_F32>(A, slots, strip_ptr_padded, nnz_padded, col_packed_out, val_out, st); break;
      case CMRS_BF16: rc = launch_fill<CMRS_BF16>(A, slots, strip_ptr_padded, nnz_padded, col_packed_out, val_out, st); break;
      default: rc = launch_fill<CMRS_BF16X2>(A, slots, strip_ptr_padded, nnz_padded, col_packed_out, val_out, st); break;
    }
    if (rc) return rc;
  }
  *out = *A;
  out->nnz = nnz_padded;
  out->flags = CMRS_PADDED | ((uint32_t)slots_log2(slots) << CMRS_PAD_SLOTS_SHIFT);
  out->max_strip_nnz = -1;
  out->strip_ptr = strip_ptr_padded;
  out->col_packed = col_packed_out;
  out->val = val_out;
  return CMRS_OK;
}
