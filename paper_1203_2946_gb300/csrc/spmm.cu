// Multi-right-hand-side SpMM Y = A X on CMRS matrices, for one matrix or a
// batch of uneven matrices in one persistent launch replayed from a CUDA
// graph.  Not in the paper; it applies the strip layout of Section 3 to k
// right-hand sides at once, so that each gathered row of X (k contiguous
// values) is shared by k accumulators.
//
// Thread mapping: a group of G lanes owns one row.  When k is a multiple of 4
// and X, Y are 16-byte aligned, lane g accumulates the four columns
// 4 (c0 + g) .. 4 (c0 + g) + 3 from one 16-byte gather of X (G =
// min(32, next_pow2(k / 4))): a k = 32 row takes 8 lanes and a warp works
// four rows at once.  Otherwise lane g accumulates column c0 + g (G =
// min(32, next_pow2(k))).  Columns beyond the group are done in further
// passes over the row.  A column's sum is one FMA chain in entry order, or two,
// of the even and the odd entries, joined at the end, where rows of 8 entries
// or more have one lane of columns (k = 1, 4).  Work units (matrix, row range)
// are fetched by warps from a device queue (one atomic per unit), which balances
// uneven matrices.
//
// What bounds a large batch is the L1 data pipe (rows that are short or long for
// a stage, and wide products whose X stays in L2, wait on round trips instead
// and are walked without one, see below): a warp's rows lie apart in the entry
// streams, so a column word and a value read from global memory cost a line
// each per row and entry, as much as the gather of X itself (78% busy, three
// lines an entry).  So a warp copies the entries of up to 32 consecutive rows
// -- one contiguous range -- into its own shared-memory stage with two bulk
// copies and reads words and values there, where the lanes of a row share one
// read.  Rows whose entries do not fit the stage, and matrices whose arrays
// are not 16-byte aligned, are read from global memory.  Where one or two
// lanes hold a row's columns, two lane groups share the row's entries (their
// sums joined by a shuffle), which halves the stage a warp needs.  And the
// warps of an SM work on neighbouring rows (see QueueHead), so that they find
// X in L1.  32 banded matrices (119M entries, rows of 10..60, one launch), all
// with k columns, before and after: k = 1 665 -> 244 us, k = 4 727 -> 371 us, k
// = 8 714 -> 527 us, k = 32 1,467 -> 1,199 us (its gathers of whole lines wait
// on L2: 7 CTAs of 4 warps keep more of them in flight than 5 or 6 with a
// larger L1; 2, 3, 6 and 8 gathers in flight per lane are slower than 4).
#include <algorithm>
#include <chrono>
#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"
#include "stage.cuh"

namespace cmrs {
namespace {

constexpr int kSpmmThreads = 128;
constexpr int kSpmmWarps = kSpmmThreads / 32;
constexpr int kSpmmCap = 704;   // entries per warp's stage
constexpr int kSpmmMinB = 7;    // resident CTAs per SM asked of the register allocator (72 registers)
constexpr int kSpmmD = 4;       // X gathers in flight per lane
constexpr int kSpmmBlock = 64;  // neighbouring units dealt to one SM together (8: k = 4, 8 products 12% slower)
constexpr int kSpmmSplit = 2;   // most lane groups per row (4 with a stage of 384: no faster, k = 8 slower)
constexpr size_t kSpmmSmem = kSpmmWarps * Stage<CMRS_F32>::bytes(kSpmmCap);

struct Desc {
  int32_t rows, height, bits, k, vec, nnz;
  int32_t stage;  // the arrays' alignment allows bulk copies
  int32_t split;  // lane groups sharing one row (1 or 2)
  const int32_t *sp;
  const uint32_t *packed;
  const float *val;
  const float *X;
  float *Y;
};

struct Unit {
  int32_t mat, row0, row1, pad;
};

// The queue: one share of the units per SM.  Units are dealt to the shares in
// blocks of `block` consecutive ones, so that the warps of an SM work on
// neighbouring rows of one matrix and find each other's rows of X in L1; a
// warp takes the next unit of its own SM's share, and of another's when that
// is used up.
constexpr int kMaxShares = 1024;
struct QueueHead {
  unsigned int taken[kMaxShares];  // units taken of each share
};
struct Shares {
  int nunits, shares, block, len;  // len: units per share, the last blocks counted whole
  __device__ __forceinline__ unsigned unit(int share, unsigned i) const {
    return ((i / (unsigned)block) * (unsigned)shares + (unsigned)share) * (unsigned)block + i % (unsigned)block;
  }
};

// First k in [lo, hi) whose RowInStrip is >= r, or hi; entry k is at cp[k - base].
__device__ __forceinline__ int lb_ris_g(const uint32_t *cp, int base, int lo, int hi, uint32_t r, uint32_t mask) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if ((cp[mid - base] & mask) < r) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Lanes that share one row: 16-byte columns when d.vec, else single ones.
__host__ __device__ __forceinline__ int spmm_lanes(int k, int vec) {
  const int c = vec ? k / 4 : k;
  int G = 1;
  while (G < c && G < 32) G <<= 1;
  return G;
}

__device__ __forceinline__ void fma_to(float &acc, float v, float x) { acc = fmaf(v, x, acc); }
__device__ __forceinline__ void fma_to(float4 &acc, float v, const float4 &x) {
  acc.x = fmaf(v, x.x, acc.x);
  acc.y = fmaf(v, x.y, acc.y);
  acc.z = fmaf(v, x.z, acc.z);
  acc.w = fmaf(v, x.w, acc.w);
}

__device__ __forceinline__ void join(float &acc, int lanes) { acc += __shfl_xor_sync(0xffffffffu, acc, lanes); }
__device__ __forceinline__ void join(float4 &acc, int lanes) {
  acc.x += __shfl_xor_sync(0xffffffffu, acc.x, lanes);
  acc.y += __shfl_xor_sync(0xffffffffu, acc.y, lanes);
  acc.z += __shfl_xor_sync(0xffffffffu, acc.z, lanes);
  acc.w += __shfl_xor_sync(0xffffffffu, acc.w, lanes);
}

// One lane's part of one row: columns g, g + G, ... (of kv, in units of V) of
// Y[row] from entries k0 + q, k0 + q + L, ... of [k0, k1), entry k at cp[k -
// base], vp[k - base]; the L lanes' sums are joined by a shuffle tree.  All
// lanes of the warp call (a lane without a row has k0 == k1 and row < 0).
// Batches of kSpmmD entries have their X gathers in flight together; whole
// batches go without guards, the last one with.
template <typename V>
__device__ __forceinline__ void spmm_row(const Desc &d, int row, int k0, int k1, int base, const uint32_t *cp,
                                         const float *vp, int g, int G, int q, int L, int kv) {
  const V *X = reinterpret_cast<const V *>(d.X);
  V *Y = reinterpret_cast<V *>(d.Y);
  for (int c0 = 0; c0 < kv; c0 += G) {  // warp-uniform
    const int col = c0 + g;
    V acc = {};
    if (col < kv) {
      const V *Xc = X + col;
      int j = k0 - base + q;
      const int end = k1 - base;
      for (; j + L * (kSpmmD - 1) < end; j += L * kSpmmD) {
        V xv[kSpmmD];
#pragma unroll
        for (int u = 0; u < kSpmmD; ++u) xv[u] = __ldg(Xc + (size_t)(cp[j + L * u] >> d.bits) * kv);
#pragma unroll
        for (int u = 0; u < kSpmmD; ++u) fma_to(acc, vp[j + L * u], xv[u]);
      }
      if (j < end) {
        V xv[kSpmmD - 1];
#pragma unroll
        for (int u = 0; u < kSpmmD - 1; ++u)
          if (j + L * u < end) xv[u] = __ldg(Xc + (size_t)(cp[j + L * u] >> d.bits) * kv);
#pragma unroll
        for (int u = 0; u < kSpmmD - 1; ++u)
          if (j + L * u < end) fma_to(acc, vp[j + L * u], xv[u]);
      }
    }
    for (int o = L >> 1; o > 0; o >>= 1) join(acc, o * G);  // the L lanes of a column are G apart
    if (row >= 0 && q == 0 && col < kv) Y[(size_t)row * kv + col] = acc;
  }
}

// A warp's stage.  Should a copy's bounded wait give up, the warp reads its
// rows from global memory from then on, so the result does not depend on it.
struct WarpStage {
  char *mem;
  uint64_t *bar;
  StageInfo *info;
  uint64_t pol;
  uint32_t phase;
  bool ok;
};

// Rows [row0, row1) of matrix d, processed by one warp.
__device__ __forceinline__ void spmm_rows(const Desc &d, int row0, int row1, WarpStage &st) {
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int kv = d.vec ? d.k >> 2 : d.k;
  const int G = spmm_lanes(d.k, d.vec);
  const int L = d.split, per = 32 / (G * L);  // rows worked at once
  const int g = lane & (G - 1), q = (lane / G) & (L - 1), sub = lane / (G * L);
  const uint32_t mask = (1u << d.bits) - 1;
  for (int ra = row0; ra < row1;) {
    // lane r: row ra + r, its strip's bounds
    const int row = ra + lane;
    const bool active = row < row1;
    int a = 0, b = 0;
    uint32_t r = 0;
    if (active) {
      const int s = d.height == 1 ? row : (int)((unsigned)row / (unsigned)d.height);
      r = (uint32_t)(row - s * d.height);
      a = __ldg(d.sp + s);
      b = __ldg(d.sp + s + 1);
    }
    // the rows whose strips fit the stage together: whole groups of `per` rows, or all that are left
    const int base = __shfl_sync(kAll, a, 0);
    int nr = 0;
    if (d.stage && st.ok) {
      nr = __popc(__ballot_sync(kAll, active && b - base <= kSpmmCap));
      if (ra + nr < row1 && nr >= per) nr = nr / per * per;
      if (2 * nr < min(per, row1 - ra)) nr = 0;  // a stage of too few rows leaves lanes idle
    }
    const bool staged = nr > 0;
    if (!staged) nr = min(per, row1 - ra);
    const uint32_t *cp = d.packed;
    int cbase = 0;
    bool use = staged;
    if (staged) {
      const int eb = __shfl_sync(kAll, b, nr - 1);
      if (lane == 0)
        issue_stage<CMRS_F32>(base, eb, d.nnz, d.packed, d.val, nullptr, st.mem, kSpmmCap, st.bar, st.pol, st.info);
      if (__all_sync(kAll, mbar_wait_bounded(st.bar, st.phase))) {
        st.phase ^= 1;
      } else {
        st.ok = use = false;
      }
    }
    if (use) {
      cp = reinterpret_cast<const uint32_t *>(st.mem);
      cbase = (int)st.info->a8;
    }
    int k0 = a, k1 = b;
    if (d.height > 1 && active && lane < nr) {
      k0 = lb_ris_g(cp, cbase, a, b, r, mask);
      k1 = lb_ris_g(cp, cbase, k0, b, r + 1, mask);
    }
    for (int g0 = 0; g0 < nr; g0 += per) {
      const int src = g0 + sub;
      int q0 = __shfl_sync(kAll, k0, src & 31), q1 = __shfl_sync(kAll, k1, src & 31);
      const bool mine = src < nr;
      if (!mine) q0 = q1 = cbase;
      const int out = mine ? ra + src : -1;
      // compiled for the stage and for global memory, so that the former's reads are shared-memory loads
      if (use) {
        const uint32_t *sc = reinterpret_cast<const uint32_t *>(st.mem);
        const float *sv = reinterpret_cast<const float *>(st.mem + Stage<CMRS_F32>::colp_bytes(kSpmmCap));
        if (d.vec) spmm_row<float4>(d, out, q0, q1, cbase, sc, sv, g, G, q, L, kv);
        else spmm_row<float>(d, out, q0, q1, cbase, sc, sv, g, G, q, L, kv);
      } else {
        if (d.vec) spmm_row<float4>(d, out, q0, q1, 0, d.packed, d.val, g, G, q, L, kv);
        else spmm_row<float>(d, out, q0, q1, 0, d.packed, d.val, g, G, q, L, kv);
      }
    }
    __syncwarp();  // every lane is done with the stage before the next copy lands in it
    ra += nr;
  }
}

__device__ __forceinline__ WarpStage warp_stage(char *smem, uint64_t *bars, StageInfo *info) {
  const int w = threadIdx.x >> 5;
  WarpStage st;
  st.mem = smem + (size_t)w * Stage<CMRS_F32>::bytes(kSpmmCap);
  st.bar = &bars[w];
  st.info = &info[w];
  if ((threadIdx.x & 31) == 0) {
    mbar_init(st.bar, 1);
    fence_barrier_init();
  }
  __syncwarp();
  st.pol = policy_evict_first();
  st.phase = 0;
  st.ok = true;
  return st;
}
// a copy whose wait gave up lands before the warp leaves
__device__ __forceinline__ void warp_stage_end(WarpStage &st) {
  if (!st.ok) mbar_wait_bounded(st.bar, st.phase);
}

__global__ void __launch_bounds__(kSpmmThreads, kSpmmMinB) k_spmm_queue(const Desc *__restrict__ descs,
                                                                            const Unit *__restrict__ units, Shares sh,
                                                                            QueueHead *q) {
  extern __shared__ __align__(128) char smem[];
  __shared__ uint64_t bars[kSpmmWarps];
  __shared__ StageInfo info[kSpmmWarps];
  WarpStage st = warp_stage(smem, bars, info);
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned smid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  const int own = (int)(smid % (unsigned)sh.shares);
  int share = own;
  for (;;) {
    unsigned i = 0;
    if (lane == 0) i = atomicAdd(&q->taken[share], 1u);
    i = __shfl_sync(kAll, i, 0);
    if (i >= (unsigned)sh.len) {
      // used up: the next share, from this SM's on, with units left
      int found = -1;
      for (int k0 = 0; k0 < sh.shares && found < 0; k0 += 32) {
        const int k = k0 + lane;
        int s = own + k;
        if (s >= sh.shares) s -= sh.shares;
        const bool left = k < sh.shares && *reinterpret_cast<volatile unsigned *>(&q->taken[s]) < (unsigned)sh.len;
        const unsigned m = __ballot_sync(kAll, left);
        if (m) found = __shfl_sync(kAll, s, __ffs(m) - 1);
      }
      if (found < 0) break;
      share = found;
      continue;
    }
    const unsigned u = sh.unit(share, i);
    if (u >= (unsigned)sh.nunits) continue;  // a block past the end
    const Unit un = units[u];
    const Desc d = descs[un.mat];
    spmm_rows(d, un.row0, un.row1, st);
  }
  warp_stage_end(st);
}

// One matrix, no queue: warp w takes rows [w*rpw, (w+1)*rpw).
__global__ void __launch_bounds__(kSpmmThreads, kSpmmMinB) k_spmm_one(Desc d, int rows_per_warp) {
  extern __shared__ __align__(128) char smem[];
  __shared__ uint64_t bars[kSpmmWarps];
  __shared__ StageInfo info[kSpmmWarps];
  const long long w = ((long long)blockIdx.x * kSpmmThreads + threadIdx.x) >> 5;
  const long long r0 = w * rows_per_warp;
  if (r0 >= d.rows) return;
  WarpStage st = warp_stage(smem, bars, info);
  const int r1 = (int)std::min<long long>(r0 + rows_per_warp, d.rows);
  spmm_rows(d, (int)r0, r1, st);
  warp_stage_end(st);
}

// ------------------------------------------------------------------ walked
// The same sums without a stage: every lane finds its row's bounds and reads
// column words and values from global memory (the lanes of a row share each
// line), at 40 warps per SM instead of 28 and with no round trip before the
// first gather.  The faster way where the stage holds too little (see
// spmm_staged, plan_staged): rows too short or too long for it, tall strips,
// and wide products whose X stays in L2.
constexpr int kWalkThreads = 256;
constexpr int kWalkD = 2;  // X gathers in flight per lane (more raise the 48 registers that 5 CTAs leave)

// Rows [row0, row1) of matrix d, processed by one warp: columns g, g + G, ...
// of a row from its entries q, q + L, ..., summed as spmm_row sums them.  Of
// 16-byte columns the next batch's column words and values are loaded while
// this batch's gathers are in flight.
template <typename V, int L>
__device__ __forceinline__ void walk_rows(const Desc &d, int row0, int row1) {
  constexpr bool kAhead = sizeof(V) == 16;
  const int lane = threadIdx.x & 31;
  const int kv = kAhead ? d.k >> 2 : d.k;
  const int G = spmm_lanes(d.k, kAhead), per = 32 / (G * L);
  const int g = lane & (G - 1), q = (lane / G) & (L - 1), sub = lane / (G * L);
  const uint32_t mask = (1u << d.bits) - 1;
  const V *X = reinterpret_cast<const V *>(d.X);
  V *Y = reinterpret_cast<V *>(d.Y);
  for (int rb = row0; rb < row1; rb += per) {
    const int row = rb + sub;
    const bool active = row < row1;
    int k0 = 0, k1 = 0;
    if (active) {
      const int s = row / d.height;
      k0 = __ldg(d.sp + s);
      k1 = __ldg(d.sp + s + 1);
      if (d.height > 1) {
        const uint32_t r = (uint32_t)(row - s * d.height);
        k0 = lb_ris_g(d.packed, 0, k0, k1, r, mask);
        k1 = lb_ris_g(d.packed, 0, k0, k1, r + 1, mask);
      }
      k0 += q;
    }
    for (int c0 = 0; c0 < kv; c0 += G) {  // warp-uniform
      const int col = c0 + g;
      V acc = {};
      if (active && col < kv) {
        uint32_t pn[kWalkD];
        float vn[kWalkD];
        if (kAhead) {
#pragma unroll
          for (int u = 0; u < kWalkD; ++u)
            if (k0 + L * u < k1) {
              pn[u] = __ldg(d.packed + k0 + L * u);
              vn[u] = __ldg(d.val + k0 + L * u);
            }
        }
        for (int j = k0; j < k1; j += L * kWalkD) {
          V xv[kWalkD];
          float vv[kWalkD];
#pragma unroll
          for (int u = 0; u < kWalkD; ++u) {
            if (kAhead) {
              vv[u] = vn[u];
              if (j + L * u < k1) xv[u] = __ldg(X + (size_t)(pn[u] >> d.bits) * kv + col);
            } else if (j + L * u < k1) {
              const uint32_t p = __ldg(d.packed + j + L * u);
              vv[u] = __ldg(d.val + j + L * u);
              xv[u] = __ldg(X + (size_t)(p >> d.bits) * kv + col);
            }
          }
          if (kAhead) {
#pragma unroll
            for (int u = 0; u < kWalkD; ++u)
              if (j + L * (kWalkD + u) < k1) {
                pn[u] = __ldg(d.packed + j + L * (kWalkD + u));
                vn[u] = __ldg(d.val + j + L * (kWalkD + u));
              }
          }
#pragma unroll
          for (int u = 0; u < kWalkD; ++u)
            if (j + L * u < k1) fma_to(acc, vv[u], xv[u]);
        }
        if (L == 1) Y[(size_t)row * kv + col] = acc;
      }
      if (L > 1) {
        join(acc, G);
        if (active && q == 0 && col < kv) Y[(size_t)row * kv + col] = acc;
      }
    }
  }
}
// kSplit: some matrices have two lane groups per row (compiled apart: together
// they spill)
template <bool kSplit>
__global__ void __launch_bounds__(kWalkThreads, 5) k_spmm_walk_queue(const Desc *__restrict__ descs,
                                                                     const Unit *__restrict__ units, int nunits,
                                                                     QueueHead *q) {
  for (;;) {
    unsigned u = 0;
    if ((threadIdx.x & 31) == 0) u = atomicAdd(&q->taken[0], 1u);
    u = __shfl_sync(0xffffffffu, u, 0);
    if (u >= (unsigned)nunits) break;
    const Unit un = units[u];
    const Desc d = descs[un.mat];
    if (kSplit && d.split > 1) {
      if (d.vec) walk_rows<float4, 2>(d, un.row0, un.row1);
      else walk_rows<float, 2>(d, un.row0, un.row1);
    } else {
      if (d.vec) walk_rows<float4, 1>(d, un.row0, un.row1);
      else walk_rows<float, 1>(d, un.row0, un.row1);
    }
  }
}

// One matrix, no queue: warp w takes rows [w*rpw, (w+1)*rpw).
template <typename V, int L>
__global__ void __launch_bounds__(kWalkThreads, 5) k_spmm_walk_one(Desc d, int rows_per_warp) {
  const long long r0 = (((long long)blockIdx.x * kWalkThreads + threadIdx.x) >> 5) * rows_per_warp;
  if (r0 >= d.rows) return;
  walk_rows<V, L>(d, (int)r0, (int)std::min<long long>(r0 + rows_per_warp, d.rows));
}
int launch_walk_one(const Desc &d, cudaStream_t st) {
  const int per = 32 / (spmm_lanes(d.k, d.vec) * d.split);
  const int grid = (int)ceil_div(ceil_div(d.rows, per) * 32, kWalkThreads);
  if (d.vec && d.split == 1) k_spmm_walk_one<float4, 1><<<grid, kWalkThreads, 0, st>>>(d, per);
  else if (d.vec) k_spmm_walk_one<float4, 2><<<grid, kWalkThreads, 0, st>>>(d, per);
  else if (d.split == 1) k_spmm_walk_one<float, 1><<<grid, kWalkThreads, 0, st>>>(d, per);
  else k_spmm_walk_one<float, 2><<<grid, kWalkThreads, 0, st>>>(d, per);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

// Whether one matrix's product takes the stage: where it was the faster way on
// 1,290 points (0.5 to 1,500 entries a row, heights 1 to 32, 1 to 64 columns; us
// walked -> staged).  A row's words have to be many, or read by many lanes, to
// pay for the copy's round trip (5-point rows, 1M: k = 1, 4 13 -> 23, 16 -> 27),
// and a group of rows has to fit the stage (200 entries a row, k = 2 78 -> 129;
// strips of 32 rows of 40, k = 8 54 -> 80); narrow products of 12 to 65 entries
// a row do both (40, 200,000 rows: k = 1 43 -> 23, k = 5 84 -> 71).  Rows of 300
// and more are read from global memory either way, few columns with four
// gathers in flight (400, 15,000 rows: k = 1 89 -> 31).
bool spmm_staged(const Desc &d) {
  const double mu = (double)d.nnz / d.rows, strip = mu * d.height;
  if (!d.stage) return false;
  if (mu >= 300.0) return d.k <= 5;
  if (strip > 600.0) return false;
  if (d.k == 1) return mu >= 12.0 && mu <= 65.0;
  if (d.k == 2) return mu >= 15.0 && mu <= 65.0;
  if (!d.vec) return (d.height >= 4 || mu >= 4.0) && mu <= 130.0;
  if (d.k == 4) return mu >= 18.0 && mu <= 55.0;
  if (d.k == 8) return d.height >= 2 && mu <= 6.0;
  return d.height >= 2 && mu <= 35.0 && d.rows >= 60000;
}

// Whether a batch does: by the sum of its products' times (nnz (24 + k), as
// one-launch batches of one k take them) with what the stage gains on each, from
// 645 batches of one matrix and 120 of many: narrow products 1.5 to 2.5 times
// the speed; wide ones whose X outgrows L2 (the blocks of the queue keep its
// rows in L1) 1.2, others 0.75 to 1.1 (15 matrices of 16,000 rows, k = 4, 8, 16:
// 74 us walked, 83 staged).
bool plan_staged(const std::vector<Desc> &descs) {
  double wide = 0.0;  // bytes of the wide products' X and Y
  for (const Desc &d : descs)
    if (d.vec && d.k >= 8) wide += 8.0 * d.rows * d.k;
  double walked = 0.0, staged = 0.0;
  for (const Desc &d : descs) {
    if (d.nnz == 0) continue;
    const double mu = (double)d.nnz / d.rows, work = (double)d.nnz * (24 + d.k);
    double gain = d.k == 1 ? 2.2 : 1.6;
    if (d.k == 1 || (d.vec && d.k == 4)) gain = mu < 3.0 ? 0.85 : mu < 5.5 ? 0.95 : gain;
    if (d.vec && d.k >= 8)
      gain = mu >= 300.0                            ? 1.3
             : wide > 128e6                         ? (mu >= 12.0 ? 1.2 : d.height > 1 ? 1.1 : 0.92)
             : mu * d.height > 600.0                ? 0.75
             : wide > 32e6                          ? (d.height > 1 ? 1.1 : 0.95)
             : d.k == 8                             ? (mu >= 110.0 ? 1.2 : 0.8)
             : d.k > 32                             ? 0.75
             : d.height > 1                         ? (mu <= 18.0 ? 1.1 : d.k > 16 ? 1.0 : 0.88)
                                                    : 0.86;
    walked += work;
    staged += work / (d.stage ? gain : 0.8);
  }
  return staged <= walked;
}

int spmm_smem_opt_in() {
  CMRS_CUDA_TRY(cudaFuncSetAttribute(k_spmm_queue, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpmmSmem));
  CMRS_CUDA_TRY(cudaFuncSetAttribute(k_spmm_one, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpmmSmem));
  return CMRS_OK;
}

int check_item(const cmrs_matrix *A, int k, const float *X, float *Y) {
  if (!A || k < 1) return CMRS_ERR_ARG;
  if (A->dtype != CMRS_F32) return CMRS_ERR_UNSUPPORTED;
  if (A->flags & (CMRS_SORTED | CMRS_PADDED)) return CMRS_ERR_UNSUPPORTED;
  if (cmrs_bits_for_height(A->height) != A->bits) return CMRS_ERR_HEIGHT;
  if (A->rows < 0 || A->nnz < 0 || A->strips != ceil_div(A->rows, A->height)) return CMRS_ERR_ARG;
  if (A->rows > 0 && (!A->strip_ptr || !Y)) return CMRS_ERR_ARG;
  if (A->nnz > 0 && (!A->col_packed || !A->val || !X)) return CMRS_ERR_ARG;
  return CMRS_OK;
}

Desc make_desc(const cmrs_matrix *A, int k, const float *X, float *Y) {
  Desc d;
  d.rows = A->rows;
  d.height = A->height;
  d.bits = A->bits;
  d.k = k;
  d.sp = A->strip_ptr;
  d.packed = A->col_packed;
  d.val = reinterpret_cast<const float *>(A->val);
  d.X = X;
  d.Y = Y;
  d.vec = (k % 4 == 0) && !((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15);
  d.nnz = A->nnz;
  d.stage = ((reinterpret_cast<uintptr_t>(A->col_packed) | reinterpret_cast<uintptr_t>(A->val)) & 15) == 0;
  // Lanes per row: with one lane a row, 32 rows at once would need a stage four
  // times as large (fewer warps, less L1 for X); rows too short to feed the
  // lanes keep fewer.
  const double mu = A->rows > 0 ? (double)A->nnz / A->rows : 0.0;
  d.split = 1;
  while (d.split < kSpmmSplit && spmm_lanes(k, d.vec) * d.split < kSpmmSplit && mu >= 8.0 * d.split) d.split <<= 1;
  return d;
}

int rows_per_unit(const cmrs_matrix *A, int k, int vec, int work_target) {
  // work of a row ~ (nnz/rows) * k entry-columns; keep units near work_target
  const double mu = A->rows > 0 ? (double)A->nnz / A->rows : 1.0;
  const int per = 32 / spmm_lanes(k, vec);
  double r = work_target / std::max(1.0, mu * k);
  int ri = (int)std::max<double>(per, std::min<double>(r, 1 << 20));
  ri = (ri + per - 1) / per * per;
  return ri;
}

}  // namespace
}  // namespace cmrs

using namespace cmrs;

// Plan: host-side object holding the schedule layout and the captured graph.
struct cmrs_spmm_plan {
  int batch = 0, nunits = 0, work_target = 0;
  Desc *d_desc = nullptr;
  Unit *d_units = nullptr;
  QueueHead *d_q = nullptr;
  int grid = 0;
  Shares sh = {};
  bool staged = false, split = false;  // split: a walked plan with two lane groups per row somewhere
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

extern "C" int cmrs_spmm(const cmrs_matrix *A, int k, const float *X, float *Y, void *stream) {
  CMRS_TRACE();
  int rc = check_item(A, k, X, Y);
  if (rc) return rc;
  if (A->rows == 0) return CMRS_OK;
  cudaStream_t st = as_stream(stream);
  if (A->nnz == 0) {
    CMRS_CUDA_TRY(cudaMemsetAsync(Y, 0, (size_t)A->rows * k * sizeof(float), st));
    return CMRS_OK;
  }
  const Desc d = make_desc(A, k, X, Y);
  // rows per warp: up to 32 (one stage), fewer while the warps would not fill
  // the SMs twice, whole groups of the rows a warp works at once
  const int per = 32 / (spmm_lanes(k, d.vec) * d.split);
  if (!spmm_staged(d)) return launch_walk_one(d, st);
  const long long resident = (long long)sm_count() * kSpmmMinB * kSpmmWarps;
  const int rpw = (int)std::max<long long>(per, std::min<long long>(32, A->rows / (2 * resident)) / per * per);
  const long long warps = ceil_div(A->rows, rpw);
  const int grid = (int)ceil_div(warps * 32, kSpmmThreads);
  const int arc = spmm_smem_opt_in();
  if (arc) return arc;
  k_spmm_one<<<grid, kSpmmThreads, kSpmmSmem, st>>>(d, rpw);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

static int build_units(int batch, const cmrs_matrix *const *A, const int32_t *k, int work_target,
                       std::vector<Unit> &units) {
  units.clear();
  for (int b = 0; b < batch; ++b) {
    const int rpu = rows_per_unit(A[b], k[b], k[b] % 4 == 0, work_target);
    for (int r0 = 0; r0 < A[b]->rows; r0 += rpu) {
      Unit u;
      u.mat = b;
      u.row0 = r0;
      u.row1 = std::min(A[b]->rows, r0 + rpu);
      u.pad = 0;
      units.push_back(u);
    }
  }
  // heaviest units first, so the queue ends on small ones
  std::stable_sort(units.begin(), units.end(), [&](const Unit &x, const Unit &y) {
    auto w = [&](const Unit &u) {
      const cmrs_matrix *m = A[u.mat];
      const double mu = m->rows ? (double)m->nnz / m->rows : 0.0;
      return (double)(u.row1 - u.row0) * mu * k[u.mat];
    };
    return w(x) > w(y);
  });
  return CMRS_OK;
}

// Shares of a plan's units: blocks of up to kSpmmBlock units, smaller ones
// while a share would hold fewer than eight.
static Shares make_shares(size_t nunits) {
  Shares sh;
  sh.nunits = (int)nunits;
  sh.shares = std::max(1, std::min(sm_count(), kMaxShares));
  sh.block = std::max(1, std::min(kSpmmBlock, sh.nunits / (8 * sh.shares)));
  sh.len = (int)ceil_div(ceil_div(sh.nunits, sh.block), sh.shares) * sh.block;
  return sh;
}

// Units of wide products are dealt one by one instead: where a row of X fills
// whole lines (four or more 16-byte lanes), neighbouring rows on one SM find
// few of each other's lines in L1, and their misses wait for each other there
// (k = 32: 1,298 us in blocks of 64, 1,212 us one by one; k = 4: 374 us in
// blocks, 423 us one by one).  The units of every full round over the shares
// are reordered so that the blocks deal them that way.
static void deal_wide(const Shares &sh, const int32_t *k, std::vector<Unit> &units) {
  const size_t round = (size_t)sh.shares * sh.block;
  std::vector<Unit> tmp(round);
  for (size_t r0 = 0; r0 + round <= units.size(); r0 += round) {
    const int ka = k[units[r0].mat], kb = k[units[r0 + round - 1].mat];
    if (spmm_lanes(ka, ka % 4 == 0) < 4 || spmm_lanes(kb, kb % 4 == 0) < 4) continue;
    for (size_t i = 0; i < round; ++i) tmp[i % sh.shares * sh.block + i / sh.shares] = units[r0 + i];
    std::copy(tmp.begin(), tmp.end(), units.begin() + r0);
  }
}

// The queue's reset and the persistent launch.
static cudaError_t enqueue_plan(const cmrs_spmm_plan *p, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(p->d_q, 0, sizeof(unsigned int) * (p->staged ? p->sh.shares : 1), st);
  if (e != cudaSuccess) return e;
  if (p->staged) k_spmm_queue<<<p->grid, kSpmmThreads, kSpmmSmem, st>>>(p->d_desc, p->d_units, p->sh, p->d_q);
  else if (p->split) k_spmm_walk_queue<true><<<p->grid, kWalkThreads, 0, st>>>(p->d_desc, p->d_units, p->nunits, p->d_q);
  else k_spmm_walk_queue<false><<<p->grid, kWalkThreads, 0, st>>>(p->d_desc, p->d_units, p->nunits, p->d_q);
  return cudaSuccess;
}

extern "C" int cmrs_spmm_plan_workspace(int batch, const cmrs_matrix *const *A, const int32_t *k, int work_target,
                                        size_t *bytes) {
  if (batch < 0 || !bytes || (batch > 0 && (!A || !k)) || work_target < 1) return CMRS_ERR_ARG;
  std::vector<Unit> units;
  for (int b = 0; b < batch; ++b)
    if (!A[b] || k[b] < 1) return CMRS_ERR_ARG;
  build_units(batch, A, k, work_target, units);
  *bytes = align256(sizeof(QueueHead)) + align256(sizeof(Desc) * (size_t)std::max(1, batch)) +
           align256(sizeof(Unit) * std::max<size_t>(1, units.size()));
  return CMRS_OK;
}

extern "C" int cmrs_spmm_plan_create(int batch, const cmrs_matrix *const *A, const int32_t *k, const float *const *X,
                                     float *const *Y, int work_target, int use_graph, void *workspace,
                                     size_t workspace_bytes, void *stream, cmrs_spmm_plan **out) {
  CMRS_TRACE();
  if (!out) return CMRS_ERR_ARG;
  *out = nullptr;
  if (batch < 1 || !A || !k || !X || !Y || work_target < 1) return CMRS_ERR_ARG;
  for (int b = 0; b < batch; ++b) {
    int rc = check_item(A[b], k[b], X[b], Y[b]);
    if (rc) return rc;
  }
  size_t need = 0;
  int rc = cmrs_spmm_plan_workspace(batch, A, k, work_target, &need);
  if (rc) return rc;
  if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255)) return CMRS_ERR_WORKSPACE;
  std::vector<Unit> units;
  build_units(batch, A, k, work_target, units);
  const Shares sh = make_shares(units.size());
  std::vector<Desc> descs(batch);
  for (int b = 0; b < batch; ++b) descs[b] = make_desc(A[b], k[b], X[b], Y[b]);
  const bool staged = plan_staged(descs);
  if (staged) deal_wide(sh, k, units);
  cmrs_spmm_plan *p = new (std::nothrow) cmrs_spmm_plan();
  if (!p) return CMRS_ERR_ARG;
  char *ws = reinterpret_cast<char *>(workspace);
  p->batch = batch;
  p->nunits = (int)units.size();
  p->sh = sh;
  p->staged = staged;
  for (const Desc &d : descs) p->split |= d.split > 1;
  p->work_target = work_target;
  p->d_q = reinterpret_cast<QueueHead *>(ws);
  p->d_desc = reinterpret_cast<Desc *>(ws + align256(sizeof(QueueHead)));
  p->d_units = reinterpret_cast<Unit *>(ws + align256(sizeof(QueueHead)) + align256(sizeof(Desc) * batch));
  cudaStream_t st = as_stream(stream);
  // Host -> device copies of the schedule; synchronised here because the host
  // vectors go out of scope (plan creation is not on the hot path).
  cudaError_t e = cudaMemcpyAsync(p->d_desc, descs.data(), sizeof(Desc) * batch, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && !units.empty())
    e = cudaMemcpyAsync(p->d_units, units.data(), sizeof(Unit) * units.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    delete p;
    return set_cuda_error(e);
  }
  if (const int arc = spmm_smem_opt_in()) {
    delete p;
    return arc;
  }
  int per_sm = 1;
  if (staged) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spmm_queue, kSpmmThreads, kSpmmSmem);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spmm_walk_queue<false>, kWalkThreads, 0);
  p->grid = std::max(1, per_sm) * sm_count();
  if (use_graph) {
    // the graph holds the queue reset and the persistent launch; replaying it
    // costs one graph launch per batch
    cudaStream_t cap = nullptr;
    e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      enqueue_plan(p, cap);
      e = cudaStreamEndCapture(cap, &p->graph);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&p->exec, p->graph, 0);
    if (cap) cudaStreamDestroy(cap);
    if (e != cudaSuccess) {
      if (p->exec) cudaGraphExecDestroy(p->exec);
      if (p->graph) cudaGraphDestroy(p->graph);
      delete p;
      return set_cuda_error(e);
    }
  }
  *out = p;
  return CMRS_OK;
}

extern "C" int cmrs_spmm_batched(cmrs_spmm_plan *p, void *stream) {
  CMRS_TRACE();
  if (!p) return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  if (p->exec) {
    CMRS_CUDA_TRY(cudaGraphLaunch(p->exec, st));
  } else {
    CMRS_CUDA_TRY(enqueue_plan(p, st));
    CMRS_LAUNCH_CHECK();
  }
  return CMRS_OK;
}

extern "C" int cmrs_spmm_plan_info(const cmrs_spmm_plan *p, int *nunits, int *grid, int *work_target) {
  if (!p) return CMRS_ERR_ARG;
  if (nunits) *nunits = p->nunits;
  if (grid) *grid = p->grid;
  if (work_target) *work_target = p->work_target;
  return CMRS_OK;
}

extern "C" int cmrs_spmm_plan_destroy(cmrs_spmm_plan *p) {
  if (!p) return CMRS_OK;
  if (p->exec) cudaGraphExecDestroy(p->exec);
  if (p->graph) cudaGraphDestroy(p->graph);
  delete p;
  return CMRS_OK;
}

// Autotuner for the batch schedule: builds a plan per candidate unit size,
// times `reps` graph replays of each with CUDA events and keeps the fastest.
extern "C" int cmrs_spmm_autotune(int batch, const cmrs_matrix *const *A, const int32_t *k, const float *const *X,
                                  float *const *Y, const int *candidates, int ncand, int reps, void *workspace,
                                  size_t workspace_bytes, void *stream, int *best_target, float *best_ms) {
  CMRS_TRACE();
  if (!candidates || ncand < 1 || reps < 1 || !best_target) return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  cudaEvent_t e0, e1;
  CMRS_CUDA_TRY(cudaEventCreate(&e0));
  CMRS_CUDA_TRY(cudaEventCreate(&e1));
  float best = 1e30f;
  int bt = candidates[0];
  int rc = CMRS_OK;
  for (int c = 0; c < ncand && rc == CMRS_OK; ++c) {
    cmrs_spmm_plan *p = nullptr;
    rc = cmrs_spmm_plan_create(batch, A, k, X, Y, candidates[c], 1, workspace, workspace_bytes, stream, &p);
    if (rc) break;
    for (int w = 0; w < 2 && rc == CMRS_OK; ++w) rc = cmrs_spmm_batched(p, stream);
    cudaEventRecord(e0, st);
    for (int r = 0; r < reps && rc == CMRS_OK; ++r) rc = cmrs_spmm_batched(p, stream);
    cudaEventRecord(e1, st);
    cudaError_t e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e != cudaSuccess && rc == CMRS_OK) rc = set_cuda_error(e);
    cmrs_spmm_plan_destroy(p);
    ms /= reps;
    if (rc == CMRS_OK && ms < best) {
      best = ms;
      bt = candidates[c];
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  *best_target = bt;
  if (best_ms) *best_ms = best;
  return CMRS_OK;
}
